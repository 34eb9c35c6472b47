// The two solid mass solves of the preconditioner (block A_22^-1, Section 5),
// temporally blocked: several Chebyshev-Jacobi steps on C_s per launch.
//
// A step on a body of a few thousand nodes is a tiny sparse product; one launch
// per step costs a graph node and three dependent memory round trips (1.8 to
// 2.7 us each in FP32 up to 32 000 nodes, 24 of them in a row).  Here the body's
// nodes are split into compact patches, one CTA each.  A CTA holds its patch
// grown by as many layers of neighbours as it takes steps, so the steps of a
// launch need no exchange: step s updates the layers it still can (a prefix of
// the patch's nodes, which are ordered by layer).  Rows live in registers, the
// iterate in shared memory.  Every node is computed by the same operations in
// the same order in whichever patches hold it, so the result does not depend on
// the patch that writes it.
//
// What bounds it: in FP32 the gathers from shared memory (a warp's 32 random
// 8-byte reads per entry); in FP64 the FP64 pipe, 64 cycles per warp
// instruction, which the repeated layers multiply, so FP64 takes fewer steps per
// launch on large bodies.  plan_solid_patches() weighs both.  Measured, both
// solves of the FP32 preconditioner with the C_f product before them: 41 -> 11.6
// us on 217 nodes, 46 -> 16.7 on 3997, 64 -> 29.6 on 32 137, 137 -> 55 on 126 691;
// FP64: 66 -> 39 on 127 nodes, 87 -> 68 on 3997.
#pragma once
#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

#include "fsi_internal.h"
#include "fsi_kernels.cuh"

namespace fsi {

constexpr int kScMaxSteps = 32;   // Chebyshev steps of one launch
constexpr int kScWide = 12;       // widest row the patches take

template <class T>
struct SolidPatches {
  int np = 0;          // patches; 0: the per-step kernels run instead
  int steps = 0;       // layers held: most steps of one launch
  int width = 0;       // entries per stored row (8 or 12)
  int rpt = 1;         // rows per thread (1 or 2)
  size_t smem = 0;     // shared memory of a CTA
  const int* poff = nullptr;       // first node of a patch in gid (np + 1)
  const int* cnt = nullptr;        // cnt[p (steps + 1) + l]: nodes of patch p in layers 0 .. l
  const int* gid = nullptr;        // solid node of every patch node
  const int* roff = nullptr;       // first row of a patch (np + 1)
  const T* val = nullptr;          // entry k of row i of patch p: roff[p] width + k rows + i
  const uint16_t* col = nullptr;   // its patch node
};

template <class T>
struct SolidChebArgs {
  SolidPatches<T> P;
  int ns = 0;                // steps of this launch
  int first = 0, last = 0;   // starts from x = d = c0 D^-1 b; writes only x
  T c0 = 0;
  T c1[kScMaxSteps], c2[kScMaxSteps];
  const T* dinv = nullptr;
  // b = scale bsrc, or with kx K kx - bsrc (K: A_s or the tangent, whole body)
  const T* bsrc = nullptr;
  T scale = 1;
  Sell<T> K;
  const T* kx = nullptr;
  const T *xin = nullptr, *din = nullptr;
  T *xout = nullptr, *dout = nullptr;
};

template <class T>
__device__ __forceinline__ typename Vec2<T>::type sc_rhs(const SolidChebArgs<T>& a, int g) {
  using T2 = typename Vec2<T>::type;
  T2 b = reinterpret_cast<const T2*>(a.bsrc)[g];
  if (!a.kx) {
    b.x *= a.scale;
    b.y *= a.scale;
    return b;
  }
  const int base = a.K.soff[g >> 3] + (g & 7), n = a.K.len[g];
  T s0 = 0, s1 = 0;
  for (int k = 0; k < n; ++k) {
    const int slot = base + (k << 3);
    const T2 x = reinterpret_cast<const T2*>(a.kx)[a.K.col[slot]];
    if (a.K.kron) {
      const T v = a.K.val[slot];
      s0 += v * x.x;
      s1 += v * x.y;
    } else {   // the tangent's 2 x 2 blocks
      const T* v = a.K.val + 4 * (size_t)slot;
      s0 += v[0] * x.x + v[1] * x.y;
      s1 += v[2] * x.x + v[3] * x.y;
    }
  }
  b.x = s0 - b.x;
  b.y = s1 - b.y;
  return b;
}

template <class T, int W, int RPT, int NT>
__global__ void __launch_bounds__(NT) k_solid_cheb(const __grid_constant__ SolidChebArgs<T> a) {
  using T2 = typename Vec2<T>::type;
  extern __shared__ __align__(16) unsigned char sc_smem[];
  const int p = blockIdx.x, tid = threadIdx.x, ns = a.ns;
  const int* cnt = a.P.cnt + (size_t)p * (a.P.steps + 1);
  const int* gid = a.P.gid + a.P.poff[p];
  const int rows = a.P.roff[p + 1] - a.P.roff[p];       // rows stored for this patch
  const int nrow = ns > 0 ? cnt[ns - 1] : 0, nloc = cnt[ns];
  // constants, before the wait for the producers: the rows in registers
  T v[RPT][W];
  unsigned c[RPT][W / 2];
  int g[RPT];
  T2 dv[RPT];
  {
    const T* val = a.P.val + (size_t)a.P.roff[p] * W;
    const uint16_t* col = a.P.col + (size_t)a.P.roff[p] * W;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int i = tid + q * NT;
      g[q] = -1;
      if (i >= nrow) continue;
      g[q] = gid[i];
      dv[q] = reinterpret_cast<const T2*>(a.dinv)[g[q]];
#pragma unroll
      for (int k = 0; k < W; ++k) v[q][k] = val[(size_t)k * rows + i];
#pragma unroll
      for (int k = 0; k < W; k += 2)
        c[q][k / 2] = (unsigned)col[(size_t)k * rows + i] | ((unsigned)col[(size_t)(k + 1) * rows + i] << 16);
    }
  }
  pdl_begin();
  T2* xc = reinterpret_cast<T2*>(sc_smem);
  T2* xn = xc + nloc;
  T2 b[RPT], d[RPT], x[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    if (g[q] < 0) continue;
    b[q] = sc_rhs<T>(a, g[q]);
    if (a.first) {
      d[q].x = a.c0 * dv[q].x * b[q].x;
      d[q].y = a.c0 * dv[q].y * b[q].y;
      x[q] = d[q];
    } else {
      x[q] = reinterpret_cast<const T2*>(a.xin)[g[q]];
      d[q] = reinterpret_cast<const T2*>(a.din)[g[q]];
    }
    xc[tid + q * NT] = x[q];
  }
  for (int i = nrow + tid; i < nloc; i += NT) {   // the outermost layer: only read
    const int gi = gid[i];
    T2 xv;
    if (a.first) {
      const T2 bv = sc_rhs<T>(a, gi), di = reinterpret_cast<const T2*>(a.dinv)[gi];
      xv.x = a.c0 * di.x * bv.x;
      xv.y = a.c0 * di.y * bv.y;
    } else {
      xv = reinterpret_cast<const T2*>(a.xin)[gi];
    }
    xc[i] = xv;
  }
  __syncthreads();
  for (int s = 0; s < ns; ++s) {
    const int act = cnt[ns - 1 - s];
    const T c1 = a.c1[s], c2 = a.c2[s];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int i = tid + q * NT;
      if (i >= act) continue;
      T s0 = 0, s1 = 0, t0 = 0, t1 = 0;
#pragma unroll
      for (int k = 0; k < W; k += 2) {
        const T2 xa = xc[c[q][k / 2] & 0xffffu], xb = xc[c[q][k / 2] >> 16];
        s0 += v[q][k] * xa.x;
        s1 += v[q][k] * xa.y;
        t0 += v[q][k + 1] * xb.x;
        t1 += v[q][k + 1] * xb.y;
      }
      d[q].x = c1 * d[q].x + c2 * dv[q].x * (b[q].x - (s0 + t0));
      d[q].y = c1 * d[q].y + c2 * dv[q].y * (b[q].y - (s1 + t1));
      x[q].x += d[q].x;
      x[q].y += d[q].y;
      xn[i] = x[q];
    }
    __syncthreads();
    T2* t = xc;
    xc = xn;
    xn = t;
  }
  const int own = cnt[0];
  for (int i = tid; i < own; i += NT) reinterpret_cast<T2*>(a.xout)[gid[i]] = xc[i];
  if (!a.last) {
#pragma unroll
    for (int q = 0; q < RPT; ++q)
      if (tid + q * NT < own) reinterpret_cast<T2*>(a.dout)[g[q]] = d[q];
  }
}

// ------------------------------------------------------------------- host
// Threads of a patch's CTA: FP32 rows take about 30 registers each, FP64 rows
// twice that, so 1024 FP32 or 512 FP64 threads hold the whole register file.
template <class T>
constexpr int sc_threads() { return sizeof(T) == 4 ? 1024 : 512; }

struct SolidPlan {
  int np = 0, launches = 1, steps = 0;
};

// Patches and launches per solve for n nodes and m Chebyshev steps.  The model
// (in us, from the measured per-step kernels): a launch costs 3, a step 0.1
// plus 0.3 per 1024 rows in FP32, 0.7 per 128 rows in FP64 (10 multiply-adds
// per row and component at 64 cycles a warp instruction); a patch of s nodes
// grown by l layers of a planar mesh holds (sqrt(s) + 2 l)^2.
inline SolidPlan plan_solid_patches(int n, int m, bool f64, int max_rows) {
  SolidPlan best;
  double best_t = 1e300;
  for (int launches = 1; launches <= std::max(1, m); ++launches) {
    const int h = (m + launches - 1) / launches;
    if (h > kScMaxSteps) continue;
    for (int np : {1, 2, 4, 8, 16, 32, 48, 76, 152, 304, 608, 1216}) {
      if (np > 1 && n / np < 8) break;
      const double own = (double)n / np, r = std::sqrt(own);
      const double rows = np == 1 ? n : std::min((double)n, (r + 2.0 * std::max(0, h - 1)) * (r + 2.0 * std::max(0, h - 1)));
      if (rows * 1.15 > max_rows) continue;
      const double step = f64 ? 0.15 + 0.7 * std::ceil(rows / 128) : 0.1 + 0.3 * rows / 1024;
      const double t = launches * (3.0 + h * step) * ((np + 151) / 152);
      if (t < best_t) {
        best_t = t;
        best.np = np;
        best.launches = launches;
        best.steps = h;
      }
    }
  }
  return best;
}

struct SolidPatchHost {
  int np = 0, steps = 0, launches = 1, width = 0, max_rows = 0, max_loc = 0;
  std::vector<int> poff, cnt, gid, roff;
  std::vector<double> val;
  std::vector<uint16_t> col;
};

// Patches of the body (recursive bisection of its reference positions), grown
// by layers of C_s neighbours.  False when the mesh does not suit (a row wider
// than kScWide, layers that outgrow the registers): the caller keeps the
// per-step kernels.
inline bool build_solid_patches(const HostBlockMatrix& Cs, const double* xy, int m, bool f64, int threads,
                                SolidPatchHost& out) {
  const int n = Cs.nrows;
  int wide = 0;
  for (int r = 0; r < n; ++r) wide = std::max(wide, Cs.ptr[r + 1] - Cs.ptr[r]);
  if (wide > kScWide || n == 0) return false;
  out.width = wide <= 8 ? 8 : kScWide;
  const SolidPlan plan = plan_solid_patches(n, m, f64, 2 * threads);
  if (plan.np == 0) return false;
  out.np = plan.np;
  out.steps = plan.steps;
  out.launches = plan.launches;
  // bisect the longer side until np parts, part sizes in proportion
  std::vector<int> ids(n), part(n, 0);
  for (int i = 0; i < n; ++i) ids[i] = i;
  struct Range { int lo, hi, p0, p1; };
  std::vector<Range> todo{{0, n, 0, plan.np}};
  while (!todo.empty()) {
    const Range r = todo.back();
    todo.pop_back();
    if (r.p1 - r.p0 == 1) {
      for (int i = r.lo; i < r.hi; ++i) part[ids[i]] = r.p0;
      continue;
    }
    double b[4] = {1e300, -1e300, 1e300, -1e300};
    for (int i = r.lo; i < r.hi; ++i)
      for (int c = 0; c < 2; ++c) {
        const double x = xy[2 * (size_t)ids[i] + c];
        b[2 * c] = std::min(b[2 * c], x);
        b[2 * c + 1] = std::max(b[2 * c + 1], x);
      }
    const int c = b[1] - b[0] >= b[3] - b[2] ? 0 : 1, pm = (r.p0 + r.p1) / 2;
    const int mid = r.lo + (int)((long long)(r.hi - r.lo) * (pm - r.p0) / (r.p1 - r.p0));
    std::nth_element(ids.begin() + r.lo, ids.begin() + mid, ids.begin() + r.hi, [&](int i, int j) {
      const double xi = xy[2 * (size_t)i + c], xj = xy[2 * (size_t)j + c];
      return xi < xj || (xi == xj && i < j);
    });
    todo.push_back({r.lo, mid, r.p0, pm});
    todo.push_back({mid, r.hi, pm, r.p1});
  }
  std::vector<std::vector<int>> own(plan.np);
  for (int i = 0; i < n; ++i) own[part[i]].push_back(i);
  std::vector<int> loc(n, -1);
  out.poff.assign(1, 0);
  out.roff.assign(1, 0);
  for (int p = 0; p < plan.np; ++p) {
    std::vector<int> nodes = own[p];   // ascending inside a layer
    for (size_t i = 0; i < nodes.size(); ++i) loc[nodes[i]] = (int)i;
    out.cnt.push_back((int)nodes.size());
    size_t from = 0;
    for (int l = 1; l <= plan.steps; ++l) {
      const size_t end = nodes.size();
      std::vector<int> next;
      for (size_t i = from; i < end; ++i)
        for (int k = Cs.ptr[nodes[i]]; k < Cs.ptr[nodes[i] + 1]; ++k)
          if (loc[Cs.col[k]] < 0) {
            loc[Cs.col[k]] = 0;
            next.push_back(Cs.col[k]);
          }
      std::sort(next.begin(), next.end());
      for (int v : next) {
        loc[v] = (int)nodes.size();
        nodes.push_back(v);
      }
      from = end;
      out.cnt.push_back((int)nodes.size());
    }
    const int* cnt = out.cnt.data() + (size_t)p * (plan.steps + 1);
    const int rows = plan.steps > 0 ? cnt[plan.steps - 1] : 0;
    out.max_rows = std::max(out.max_rows, rows);
    out.max_loc = std::max(out.max_loc, (int)nodes.size());
    if (rows > 2 * threads || nodes.size() > 65535) return false;
    const size_t base = out.val.size();
    out.val.resize(base + (size_t)rows * out.width, 0.0);
    out.col.resize(base + (size_t)rows * out.width);
    for (int i = 0; i < rows; ++i) {
      const int r = nodes[i], len = Cs.ptr[r + 1] - Cs.ptr[r];
      for (int k = 0; k < out.width; ++k) {
        const size_t e = base + (size_t)k * rows + i;
        out.val[e] = k < len ? Cs.val[Cs.ptr[r] + k] : 0.0;
        out.col[e] = (uint16_t)(k < len ? loc[Cs.col[Cs.ptr[r] + k]] : i);
      }
    }
    out.gid.insert(out.gid.end(), nodes.begin(), nodes.end());
    out.poff.push_back((int)out.gid.size());
    out.roff.push_back(out.roff.back() + rows);
    for (int v : nodes) loc[v] = -1;
  }
  return true;
}

}  // namespace fsi
