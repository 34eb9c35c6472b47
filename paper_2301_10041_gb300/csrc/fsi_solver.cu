// GB300 (sm_103a) solver for one time step of the DLM fictitious-domain FSI
// method (Boffi, Credali, Gastaldi, Scacchi, arXiv:2301.10041), and the C ABI
// declared in include/fsi.h.
//
// Per step (Section 4): S1 right-hand side, S2 point location, S3 binning of
// the coupling entries by fluid node, S4 C_f(X^n) and its transpose, S5 the
// block operator of Eq. (matrix), S6 the block-diagonal / block-triangular
// preconditioner of Section 5, S7 flexible GMRES (CGS2, Givens on device,
// the whole Arnoldi loop inside one CUDA graph WHILE node), S8 FP64 iterative
// refinement around FP32 operators, S9 advance.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <stdexcept>
#include <string>
#include <tuple>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/fsi.h"
#include "fsi_cluster.cuh"
#include "fsi_cluster_host.h"
#include "fsi_coupling.cuh"
#include "fsi_internal.h"
#include "fsi_kernels.cuh"
#include "fsi_mgfused.cuh"
#include "fsi_mfop.cuh"
#include "fsi_solid.cuh"
#include "fsi_solid_cheb.cuh"

namespace fsi {

struct CudaError : std::runtime_error {
  cudaError_t code;
  explicit CudaError(cudaError_t c, const char* what) : std::runtime_error(what), code(c) {}
};
#define CK(x)                                                                 \
  do {                                                                        \
    cudaError_t e_ = (x);                                                     \
    if (e_ != cudaSuccess) throw CudaError(e_, #x);                           \
  } while (0)

static inline unsigned nblk(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Every kernel of a step but the two cluster launches (the coarse levels of a
// V-cycle, the orthogonalisation of a small problem) is launched through here.  The launches carry programmatic stream serialisation, so a kernel may
// be scheduled while its predecessor on the stream finishes; each kernel
// waits for its producers (griddepcontrol.wait, in pdl_begin() or the fused
// kernels' wrapper) before it touches memory.  With the fused multigrid
// levels this measured faster than plain launches (12.5 against 11.6 steps/s
// mixed, 3.71 against 3.54 FP64, on the 128 x 128 cavity); with the per-level
// sparse kernels alone it had measured slower.  FSI_PDL=0 in the environment
// turns it off.
static bool pdl_enabled() {
  static const bool on = [] {
    const char* e = getenv("FSI_PDL");
    return !(e && e[0] == '0');
  }();
  return on;
}

template <typename... KArgs, typename... Args>
static void launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                   Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(std::forward<Args>(args))...);
  if (e != cudaSuccess) throw CudaError(e, "cudaLaunchKernelEx");
}


// ------------------------------------------------------------ device memory
struct Arena {
  std::vector<void*> ptrs;
  size_t bytes = 0, peak = 0;   // held now, and at most so far
  // bytes less than the form with every matrix and the full coarsest inverses
  // stored takes: what the tables that replace work by memory may take, so that a
  // budget for that form still admits the problem
  long long spared = 0;
  bool count_only = false;
  template <class T>
  static size_t size(size_t n) {
    return (std::max<size_t>(n, 1) * sizeof(T) + 255) & ~(size_t)255;
  }
  template <class T>
  T* alloc(size_t n) {
    const size_t b = std::max<size_t>(n, 1) * sizeof(T);
    bytes += size<T>(n);
    peak = std::max(peak, bytes);
    if (count_only) return nullptr;
    void* p = nullptr;
    if (cudaMalloc(&p, b) != cudaSuccess) throw std::bad_alloc();
    ptrs.push_back(p);
    return (T*)p;
  }
  template <class T>
  T* upload(const std::vector<T>& h) {
    T* d = alloc<T>(h.size());
    if (d && !h.empty()) CK(cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
    return d;
  }
  // give back an array of n entries that only the creation of the problem needs
  template <class T>
  void drop(T*& p, size_t n) {
    bytes -= size<T>(n);
    if (p) {
      ptrs.erase(std::find(ptrs.begin(), ptrs.end(), (void*)p));
      CK(cudaFree(p));
    }
    p = nullptr;
  }
  void release() {
    for (void* p : ptrs) cudaFree(p);
    ptrs.clear();
  }
};

template <class T>
static Sell<T> upload_sell(Arena& ar, const SellHost& s) {
  Sell<T> d;
  d.nrows = s.nrows; d.BR = s.BR; d.BC = s.BC; d.NV = s.NV; d.kron = s.kron;
  d.soff = ar.upload(s.soff);
  d.len = ar.upload(s.len);
  // runs of equal slice width (structured-grid matrices have at most 15)
  std::vector<int> rs, rw, ro;
  for (int sl = 0; sl < s.nslices; ++sl) {
    const int w = (s.soff[sl + 1] - s.soff[sl]) / kSliceRows;
    if (rw.empty() || w != rw.back()) {
      rs.push_back(sl);
      rw.push_back(w);
      ro.push_back(s.soff[sl]);
    }
  }
  std::vector<int> col = s.col;
  if (!rs.empty() && rs.size() <= (size_t)Sell<T>::kMaxRuns) {
    d.nrun = (int)rs.size();
    for (int k = 0; k < d.nrun; ++k) {
      d.run_s[k] = rs[k];
      d.run_w[k] = rw[k];
      d.run_off[k] = ro[k];
    }
    for (int r = 0; r < s.nrows; ++r) {  // mark the padding slots
      const int sl = r / kSliceRows, lane = r % kSliceRows;
      const int w = (s.soff[sl + 1] - s.soff[sl]) / kSliceRows;
      for (int k = s.len[r]; k < w; ++k) col[(size_t)s.soff[sl] + (size_t)k * kSliceRows + lane] = -1;
    }
  }
  d.col = ar.upload(col);
  std::vector<T> v(s.val.begin(), s.val.end());
  d.val = ar.upload(v);
  return d;
}

template <class T>
static T* upload_as(Arena& ar, const std::vector<double>& h) {
  std::vector<T> v(h.begin(), h.end());
  return ar.upload(v);
}

// values and columns of a matrix's stored blocks: what leaving it out spares at least
template <class T>
static double sell_bytes(const HostBlockMatrix& A) {
  return (double)A.nnzb() * (A.NV * sizeof(T) + sizeof(int));
}

// ------------------------------------------------------------- SpMV launch
template <class T, int BR, int BC, bool KRON, int NV, int TPR>
static void sell_launch_tpr(const Sell<T>& A, int mode, const SpmvArgs<T>& a, cudaStream_t s) {
  const unsigned g = nblk(A.nrows, 4 * (32 / TPR));  // 4 warps x 32/TPR block rows
  switch (mode) {
    case MODE_AXPBY: launch(k_sell<T, BR, BC, KRON, NV, MODE_AXPBY, TPR>, g, 128, 0, s, A, a); break;
    case MODE_CHEB: launch(k_sell<T, BR, BC, KRON, NV, MODE_CHEB, TPR>, g, 128, 0, s, A, a); break;
    case MODE_CHEB0: launch(k_sell<T, BR, BC, KRON, NV, MODE_CHEB0, TPR>, g, 128, 0, s, A, a); break;
    default: launch(k_sell<T, BR, BC, KRON, NV, MODE_INIT, TPR>, g, 128, 0, s, A, a); break;
  }
}

template <class T, int BR, int BC, bool KRON, int NV>
static void sell_launch_shape(const Sell<T>& A, int mode, const SpmvArgs<T>& a, cudaStream_t s) {
  if (A.tpr == 8) return sell_launch_tpr<T, BR, BC, KRON, NV, 8>(A, mode, a, s);
  sell_launch_tpr<T, BR, BC, KRON, NV, 4>(A, mode, a, s);
}

// Fused residual + restriction (k_resrestrict) of the pressure levels: full
// 3x3 restriction blocks, R L with full blocks.
template <class T, int B, bool RKRON, int RNV, int TPR>
static void resrestrict_shape(const Sell<T>& R, const Sell<T>& RA, int mode, const SpmvArgs<T>& a, cudaStream_t s) {
  const unsigned g = nblk(R.nrows, 4 * (32 / TPR));
  if (mode == MODE_INIT) launch(k_resrestrict<T, B, RKRON, RNV, MODE_INIT, TPR>, g, 128, 0, s, R, RA, a);
  else launch(k_resrestrict<T, B, RKRON, RNV, MODE_AXPBY, TPR>, g, 128, 0, s, R, RA, a);
}

template <class T>
static void resrestrict_launch(const Sell<T>& R, const Sell<T>& RA, int mode, const SpmvArgs<T>& a, cudaStream_t s) {
  if (R.nrows == 0) return;
  if (!R.kron && R.BR == 3 && RA.BR == 3) return resrestrict_shape<T, 3, false, 9, 4>(R, RA, mode, a, s);
  throw std::logic_error("unsupported restriction shape");
}

template <class T>
static void sell_launch(const Sell<T>& A, int mode, const SpmvArgs<T>& a, cudaStream_t s) {
  if (A.nrows == 0) return;
  if (A.kron && A.BR == 2) return sell_launch_shape<T, 2, 2, true, 1>(A, mode, a, s);
  if (A.BR == 2 && A.BC == 2) return sell_launch_shape<T, 2, 2, false, 4>(A, mode, a, s);
  if (A.BR == 2 && A.BC == 3) return sell_launch_shape<T, 2, 3, false, 6>(A, mode, a, s);
  if (A.BR == 3 && A.BC == 2) return sell_launch_shape<T, 3, 2, false, 6>(A, mode, a, s);
  if (A.BR == 3 && A.BC == 3) return sell_launch_shape<T, 3, 3, false, 9>(A, mode, a, s);
  throw std::logic_error("unsupported block shape");
}

template <class T>
static SpmvArgs<T> axpby(const T* x, T* y, const T* z, T alpha, T beta) {
  SpmvArgs<T> a;
  a.x = x; a.y = y; a.z = z; a.alpha = alpha; a.beta = beta;
  return a;
}

// ------------------------------------------------------------- autotuner
// Tile shape of the per-level SpMV: 4 or 8 threads per block row, chosen per
// matrix by timing both on the device in the form a V-cycle runs it (the
// Chebyshev-Jacobi smoothing step, 20 dependent launches captured in a CUDA
// graph and replayed once warm: the conditions inside a solve); 8 is kept
// only when at least 5 % faster.
// Results are cached per (device, block shape, rows, slots, precision) for
// the life of the process, so instances of one size tune once and problems
// created in one process take the same shapes (the same rounding).
static std::mutex g_tune_mu;
static std::map<std::tuple<int, int, int, int, int, int, int>, int> g_tune;

template <class T>
static void autotune_sell(Sell<T>& A, int nslots) {
  if (A.nrows == 0 || A.BR != A.BC) return;
  int dev = 0;
  CK(cudaGetDevice(&dev));
  const auto key = std::make_tuple(dev, A.BR, A.BC, (int)A.kron, A.nrows, nslots, (int)sizeof(T));
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    const auto it = g_tune.find(key);
    if (it != g_tune.end()) {
      A.tpr = it->second;
      return;
    }
  }
  const size_t nx = (size_t)A.nrows * A.BR;
  T* buf = nullptr;   // x, y, b, d, dinv
  CK(cudaMalloc(&buf, 5 * nx * sizeof(T)));
  CK(cudaMemset(buf, 0, 5 * nx * sizeof(T)));
  T* x = buf;
  T* y = buf + nx;
  cudaStream_t s;
  CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  float t[2] = {0.f, 0.f};
  SpmvArgs<T> axy;
  axy.z = buf + 2 * nx; axy.d = buf + 3 * nx; axy.dinv = buf + 4 * nx;
  axy.c1 = (T)0.5; axy.c2 = (T)0.5;
  SpmvArgs<T> ayx = axy;
  axy.x = x; axy.y = y;
  ayx.x = y; ayx.y = x;
  for (int v = 0; v < 2; ++v) {
    // 20 dependent launches (x -> y -> x ...) in a CUDA graph, as in a solve
    Sell<T> B = A;
    B.tpr = v == 0 ? 4 : 8;
    cudaGraph_t gr;
    cudaGraphExec_t ge;
    CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    for (int r = 0; r < 20; ++r) sell_launch(B, MODE_CHEB, (r & 1) ? ayx : axy, s);
    CK(cudaStreamEndCapture(s, &gr));
    CK(cudaGraphInstantiate(&ge, gr, 0));
    CK(cudaGraphLaunch(ge, s));
    CK(cudaEventRecord(e0, s));
    CK(cudaGraphLaunch(ge, s));
    CK(cudaEventRecord(e1, s));
    CK(cudaEventSynchronize(e1));
    CK(cudaEventElapsedTime(&t[v], e0, e1));
    cudaGraphExecDestroy(ge);
    cudaGraphDestroy(gr);
  }
  A.tpr = (t[1] < 0.95f * t[0]) ? 8 : 4;
  if (const char* v = getenv("FSI_TUNE_VERBOSE"); v && v[0] == '1')
    fprintf(stderr, "fsi autotune: %dx%d blocks, %d rows, %s: 4 threads/row %.2f us, 8 threads/row %.2f us -> %d\n",
            A.BR, A.BC, A.nrows, sizeof(T) == 4 ? "fp32" : "fp64", t[0] * 50.f, t[1] * 50.f, A.tpr);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaStreamDestroy(s);
  cudaFree(buf);
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune[key] = A.tpr;
}

// ---------------------------------------------------------------- multigrid
struct Cheb {
  double c0;                 // first step: d = c0 dinv r
  std::vector<double> c1, c2;  // steps 1..k-1
};

static Cheb cheb_coeffs(double lo, double hi, int k) {
  Cheb c;
  const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
  c.c0 = 1.0 / theta;
  double rho_old = 1.0 / sigma;
  for (int i = 1; i < k; ++i) {
    const double rho = 1.0 / (2.0 * sigma - rho_old);
    c.c1.push_back(rho * rho_old);
    c.c2.push_back(2.0 * rho / delta);
    rho_old = rho;
  }
  return c;
}

template <class T>
struct MGLevel {
  Sell<T> A, P, R;  // P: prolongation from the next coarser level, R: restriction to it
  Sell<T> RA;       // pressure levels: R L, so that R (b - L x) = R b - (R L) x takes one pass
  T* dinv = nullptr;
  T *x = nullptr, *x2 = nullptr, *b = nullptr, *r = nullptr, *d = nullptr;
  int n = 0;        // scalar unknowns
  int N = 0;        // cells per side
  Cheb ch;
  // the level's stencils for the fused matrix-free kernels (fsi_mgfused.cuh),
  // and whether the V-cycle runs them on this level
  bool mf = false;
  MfVelOp<T> mfu;        // velocity hierarchy
  bool mf_ok = false;    // the stencils have the form the kernels use
  T* mftab = nullptr;    // pressure hierarchy: kMfPresTab values
  MfOp<T> mfo;           // velocity hierarchy: the level's product matrix-free (mfo.N > 0)
  bool mfl = false;      // pressure hierarchy: the same, from mftab
  T divB[3][9][2] = {};  // entries of -B and -B^T on this level (residual start)
};

// Coarse levels run as one thread-block-cluster launch per V-cycle
// (fsi_cluster.cuh): levels lc .. last.
template <class T>
struct ClusterMG {
  bool on = false;
  int lc = 0;
  size_t smem = 0;
  ClArgs<T> args;
};

template <class T>
struct MG {
  std::vector<MGLevel<T>> lv;
  T* coarse_inv = nullptr;   // dense inverse of the coarsest level, rows of coarse_ld entries (none with sym_inv)
  int coarse_n = 0;
  int coarse_ld = 0;         // coarse_n rounded up to 16 bytes (the row padding is zero)
  SymMap sym;                // its mirror images, and the class matrices (k_dense_sym)
  T* sym_inv = nullptr;      // 4 x sym.R rows of sym_ld entries
  int sym_ld = 0;
  int degree = 2;
  bool pressure = false;
  ClusterMG<T> cl;
};

constexpr double kChebRatioU = 6.0;   // smoothing interval [hi/ratio, hi]
constexpr double kChebRatioP = 8.0;

// Dense inverse of the coarsest level in place on the device (FP64, rows of
// ld entries, the padding zero): Gauss-Jordan elimination, one launch per
// pivot (k_gj_step).  M holds the dense matrix on entry.
static void dense_inverse_device(Arena& ar, double* M, int n, int ld, cudaStream_t s) {
  double* rc = ar.alloc<double>(4 * (size_t)n);   // row and column copies, two pairs
  if (!ar.count_only) {
    double *r0 = rc, *c0 = rc + n, *r1 = rc + 2 * n, *c1 = rc + 3 * n;
    k_gj_first<<<nblk(n, 256), 256, 0, s>>>(n, ld, M, r0, c0);
    CK(cudaGetLastError());
    const dim3 blk(32, 8), grd((n + 31) / 32, (n + 7) / 8);
    for (int k = 0; k < n; ++k) {
      k_gj_step<<<grd, blk, 0, s>>>(n, ld, k, M, r0, c0, r1, c1);
      std::swap(r0, r1);
      std::swap(c0, c1);
    }
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(s));
  }
  ar.drop(rc, 4 * (size_t)n);
}

// 16-byte row length of the dense coarsest inverse, in entries
template <class T>
static int dense_ld(int n) {
  constexpr int w = 16 / (int)sizeof(T);
  return (n + w - 1) / w * w;
}

// Representatives of the coarsest level under the two mirrors (SymMap): scalar
// unknown i at mirrored positions.  Velocity: 2 node + component, the component
// along the mirror's normal flips; pressure: 3 cell + coefficient, the linear
// coefficient in the mirrored direction flips.
static void sym_images(int N, bool pressure, std::vector<int4>& img, std::vector<int>& sgn) {
  const VNum vn(pressure ? 0 : N);
  const int half = pressure ? (N + 1) / 2 : N, lo = pressure ? 0 : 1, nk = pressure ? 3 : 2;
  auto id = [&](int x, int y, int k) { return pressure ? 3 * (y * N + x) + k : 2 * vn.id(x, y) + k; };
  const int mir = pressure ? N - 1 : 2 * N;
  for (int y = lo; y < lo + half; ++y)
    for (int x = lo; x < lo + half; ++x)
      for (int k = 0; k < nk; ++k) {
        int4 j;
        j.x = id(x, y, k);
        j.y = id(mir - x, y, k);
        j.z = id(x, mir - y, k);
        j.w = id(mir - x, mir - y, k);
        img.push_back(j);
        sgn.push_back(pressure ? (k == 1 ? 1 : 0) | (k == 2 ? 2 : 0) : (k == 0 ? 1 : 2));
      }
}

constexpr int kSymMinF32 = 1500;   // coarsest unknowns from which the FP32 product goes by classes
constexpr int kSymThreadsF32 = 256, kSymThreadsF64 = 512;   // two and four representatives per CTA
template <class T>
constexpr int sym_threads() { return sizeof(T) == 8 ? kSymThreadsF64 : kSymThreadsF32; }

// cluster-resident coarse levels, below
template <class T>
static void setup_cluster(Arena& ar, const HostSetup& hs, MG<T>& mg, bool pressure, int max_n);

// The class matrices of the coarsest level, rounded from the FP64 ones (host,
// 4 x R rows of R entries).
template <class T>
static void upload_classes(Arena& ar, MG<T>& mg, const SymMap& sym, const std::vector<double>& g) {
  const int R = sym.R;
  mg.sym = sym;
  mg.sym_ld = dense_ld<T>(R);
  const size_t ld = mg.sym_ld;
  mg.sym_inv = ar.alloc<T>(4 * (size_t)R * ld);
  ar.spared -= Arena::size<T>(4 * (size_t)R * ld);
  if (ar.count_only) return;
  std::vector<T> v(4 * (size_t)R * ld, (T)0);
  for (size_t r = 0; r < 4 * (size_t)R; ++r)
    for (int q = 0; q < R; ++q) v[r * ld + q] = (T)g[r * R + q];
  CK(cudaMemcpy(mg.sym_inv, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
  if (4 * ld * sizeof(T) > 48 * 1024)
    CK(cudaFuncSetAttribute(k_dense_sym<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
}

// The coarsest levels' solves of one hierarchy in both precisions (m32: null
// without the FP32 one): the assembled matrix is inverted in place in FP64, and
// what the V-cycles read is formed from that.  A hierarchy whose coarse levels
// run as one cluster launch reads the full inverse; else the dense product takes
// the class matrices (k_dense_sym) in FP64, and in FP32 from some 1500 unknowns on
// (1922: 2.93 -> 2.61 us, but 1058: 2.19 -> 2.38, 768: 1.69 -> 1.90, the class sums
// outweighing the shorter read; in FP64 the multiply-adds saved always pay, 1922:
// 11.7 -> 7.3 us, 768: 5.6 -> 4.9).  The full FP64 inverse stays on the device only
// where a cluster launch reads it, and the classes go through the host one at a time,
// so that nothing but one class stands beside it: a mixed problem of 16 cells and
// 271 solid nodes takes 33 MB at most, 73 with the inverses kept beside the classes.
static void build_coarse(Arena& ar, const HostSetup& hs, bool pressure, MG<double>& m64, MG<float>* m32, int cl_max,
                         cudaStream_t s) {
  const int n = pressure ? hs.coarse_nL : hs.coarse_nA, ld = dense_ld<double>(n);
  double* full = ar.alloc<double>((size_t)n * ld);
  m64.coarse_n = n;
  m64.coarse_ld = ld;
  m64.coarse_inv = full;
  if (!ar.count_only) {
    const std::vector<double>& D = pressure ? hs.coarseL : hs.coarseA;
    CK(cudaMemsetAsync(full, 0, (size_t)n * ld * sizeof(double), s));
    CK(cudaMemcpy2DAsync(full, (size_t)ld * sizeof(double), D.data(), (size_t)n * sizeof(double),
                         (size_t)n * sizeof(double), n, cudaMemcpyHostToDevice, s));
  }
  dense_inverse_device(ar, full, n, ld, s);
  if (cl_max >= 0) setup_cluster<double>(ar, hs, m64, pressure, cl_max);
  bool cls32 = false;
  if (m32) {
    m32->coarse_n = n;
    m32->coarse_ld = dense_ld<float>(n);
    if (cl_max >= 0) setup_cluster<float>(ar, hs, *m32, pressure, cl_max);
    cls32 = !m32->cl.on && n >= kSymMinF32;
    if (!cls32) {
      m32->coarse_inv = ar.alloc<float>((size_t)n * m32->coarse_ld);
      m32->cl.args.dense_inv = m32->coarse_inv;
      if (!ar.count_only) {
        k_dense_round<float><<<dim3((m32->coarse_ld + 255) / 256, n), 256, 0, s>>>(n, full, ld, m32->coarse_inv,
                                                                                  m32->coarse_ld);
        CK(cudaGetLastError());
        CK(cudaStreamSynchronize(s));
      }
    }
  }
  const bool cls64 = !m64.cl.on;
  if (!cls64 && !cls32) return;
  SymMap sym;
  std::vector<int4> img;
  std::vector<int> sgn;
  sym_images(hs.levels[(pressure ? hs.nlev_p : hs.nlev_u) - 1].N, pressure, img, sgn);
  sym.R = (int)img.size();
  sym.img = ar.upload(img);
  sym.sgn = ar.upload(sgn);
  ar.spared -= Arena::size<int4>(img.size()) + Arena::size<int>(sgn.size());
  const size_t RR = (size_t)sym.R * sym.R;
  double* one = ar.alloc<double>(RR);
  std::vector<double> g(ar.count_only ? 0 : 4 * RR);
  for (int c = 0; c < 4 && !ar.count_only; ++c) {
    k_sym_build<<<dim3(nblk(sym.R, 128), sym.R), 128, 0, s>>>(sym, c, full, ld, one);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(g.data() + c * RR, one, RR * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
  }
  ar.drop(one, RR);
  if (cls64) {
    m64.coarse_inv = nullptr;
    ar.drop(full, (size_t)n * ld);
    ar.spared += Arena::size<double>((size_t)n * ld);
    upload_classes<double>(ar, m64, sym, g);
  }
  if (cls32) {
    ar.spared += Arena::size<float>((size_t)n * m32->coarse_ld);
    upload_classes<float>(ar, *m32, sym, g);
  }
}

// The level's velocity stencils as MfOp; none (N = 0) when the grid has none or
// a block is not of the form the kernels use: equal off-diagonal entries, zero
// for two nodes on one grid line.
template <class T>
static MfOp<T> make_mfop(const FluidLevelHost& H) {
  MfOp<T> m;
  if (!H.mf) return m;
  for (int t = 0; t < 4; ++t)
    for (int y = 0; y < 5; ++y)
      for (int x = 0; x < 5; ++x) {
        const double* c = H.stenA[t][y][x];
        if (c[1] != c[2] || ((x == 2 || y == 2) && c[1] != 0.0)) return m;
        m.c[t][y][x][0] = (T)c[0];
        m.c[t][y][x][1] = (T)c[1];
        m.c[t][y][x][2] = (T)c[3];
      }
  for (int k = 0; k < 3; ++k)
    for (int q = 0; q < 9; ++q)
      for (int d = 0; d < 2; ++d) m.divB[k][q][d] = (T)H.divB[k][q][d];
  m.N = H.N;
  return m;
}

// Smallest grids of the FP64 matrix-free products: below, a row's serial chain of
// FP64 multiply-adds is longer than the sparse kernels' (which split it four
// ways).  One smoothing step, sparse against matrix-free: velocity 20.3 -> 10.0 us
// on 128 cells, 7.4 -> 4.8 on 64, 4.7 -> 4.4 on 32; pressure 9.9 -> 4.6 on 128,
// 5.2 -> 3.3 on 64.  Full operator 33.9 -> 19.2 on 128 cells, but 7.2 against
// 10.3 us on 16.
constexpr int kMfo64MinN = 32;       // velocity and pressure levels
constexpr int kMfo64MinNFull = 64;   // full operator and Stokes residual

// One product of a level with the epilogue of a.mode: matrix-free where the
// level says so, else the sliced-ELL kernel.
template <class T>
static void level_launch(const MGLevel<T>& L, int mode, const SpmvArgs<T>& a, cudaStream_t s) {
  if constexpr (std::is_same<T, double>::value) {   // the FP32 levels take the fused kernels
    if (L.mfo.N > 0) {
      const unsigned g = mfop_grid<T>(L.mfo.N);
      if (mode == MODE_AXPBY) launch(k_mfv<T, MODE_AXPBY>, g, 128, 0, s, L.mfo, a);
      else if (mode == MODE_CHEB) launch(k_mfv<T, MODE_CHEB>, g, 128, 0, s, L.mfo, a);
      else if (mode == MODE_CHEB0) launch(k_mfv<T, MODE_CHEB0>, g, 128, 0, s, L.mfo, a);
      else throw std::logic_error("level_launch");
      return;
    }
    if (L.mfl) {
      const unsigned g = nblk(3 * (size_t)L.N * L.N, 96);
      if (mode == MODE_CHEB) launch(k_mfp<T, MODE_CHEB>, g, 96, 0, s, L.N, (const T*)L.mftab, a);
      else if (mode == MODE_CHEB0) launch(k_mfp<T, MODE_CHEB0>, g, 96, 0, s, L.N, (const T*)L.mftab, a);
      else throw std::logic_error("level_launch");
      return;
    }
  }
  sell_launch(L.A, mode, a, s);
}

// What needs no device memory of a hierarchy: sizes, smoothing coefficients and
// stencils of its levels.
template <class T>
static void plan_mg(const HostSetup& hs, bool pressure, int degree, MG<T>& mg, bool mfree) {
  const int nl = pressure ? hs.nlev_p : hs.nlev_u;
  mg.degree = degree;
  mg.pressure = pressure;
  mg.lv.resize(nl);
  for (int l = 0; l < nl; ++l) {
    const FluidLevelHost& H = hs.levels[l];
    MGLevel<T>& L = mg.lv[l];
    const HostBlockMatrix& A = pressure ? H.L : H.A;
    L.n = A.nrows * A.BR;
    L.N = H.N;
    const double hi = 1.05 * (pressure ? H.lmaxL : H.lmaxA);
    L.ch = cheb_coeffs(hi / (pressure ? kChebRatioP : kChebRatioU), hi, degree);
    if (H.mf)
      for (int k = 0; k < 3; ++k)
        for (int q = 0; q < 9; ++q)
          for (int d = 0; d < 2; ++d) L.divB[k][q][d] = (T)H.divB[k][q][d];
    if (H.mf && !pressure) {
      L.mfu.N = H.N;
      L.mf_ok = make_mfop<T>(H).N > 0;
      for (int t = 0; t < 4; ++t) {
        for (int y = 0; y < 5; ++y)
          for (int x = 0; x < 5; ++x)
            for (int q = 0; q < 4; ++q) {
              L.mfu.c[t][y][x][q] = (T)H.stenA[t][y][x][q];
              constexpr int kPack[4] = {0, 3, 1, 1};
              L.mfu.pk[t][y][x][q] = (T)H.stenA[t][y][x][kPack[q]];
            }
        for (int c = 0; c < 2; ++c) L.mfu.dinv[t][c] = (T)H.dinvAt[t][c];
      }
    } else if (H.mf) {
      L.mf_ok = true;
      L.mfl = mfree && H.N >= kMfo64MinN;
    }
    if (mfree && !pressure && H.N >= kMfo64MinN) L.mfo = make_mfop<T>(H);
  }
}

// Vectors of the levels and the matrices that the V-cycle reads, after
// build_coarse and select_mf: none on the coarsest level (dense product), on the
// fused levels and in the cluster (their own images; a count without a device takes
// the cluster for granted and so counts its levels here too), and not A where the
// level's product is matrix-free.  With the level-0 rows of the operator, which
// make_op leaves out likewise: 7.6 -> 4.4 GB on 512 cells in mixed precision with
// 60 basis vectors.
template <class T>
static void alloc_mg(Arena& ar, const HostSetup& hs, MG<T>& mg, bool tune, cudaStream_t s) {
  const bool pressure = mg.pressure;
  const int nl = (int)mg.lv.size();
  for (int l = 0; l < nl; ++l) {
    const FluidLevelHost& H = hs.levels[l];
    MGLevel<T>& L = mg.lv[l];
    const bool stored = l + 1 < nl && !L.mf && !(mg.cl.on && l >= mg.cl.lc && !ar.count_only);
    if (stored && !L.mfl && L.mfo.N == 0) {
      const SellHost sa = to_sell(pressure ? H.L : H.A);
      L.A = upload_sell<T>(ar, sa);
      if (tune && !ar.count_only) autotune_sell<T>(L.A, sa.soff[sa.nslices]);
    } else if (!(mg.cl.on && l >= mg.cl.lc)) {
      ar.spared += (long long)sell_bytes<T>(pressure ? H.L : H.A);
    }
    L.dinv = upload_as<T>(ar, pressure ? H.dinvL : H.dinvA);
    if (stored) {
      L.P = upload_sell<T>(ar, to_sell(pressure ? H.Pp : H.Pu));
      L.R = upload_sell<T>(ar, to_sell(pressure ? H.Rp : H.Ru));
      if (pressure) L.RA = upload_sell<T>(ar, to_sell(H.RAp));
    }
    L.x = ar.alloc<T>(L.n); L.x2 = ar.alloc<T>(L.n);
    if (l + 1 < nl) {
      L.b = ar.alloc<T>(L.n);
    } else {   // the coarsest right-hand side, padded to the rows' length with zeros for the dense product
      L.b = ar.alloc<T>(mg.coarse_ld);
      if (!ar.count_only) {
        CK(cudaMemsetAsync(L.b, 0, (size_t)mg.coarse_ld * sizeof(T), s));
        CK(cudaStreamSynchronize(s));
      }
    }
    if (stored && !pressure) L.r = ar.alloc<T>(L.n);
    L.d = ar.alloc<T>(L.n);
    if (H.mf && pressure) {
      std::vector<double> tab(kMfPresTab);
      for (int v = 0; v < 9; ++v)
        for (int y = 0; y < 3; ++y)
          for (int x = 0; x < 3; ++x)
            for (int q = 0; q < 9; ++q) tab[mf_pres_blk(v, y, x) + q] = H.stenL[v][y][x][q];
      for (int v = 0; v < 9; ++v)
        for (int k = 0; k < 3; ++k) tab[kMfPresDinv + 3 * v + k] = H.dinvLv[v][k];
      L.mftab = upload_as<T>(ar, tab);
    }
  }
}

// ------------------------------------------- cluster-resident coarse levels
constexpr size_t kClSmemCap = 227 * 1024;   // dynamic shared memory per CTA

// The shared-memory limit is a property of the kernel, shared by every
// problem alive in the process: always raise it to the cap.
template <class T, int B, bool TKRON>
static void cluster_kernel_setup() {
  auto kern = k_vcycle_cluster<T, B, TKRON>;
  CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmemCap));
  CK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
}

template <class T, int B, bool TKRON>
static int cluster_fits(size_t smem, int csize) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = csize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_vcycle_cluster<T, B, TKRON>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

// Cluster of 16 CTAs (non-portable size) when the device schedules one,
// else 8; nothing when neither fits (the per-level kernels run instead).
template <class T>
static void setup_cluster(Arena& ar, const HostSetup& hs, MG<T>& mg, bool pressure, int max_n) {
  int lc_min = 0;   // with max_n > 0 the cluster's finest level has at most max_n cells a side
  if (max_n > 0)
    while (lc_min + 1 < (int)mg.lv.size() && hs.levels[lc_min].N > max_n) ++lc_min;
  for (int cs : {16, 8}) {
    auto viable = [&](size_t smem) {
      if (ar.count_only) return true;
      if (pressure) {
        cluster_kernel_setup<T, 3, false>();
        return cluster_fits<T, 3, false>(smem, cs) > 0;
      }
      cluster_kernel_setup<T, 2, true>();
      return cluster_fits<T, 2, true>(smem, cs) > 0;
    };
    if (build_cluster<T>(ar, hs, pressure, mg, cs, kClSmemCap, viable, lc_min)) return;
  }
}

template <class T>
static void cluster_launch(MG<T>& mg, const T* in_b, T* out_x, cudaStream_t s) {
  ClArgs<T> a = mg.cl.args;
  a.in_b = in_b;
  a.out_x = out_x;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.csize);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = mg.cl.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = a.csize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = mg.pressure ? cudaLaunchKernelEx(&cfg, k_vcycle_cluster<T, 3, false>, a)
                                    : cudaLaunchKernelEx(&cfg, k_vcycle_cluster<T, 2, true>, a);
  if (e != cudaSuccess) throw CudaError(e, "cudaLaunchKernelEx (cluster V-cycle)");
}

// The finest levels, down to the first one that runs inside the cluster
// launch (or is the coarsest, or is below 16 cells a side), take the fused
// matrix-free kernels when the hierarchy is FP32 and the smoothing degree is
// at most kMfMaxDeg.
template <class T>
static void select_mf(MG<T>& mg, const HostSetup& hs, int mg_fused, bool count_only) {
  const int last = (int)mg.lv.size() - 1;
  if (mg_fused == -1 || !std::is_same<T, float>::value || mg.degree > kMfMaxDeg) return;
  bool any = false;
  for (int l = 0; l < last; ++l) {
    if (mg.cl.on && l >= mg.cl.lc) break;
    if (!mg.lv[l].mf_ok || hs.levels[l].N < 16) break;
    mg.lv[l].mf = true;
    any = true;
  }
  if (any && !count_only) {
    static std::once_flag once;
    std::call_once(once, [] {
      auto vel = [](auto tc) {
        for (int K = 1; K <= kMfMaxDeg; ++K)
          mf_with_degree(K, [&](auto kc) {
            constexpr int TC = decltype(tc)::value, KD = decltype(kc)::value;
            constexpr int ND = mf_threads_ud(TC), NU = mf_threads_uu(TC);
            CK(cudaFuncSetAttribute(k_mfu_down<float, TC, KD, ND, mf_minb_u(TC)>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)mfu_down_smem<float>(TC, KD)));
            CK(cudaFuncSetAttribute(k_mfu_up<float, TC, KD, NU, mf_minb_u(TC)>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)mfu_up_smem<float>(TC, KD)));
          });
      };
      auto pres_down = [](auto tp, auto mb) {
        for (int K = 1; K <= kMfMaxDeg; ++K)
          mf_with_degree(K, [&](auto kc) {
            constexpr int TP = decltype(tp)::value, KD = decltype(kc)::value, NT = mf_threads_p(TP);
            CK(cudaFuncSetAttribute(k_mfp_down<float, TP, KD, NT, decltype(mb)::value>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mfp_down_smem<float>(TP, KD)));
          });
      };
      auto pres_up = [](auto tp, auto mb) {
        for (int K = 1; K <= kMfMaxDeg; ++K)
          mf_with_degree(K, [&](auto kc) {
            constexpr int TP = decltype(tp)::value, KD = decltype(kc)::value, NT = mf_threads_p(TP);
            CK(cudaFuncSetAttribute(k_mfp_up<float, TP, KD, NT, decltype(mb)::value>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mfp_up_smem<float>(TP, KD)));
          });
      };
      for (int N : {32, 128, 256, 512}) {   // every kernel the maps choose
        mf_with_tile_u(N, vel);
        mf_with_launch_p<false>(N, pres_down);
        mf_with_launch_p<true>(N, pres_up);
      }
    });
  }
}

template <class T>
static MfCheb<T> mf_cheb(const MGLevel<T>& L, int degree) {
  MfCheb<T> c;
  c.k = degree;
  c.c0 = (T)L.ch.c0;
  for (int i = 0; i + 1 < degree; ++i) {
    c.c1[i] = (T)L.ch.c1[i];
    c.c2[i] = (T)L.ch.c2[i];
  }
  return c;
}

template <class T>
static T* vcycle(MG<T>& mg, int l, cudaStream_t s, T* out, const SpmvArgs<T>* fin = nullptr, bool* fused = nullptr);

// The down launch of fused level l: pre-smoothing from x0 = c0 D^-1 b, the
// residual and its restriction; the pre-smoothed iterate goes to L.x2, the
// coarse right-hand side to C.b (and the coarse smoother start when the next
// level runs the per-level sparse kernels).
static void mf_down_launch(MG<float>& mg, int l, const float* b, cudaStream_t s, const MfRes<float>* res = nullptr) {
  using T = float;
  const int last = (int)mg.lv.size() - 1;
  MGLevel<T>& L = mg.lv[l];
  MGLevel<T>& C = mg.lv[l + 1];
  const bool c_cluster = mg.cl.on && l + 1 == mg.cl.lc;
  const bool c_sell = !C.mf && !c_cluster && l + 1 != last;
  const int N = L.N, K = mg.degree;
  MfInit<T> ci;
  if (c_sell) { ci.x = C.x; ci.d = C.d; ci.dinv = C.dinv; ci.c0 = (T)C.ch.c0; }
  MfRes<T> r;
  if (res) {
    r = *res;
    std::memcpy(r.divB, L.divB, sizeof(r.divB));
  }
  if (mg.pressure) {
    MfPresArgs<T> a;
    a.N = N; a.tab = L.mftab; a.ch = mf_cheb(L, K);
    a.b = b; a.xout = L.x2; a.bc = C.b; a.ci = ci; a.res = r;
    mf_with_launch_p<false>(N, [&](auto tp, auto mb) {
      mf_with_degree(K, [&](auto kc) {
        constexpr int TP = decltype(tp)::value, KD = decltype(kc)::value, NT = mf_threads_p(TP);
        const unsigned g = nblk(N / 2, TP);
        launch(k_mfp_down<T, TP, KD, NT, decltype(mb)::value>, dim3(g, g), NT,
               mfp_down_smem<T>(TP, KD), s, a);
      });
    });
  } else {
    MfVelArgs<T> a;
    a.op = L.mfu; a.ch = mf_cheb(L, K);
    a.b = b; a.xout = L.x2; a.bc = C.b; a.ci = ci; a.res = r;
    mf_with_tile_u(N, [&](auto tc) {
      mf_with_degree(K, [&](auto kc) {
        constexpr int TC = decltype(tc)::value, KD = decltype(kc)::value, NT = mf_threads_ud(TC);
        const unsigned g = nblk(N, TC);
        launch(k_mfu_down<T, TC, KD, NT, mf_minb_u(TC)>, dim3(g, g), NT, mfu_down_smem<T>(TC, KD), s, a);
      });
    });
  }
}

// The up launch of fused level l: x = L.x2 + P xc, post-smoothing, result to
// dst (never L.x2), with the epilogue fin.
static void mf_up_launch(MG<float>& mg, int l, const float* b, const float* xc, float* dst, const MfFin<float>* fin,
                         cudaStream_t s) {
  using T = float;
  MGLevel<T>& L = mg.lv[l];
  if (dst == L.x2) throw std::logic_error("mf_up_launch: the result may not overwrite the pre-smoothed iterate");
  const int N = L.N, K = mg.degree;
  if (mg.pressure) {
    MfPresArgs<T> a;
    a.N = N; a.tab = L.mftab; a.ch = mf_cheb(L, K);
    a.b = b; a.xpre = L.x2; a.xc = xc; a.xout = dst;
    if (fin) a.fin = *fin;
    mf_with_launch_p<true>(N, [&](auto tp, auto mb) {
      mf_with_degree(K, [&](auto kc) {
        constexpr int TP = decltype(tp)::value, KD = decltype(kc)::value, NT = mf_threads_p(TP);
        const unsigned g = nblk(N, 2 * TP);
        launch(k_mfp_up<T, TP, KD, NT, decltype(mb)::value>, dim3(g, g), NT,
               mfp_up_smem<T>(TP, KD), s, a);
      });
    });
  } else {
    MfVelArgs<T> a;
    a.op = L.mfu; a.ch = mf_cheb(L, K);
    a.b = b; a.xpre = L.x2; a.xc = xc; a.xout = dst;
    if (fin) a.fin = *fin;
    mf_with_tile_u(N, [&](auto tc) {
      mf_with_degree(K, [&](auto kc) {
        constexpr int TC = decltype(tc)::value, KD = decltype(kc)::value, NT = mf_threads_uu(TC);
        const unsigned g = nblk(2 * N, 2 * TC);
        launch(k_mfu_up<T, TC, KD, NT, mf_minb_u(TC)>, dim3(g, g), NT, mfu_up_smem<T>(TC, KD), s, a);
      });
    });
  }
}

// One V-cycle from fused level l (mg.lv[l].mf) with right-hand side b: the
// down launch, the coarser levels, the up launch.  The result goes to `out`,
// else to L.x.  With res, the down launch starts from the Stokes residual
// (MfRes) and the up launch reads the right-hand side it wrote to res->bout.
template <class T>
static T* vcycle_mf(MG<T>& mg, int l, const T* b, cudaStream_t s, T* out, const MfFin<T>* fin,
                    const MfRes<T>* res = nullptr) {
  if constexpr (std::is_same<T, float>::value) {
    MGLevel<T>& L = mg.lv[l];
    MGLevel<T>& C = mg.lv[l + 1];
    T* dst = out ? out : L.x;
    mf_down_launch(mg, l, b, s, res);
    T* xc = C.mf ? vcycle_mf<T>(mg, l + 1, C.b, s, nullptr, nullptr) : vcycle<T>(mg, l + 1, s, (T*)nullptr);
    mf_up_launch(mg, l, res ? res->bout : b, xc, dst, fin, s);
    return dst;
  } else {
    throw std::logic_error("the fused levels are FP32 (select_mf)");
  }
}

// Algorithmic work of the fused launches of level l (not counting the work
// the tiles repeat on their overlaps): bytes of the vectors read and written
// once, and floating-point operations of the K operator applications (two per
// stored scalar entry), the transfer (two per entry of R or P) and the
// Chebyshev and epilogue updates (about six per unknown per step).
struct MfWork {
  double bytes = 0, flops = 0;
};
static MfWork mf_work(const HostSetup& hs, int l, bool pressure, bool up, int K, size_t tsize) {
  const FluidLevelHost& H = hs.levels[l];
  const FluidLevelHost& Hc = hs.levels[l + 1];
  const HostBlockMatrix& A = pressure ? H.L : H.A;
  const HostBlockMatrix& Tr = pressure ? (up ? H.Pp : H.Rp) : (up ? H.Pu : H.Ru);
  const double n = (double)A.nrows * A.BR, nc = pressure ? 3.0 * Hc.N * Hc.N : 2.0 * Hc.A.nrows;
  const double a_entries = (double)A.nnzb() * A.BR * A.BC;
  const double t_entries = (double)Tr.nnzb() * (Tr.kron ? Tr.BR : Tr.BR * Tr.BC);
  MfWork w;
  w.flops = K * 2.0 * a_entries + 2.0 * t_entries + 6.0 * K * n;
  w.bytes = up ? (3.0 * n + nc) * tsize : (2.0 * n + nc) * tsize;
  return w;
}

// Algorithmic work of one V-cycle of hierarchy mg from its finest level:
// the fused levels' launches (mf_work), the per-level sparse kernels of the
// other levels above the coarsest (2K applications of the stored level
// matrix and one residual, the transfers, a few vectors each), and the
// dense coarsest product (the inverse read once).
template <class T>
static MfWork vcycle_work(const HostSetup& hs, const MG<T>& mg, bool pressure) {
  MfWork w;
  const int last = (int)mg.lv.size() - 1, K = mg.degree;
  const double ts = sizeof(T);
  for (int l = 0; l < last; ++l) {
    if (mg.lv[l].mf) {
      for (bool up : {false, true}) {
        const MfWork m = mf_work(hs, l, pressure, up, K, sizeof(T));
        w.bytes += m.bytes;
        w.flops += m.flops;
      }
      continue;
    }
    const FluidLevelHost& H = hs.levels[l];
    const HostBlockMatrix& A = pressure ? H.L : H.A;
    const HostBlockMatrix& R = pressure ? H.Rp : H.Ru;
    const HostBlockMatrix& Pm = pressure ? H.Pp : H.Pu;
    const double n = (double)A.nrows * A.BR;
    const double a_bytes = (double)A.nnzb() * (A.NV * ts + 4.0);
    const double t_bytes = (double)(R.nnzb() * (R.NV * ts + 4.0) + Pm.nnzb() * (Pm.NV * ts + 4.0));
    const double a_flops = 2.0 * A.nnzb() * A.BR * A.BC;
    w.bytes += (2 * K + 1) * (a_bytes + 4.0 * n * ts) + t_bytes;
    w.flops += (2 * K + 1) * a_flops + 2.0 * (R.nnzb() + Pm.nnzb()) * (R.kron ? R.BR : R.BR * R.BC);
  }
  const double nc = mg.coarse_n, R = mg.sym.R;   // the inverse, or its four class matrices, once
  w.bytes += (R > 0 ? 4.0 * R * R : nc * mg.coarse_ld) * ts + 2.0 * nc * ts;
  w.flops += R > 0 ? 8.0 * R * R : 2.0 * nc * nc;
  return w;
}

template <class T>
static MfFin<T> mf_fin(const SpmvArgs<T>& f) {
  MfFin<T> m;
  m.sv = f.sv; m.smp = f.smp; m.sout = f.sout; m.snu = f.snu; m.srdt = f.srdt; m.acc = f.acc; m.omega = f.omega;
  return m;
}

// Level l input: L.b, with L.x = L.d = c0 dinv b already set (l < last).
// Result of the level is written to `out` (if given) or returned.  Levels
// from mg.cl.lc down run as one cluster launch when mg.cl.on.
// `fin`, when given, adds its Schur / accumulate epilogue (SpmvArgs sv ..
// omega) to the last smoothing step of level l; *fused tells whether it was
// applied (not when level l is solved by the cluster launch or densely).
template <class T>
static T* vcycle(MG<T>& mg, int l, cudaStream_t s, T* out, const SpmvArgs<T>* fin, bool* fused) {
  const int last = (int)mg.lv.size() - 1;
  MGLevel<T>& L = mg.lv[l];
  if (fused) *fused = false;
  if (L.mf) {  // fused levels need only L.b
    MfFin<T> mfin;
    if (fin) mfin = mf_fin(*fin);
    if (fused) *fused = fin != nullptr;
    return vcycle_mf<T>(mg, l, L.b, s, out, fin ? &mfin : nullptr);
  }
  if (mg.cl.on && l == mg.cl.lc) {
    T* dst = out ? out : L.x;
    cluster_launch<T>(mg, L.b, dst, s);
    return dst;
  }
  if (l == last) {
    if constexpr (sizeof(T) == 4) {
      if (mg.sym.R == 0) {
        launch(k_dense_mv<T>, nblk(mg.coarse_n, 8), 256, 0, s, mg.coarse_n, mg.coarse_ld, (const T*)mg.coarse_inv,
               (const T*)L.b, out ? out : L.x);
        return out ? out : L.x;
      }
    }
    launch(k_dense_sym<T>, nblk(mg.sym.R, sym_threads<T>() / 128), sym_threads<T>(),
           4 * (size_t)mg.sym_ld * sizeof(T), s, mg.sym, mg.sym_ld, (const T*)mg.sym_inv, (const T*)L.b, out ? out : L.x);
    return out ? out : L.x;
  }
  T* xc = L.x;
  T* xn = L.x2;
  const int k = mg.degree;
  for (int i = 1; i < k; ++i) {  // pre-smoothing, zero initial guess
    SpmvArgs<T> a;
    a.x = xc; a.y = xn; a.z = L.b; a.d = L.d; a.dinv = L.dinv;
    a.c1 = (T)L.ch.c1[i - 1]; a.c2 = (T)L.ch.c2[i - 1];
    level_launch(L, MODE_CHEB, a, s);
    std::swap(xc, xn);
  }
  MGLevel<T>& C = mg.lv[l + 1];
  if (L.RA.nrows == 0) {  // residual, then its restriction
    level_launch(L, MODE_AXPBY, axpby<T>(xc, L.r, L.b, (T)-1, (T)1), s);
    if (l + 1 == last || (mg.cl.on && l + 1 == mg.cl.lc)) {
      sell_launch(L.R, MODE_AXPBY, axpby<T>(L.r, C.b, nullptr, (T)1, (T)0), s);
    } else {
      SpmvArgs<T> a = axpby<T>(L.r, C.b, nullptr, (T)1, (T)0);
      a.d = C.d; a.dinv = C.dinv; a.xo = C.x; a.c2 = (T)C.ch.c0;
      sell_launch(L.R, MODE_INIT, a, s);
    }
  } else {  // the coarse right-hand side R (b - A x) = R b - (R A) x in one launch
    SpmvArgs<T> ra;
    ra.x = xc; ra.z = L.b; ra.y = C.b;
    if (l + 1 == last || (mg.cl.on && l + 1 == mg.cl.lc)) {
      resrestrict_launch(L.R, L.RA, MODE_AXPBY, ra, s);
    } else {
      ra.d = C.d; ra.dinv = C.dinv; ra.xo = C.x; ra.c2 = (T)C.ch.c0;
      resrestrict_launch(L.R, L.RA, MODE_INIT, ra, s);
    }
  }
  T* xcoarse = vcycle<T>(mg, l + 1, s, (T*)nullptr);
  sell_launch(L.P, MODE_AXPBY, axpby<T>(xcoarse, xc, xc, (T)1, (T)1), s);
  for (int i = 0; i < k; ++i) {  // post-smoothing
    SpmvArgs<T> a;
    T* dst = (i == k - 1 && out) ? out : xn;
    if (i == k - 1 && fin) {
      a.sv = fin->sv; a.smp = fin->smp; a.sout = fin->sout; a.snu = fin->snu; a.srdt = fin->srdt;
      a.acc = fin->acc; a.omega = fin->omega;
      if (fused) *fused = true;
    }
    a.x = xc; a.y = dst; a.z = L.b; a.d = L.d; a.dinv = L.dinv;
    if (i == 0) { a.c2 = (T)L.ch.c0; level_launch(L, MODE_CHEB0, a, s); }
    else { a.c1 = (T)L.ch.c1[i - 1]; a.c2 = (T)L.ch.c2[i - 1]; level_launch(L, MODE_CHEB, a, s); }
    if (dst == out) return out;
    std::swap(xc, xn);
  }
  return xc;
}

// ----------------------------------------------------------- preconditioner
template <class T>
struct Prec {
  MG<T> mgU, mgP;
  FullOp<T> op;          // operator in this precision (shares structure arrays)
  MfOp<T> mf;            // its fluid rows matrix-free (mf.N > 0)
  Sell<T> Cs, As;
  T* mpinv = nullptr;    // inverse P1disc mass diagonal
  T* csdinv = nullptr;   // inverse diagonal of the solid mass
  T* vin = nullptr;      // preconditioner input (n)
  T* zw = nullptr;       // preconditioner output (n)
  T *sb = nullptr, *sx = nullptr, *sx2 = nullptr, *sd = nullptr;  // solid work (2 nS)
  T* sd2 = nullptr;      // second direction buffer, when a mass solve takes several launches
  SolidPatches<T> sc;    // patches of the mass solves (fsi_solid_cheb.cuh); np = 0: one launch per step
  int sc_launches = 1;   // launches per mass solve
  Cheb chs;              // Chebyshev for D^-1 C_s on Wathen's interval ([1/2, 2] for P1)
  int cs_k = 16;
  // inner Richardson on the Stokes block: velocity right-hand side, residual
  // and correction, each [u (2 nU) | p (3 nP)]
  T *ru = nullptr, *t = nullptr, *dz = nullptr;
  int stokes_its = 1;
  T stokes_omega = 1;
  Sell<T> KT;            // nonlinear solid: the tangent as 2x2 blocks (pattern of the solid pair matrix)
};

struct Problem;
template <class T> static void precond_launch(Problem& P, Prec<T>& pr, cudaStream_t s);

// -------------------------------------------------------------- the problem
struct Problem {
  fsi_params prm{};
  int N = 0, nU = 0, nP = 0, nS = 0, nTri = 0, nPts = 0;
  size_t n = 0, offP = 0, offX = 0, offL = 0;
  cudaStream_t stream = nullptr, s2 = nullptr, s3 = nullptr, s4 = nullptr, s5 = nullptr;  // capture helpers
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr, ev_fork2 = nullptr, ev_join2 = nullptr;
  bool own_stream = false;
  bool by_counts = false;   // a footprint count without the mesh itself
  int device = 0;
  Arena ar;
  HostSetup hs;
  // operators
  FullOp<double> op64;
  FullOp<float> op32;
  Sell<double> M64, Cs64;
  // coupling
  int* tris = nullptr; double* area = nullptr; int* ntp = nullptr; int* nt = nullptr;
  int* l2n = nullptr; double* wall = nullptr;
  int* cell = nullptr; double* xi = nullptr; double* eta = nullptr;
  int cf_cap = 64;
  double* pairs = nullptr;   // exact rule: contributions per (triangle, cell) pair (k_exact_pairs), or none
  // nonlinear solid: reference gradients of the P1 basis per triangle (3 x 2),
  // tangent blocks in the slots of the solid pair matrix (4 per slot)
  double* tgrad = nullptr;
  double* kt64 = nullptr;
  float* kt32 = nullptr;
  int* cf_len = nullptr; int* cf_col = nullptr; double* cf_val = nullptr; float* cf_val32 = nullptr;
  double* cflift = nullptr;
  int* cft_ptr = nullptr; int* cft_col = nullptr; double* cft_val = nullptr; float* cft_val32 = nullptr;
  int* cft_cnt = nullptr; int* cft_cur = nullptr; int* scan_bsum = nullptr;
  // state
  double *x = nullptr, *b = nullptr, *uold = nullptr, *Xold = nullptr, *lift_u = nullptr, *w = nullptr;
  // Krylov
  int m = 200;
  double *V = nullptr, *H = nullptr, *cs = nullptr, *sn = nullptr, *g = nullptr, *y = nullptr, *part = nullptr;
  void* Z = nullptr;
  Ctl* ctl = nullptr;
  Ctl* ctl_host = nullptr;   // pinned mirror
  int red_blocks = 0;
  bool gs_cluster = false;   // the orthogonalisation runs as one cluster (small problems)
  // preconditioners
  Prec<double> p64;
  Prec<float> p32;
  // graphs
  cudaGraphExec_t g_assemble = nullptr, g_begin = nullptr, g_cycle = nullptr, g_finish = nullptr;
  cudaGraph_t gr_assemble = nullptr, gr_begin = nullptr, gr_cycle = nullptr, gr_finish = nullptr;
  // host-driven Arnoldi loop (FSI_HOST_LOOP=1): no conditional nodes, so that
  // per-kernel profilers can see the kernels; same kernels, one sync per iteration
  bool host_loop = false;
  cudaGraphExec_t g_cstart = nullptr, g_body = nullptr, g_cend = nullptr;
  cudaGraph_t gr_cstart = nullptr, gr_body = nullptr, gr_cend = nullptr;
  bool assembled = false;
  int kn_assemble = 0, kn_begin = 0, kn_cycle = 0, kn_body = 0, kn_finish = 0;  // kernel nodes per graph
};

// ------------------------------------------------------- solid block A_22^-1
// One mass solve C_s x = b by its patches: cs_k Chebyshev-Jacobi steps (the
// first one the start x = d = c0 D^-1 b) over sc_launches launches.  b is
// scale bsrc, or K kx - bsrc when kx is given.
template <class T, int W, int RPT>
static void solid_patch_kernel(const Prec<T>& pr, const SolidChebArgs<T>& a, cudaStream_t s) {
  launch(k_solid_cheb<T, W, RPT, sc_threads<T>()>, pr.sc.np, sc_threads<T>(), pr.sc.smem, s, a);
}

template <class T>
static void solid_patch_solve(Prec<T>& pr, const T* bsrc, T scale, const Sell<T>* K, const T* kx, T* out,
                              cudaStream_t s) {
  SolidChebArgs<T> a;
  a.P = pr.sc;
  a.c0 = (T)pr.chs.c0;
  a.dinv = pr.csdinv;
  a.bsrc = bsrc;
  a.scale = scale;
  if (K) a.K = *K;
  a.kx = kx;
  T *x[2] = {pr.sx, pr.sx2}, *d[2] = {pr.sd, pr.sd2};
  const int m = pr.cs_k - 1;
  int done = 0;
  for (int l = 0; l < pr.sc_launches; ++l) {
    a.ns = std::min(pr.sc.steps, m - done);
    a.first = l == 0;
    a.last = l + 1 == pr.sc_launches;
    for (int i = 0; i < a.ns; ++i) {
      a.c1[i] = (T)pr.chs.c1[done + i];
      a.c2[i] = (T)pr.chs.c2[done + i];
    }
    done += a.ns;
    a.xin = x[(l + 1) & 1];
    a.din = d[(l + 1) & 1];
    a.xout = a.last ? out : x[l & 1];
    a.dout = d[l & 1];
    if (pr.sc.width == 8 && pr.sc.rpt == 1) solid_patch_kernel<T, 8, 1>(pr, a, s);
    else if (pr.sc.width == 8) solid_patch_kernel<T, 8, 2>(pr, a, s);
    else if (pr.sc.rpt == 1) solid_patch_kernel<T, kScWide, 1>(pr, a, s);
    else solid_patch_kernel<T, kScWide, 2>(pr, a, s);
  }
}

// The patches of a problem's body on the device; none (np = 0) when the mesh
// does not suit or they take more than the counts' bound (planar growth of the
// planned patches, with room for rows of kScWide entries) or than the memory spared
// elsewhere (a body much finer than the grid).  A footprint by counts alone (no
// mesh) takes that most of them.
template <class T>
static void setup_solid_patches(Arena& ar, const HostSetup& hs, const double* ref_xy, bool by_counts, Prec<T>& pr) {
  constexpr bool f64 = std::is_same<T, double>::value;
  constexpr int NT = sc_threads<T>();
  const SolidPlan pl = plan_solid_patches(hs.Cs.nrows, pr.cs_k - 1, f64, 2 * NT);
  if (pl.np == 0) return;
  const double r = std::sqrt((double)hs.Cs.nrows / pl.np) + 2.0 * pl.steps;
  const double loc = pl.np * std::min((double)hs.Cs.nrows, r * r);
  const long long bound = (long long)(1.3 * loc * (kScWide * (sizeof(T) + 2) + 4)) + 4096 +
                          (pl.launches > 1 ? (long long)Arena::size<T>(2 * (size_t)hs.Cs.nrows) : 0);
  const long long room = std::max(0LL, std::min(bound, ar.spared));
  ar.spared -= room;
  if (by_counts) {
    ar.bytes += room;
    ar.peak = std::max(ar.peak, ar.bytes);
    return;
  }
  SolidPatchHost h;
  if (!build_solid_patches(hs.Cs, ref_xy, pr.cs_k - 1, f64, NT, h) ||
      4 * sizeof(T) * (size_t)h.max_loc > kClSmemCap)   // an outer layer too long for the iterate's two copies
    return;
  const size_t need = Arena::size<int>(h.poff.size()) + Arena::size<int>(h.cnt.size()) + Arena::size<int>(h.gid.size()) +
                      Arena::size<int>(h.roff.size()) + Arena::size<T>(h.val.size()) +
                      Arena::size<uint16_t>(h.col.size()) +
                      (h.launches > 1 ? Arena::size<T>(2 * (size_t)hs.Cs.nrows) : 0);
  if ((long long)need > room) return;
  SolidPatches<T>& d = pr.sc;
  d.np = h.np;
  d.steps = h.steps;
  d.width = h.width;
  d.rpt = h.max_rows > NT ? 2 : 1;
  d.smem = 4 * sizeof(T) * (size_t)h.max_loc;
  pr.sc_launches = h.launches;
  d.poff = ar.upload(h.poff);
  d.cnt = ar.upload(h.cnt);
  d.gid = ar.upload(h.gid);
  d.roff = ar.upload(h.roff);
  d.val = upload_as<T>(ar, h.val);
  d.col = ar.upload(h.col);
  if (h.launches > 1) pr.sd2 = ar.alloc<T>(2 * (size_t)hs.Cs.nrows);
  if (!ar.count_only && d.smem > 48 * 1024) {   // the limit belongs to the kernel: raise it to the cap
    const int cap = (int)kClSmemCap;
    CK(cudaFuncSetAttribute(k_solid_cheb<T, 8, 1, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    CK(cudaFuncSetAttribute(k_solid_cheb<T, 8, 2, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    CK(cudaFuncSetAttribute(k_solid_cheb<T, kScWide, 1, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    CK(cudaFuncSetAttribute(k_solid_cheb<T, kScWide, 2, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  }
}

// The mass solves' matrices: patches, or C_s itself for the per-step launches.
template <class T>
static void setup_mass_solves(Problem& P, Prec<T>& pr, const double* ref_xy) {
  setup_solid_patches<T>(P.ar, P.hs, ref_xy, P.by_counts, pr);
  if (pr.sc.np == 0) pr.Cs = upload_sell<T>(P.ar, to_sell(P.hs.Cs));
}

// Exact up to the two C_s solves (Chebyshev-Jacobi on [1/2, 2], Wathen's
// bounds for the Jacobi-scaled P1 mass matrix):
//   X = -dt C_s^-1 r_l,   lambda = C_s^-1 (A_s X - r_X),
// with r_l = v_l - C_f z_u for the block-triangular preconditioner.
template <class T>
static void solid_launch(Problem& P, Prec<T>& pr, cudaStream_t s) {
  const int n2 = 2 * P.nS;
  if (n2 == 0) return;
  const T* vX = pr.vin + P.offX;
  const T* vL = pr.vin + P.offL;
  T* zX = pr.zw + P.offX;
  T* zL = pr.zw + P.offL;
  const T dt = (T)P.prm.dt;
  const unsigned gcf = nblk(P.nS, 32);
  if (pr.sc.np > 0) {
    const T* bsrc = vL;
    T scale = -dt;
    if (P.prm.precond == 1) {  // lower block-triangular: -dt (v_l - C_f z_u)
      SpmvArgs<T> a;
      a.x = pr.zw; a.y = pr.sb; a.z = vL; a.alpha = dt; a.beta = -dt;
      launch(k_cf_apply<T>, gcf, 128, 0, s, P.nS, P.cf_cap, P.cf_len, P.cf_col, pr.op.cf_val, a, MODE_AXPBY);
      bsrc = pr.sb;
      scale = 1;
    }
    solid_patch_solve<T>(pr, bsrc, scale, nullptr, nullptr, zX, s);
    solid_patch_solve<T>(pr, vX, (T)1, P.prm.solid_law == 1 ? &pr.KT : &pr.As, zX, zL, s);
    return;
  }
  auto cheb_rest = [&](T* out) {
    T* xc = pr.sx;
    T* xn = pr.sx2;
    if (pr.cs_k == 1) { launch(k_copy<T>, nblk(n2, 256), 256, 0, s, n2, pr.sx, out); return; }
    for (int i = 1; i < pr.cs_k; ++i) {
      SpmvArgs<T> a;
      T* dst = (i == pr.cs_k - 1) ? out : xn;
      a.x = xc; a.y = dst; a.z = pr.sb; a.d = pr.sd; a.dinv = pr.csdinv;
      a.c1 = (T)pr.chs.c1[i - 1]; a.c2 = (T)pr.chs.c2[i - 1];
      sell_launch(pr.Cs, MODE_CHEB, a, s);
      std::swap(xc, xn);
    }
  };
  if (P.prm.precond == 1) {  // lower block-triangular: r_l = v_l - C_f z_u
    SpmvArgs<T> a;
    a.x = pr.zw; a.y = pr.sb; a.z = vL; a.alpha = dt; a.beta = -dt;
    a.d = pr.sd; a.dinv = pr.csdinv; a.xo = pr.sx; a.c2 = (T)pr.chs.c0;
    launch(k_cf_apply<T>, gcf, 128, 0, s, P.nS, P.cf_cap, P.cf_len, P.cf_col, pr.op.cf_val, a, MODE_INIT);
  } else {
    launch(k_cheb_first<T>, nblk(n2, 256), 256, 0, s, n2, vL, pr.csdinv, (T)pr.chs.c0, pr.sd, pr.sx, -dt, pr.sb);
  }
  cheb_rest(zX);
  SpmvArgs<T> a2;
  a2.x = zX; a2.y = pr.sb; a2.z = vX; a2.alpha = 1; a2.beta = -1;
  a2.d = pr.sd; a2.dinv = pr.csdinv; a2.xo = pr.sx; a2.c2 = (T)pr.chs.c0;
  sell_launch(P.prm.solid_law == 1 ? pr.KT : pr.As, MODE_INIT, a2, s);
  cheb_rest(zL);
}

// C_f^T applied to the multiplier part: y_u = z_u - C_f^T lambda (CSR over interior nodes)
template <class T>
__global__ void k_cft_sub(int nU, const int* __restrict__ ptr, const int* __restrict__ col, const T* __restrict__ val,
                          const T* __restrict__ lam, const T* __restrict__ zu, T* __restrict__ y) {
  pdl_begin();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nU) return;
  T a0 = zu[2 * r], a1 = zu[2 * r + 1];
  for (int k = ptr[r]; k < ptr[r + 1]; ++k) {
    const T v = val[k];
    const int c = col[k];
    a0 -= v * lam[2 * c];
    a1 -= v * lam[2 * c + 1];
  }
  y[2 * r] = a0;
  y[2 * r + 1] = a1;
}

// Pressure part of one application of the upper block-triangular Stokes
// approximation [[A_f, -B^T], [0, -S]]^-1: p = -S^-1 in_p with the
// Cahouet-Chabard Schur approximation S^-1 ~ nu M_p^-1 + (rho/dt) L_p^-1
// (one V-cycle on the pressure Laplacian L_p = B diag(M_f)^-1 B^T).
//
// With started = true the caller has already set L0.b = in_p and
// L0.x = L0.d = c0 D^-1 in_p (k_stokes_res does it); with acc, also
// acc += omega * out_p.  Both the Schur combination and the update ride on
// the last smoothing kernel of the finest pressure level when it is a
// per-level kernel.  With zu (fused finest level only) the input is the
// residual in_p - (-B) zu, formed by the finest down launch.
template <class T>
static void stokes_pressure(Problem& P, Prec<T>& pr, const T* in_p, T* out_p, cudaStream_t s, bool started = false,
                            T* acc = nullptr, T omega = 1, const T* zu = nullptr) {
  const int n3 = 3 * P.nP;
  MGLevel<T>& L0p = pr.mgP.lv[0];
  SpmvArgs<T> fin;
  fin.sv = in_p; fin.smp = pr.mpinv; fin.sout = out_p;
  fin.snu = (T)P.prm.nu; fin.srdt = (T)(P.prm.rho_f / P.prm.dt);
  fin.acc = acc; fin.omega = omega;
  if (L0p.mf) {  // the fused finest level reads in_p itself and applies the epilogue
    if (zu) {   // the Schur combination takes the residual the down launch wrote
      MfRes<T> r;
      r.zu = zu;
      r.bout = L0p.b;
      fin.sv = L0p.b;
      const MfFin<T> mfin = mf_fin(fin);
      vcycle_mf<T>(pr.mgP, 0, in_p, s, nullptr, &mfin, &r);
      return;
    }
    const MfFin<T> mfin = mf_fin(fin);
    vcycle_mf<T>(pr.mgP, 0, in_p, s, nullptr, &mfin);
    return;
  }
  if (zu) throw std::logic_error("stokes_pressure: the residual start needs the fused finest level");
  if (!started)
    launch(k_cheb_first<T>, nblk(n3, 256), 256, 0, s, n3, in_p, L0p.dinv, (T)L0p.ch.c0, L0p.d, L0p.x, (T)1, L0p.b);
  bool fused = false;
  T* sp = vcycle<T>(pr.mgP, 0, s, (T*)nullptr, &fin, &fused);
  if (!fused) {
    launch(k_schur<T>, nblk(n3, 256), 256, 0, s, n3, in_p, sp, pr.mpinv, (T)P.prm.nu, (T)(P.prm.rho_f / P.prm.dt),
           out_p);
    if (acc) launch(k_axpy<T>, nblk(n3, 256), 256, 0, s, (size_t)n3, omega, (const T*)out_p, acc);
  }
}

// Velocity part: u = A_f^-1 (in_u + B^T p) by one V-cycle with
// Chebyshev-Jacobi smoothing on the Q2 hierarchy (p = nullptr: u = A_f^-1 in_u).
// With acc, also acc += omega * out_u (on the last smoothing kernel when the
// finest level is a per-level kernel).  With zu (fused finest level only)
// the input is the residual in_u - A_f zu + B^T p.  On the fused level the
// finest down launch forms the input itself.
template <class T>
static void stokes_velocity(Problem& P, Prec<T>& pr, const T* in_u, const T* p, T* out_u, cudaStream_t s,
                            T* acc = nullptr, T omega = 1, const T* zu = nullptr) {
  MGLevel<T>& L0u = pr.mgU.lv[0];
  if (L0u.mf) {  // the fused finest level starts its smoother itself
    MfFin<T> mfin;
    mfin.acc = acc; mfin.omega = omega;
    if (p || zu) {
      MfRes<T> r;
      r.zu = zu;
      r.zp = p;
      r.bout = L0u.b;
      vcycle_mf<T>(pr.mgU, 0, in_u, s, out_u, acc ? &mfin : nullptr, &r);
    } else {
      vcycle_mf<T>(pr.mgU, 0, in_u, s, out_u, acc ? &mfin : nullptr);
    }
    return;
  }
  if (zu) throw std::logic_error("stokes_velocity: the residual start needs the fused finest level");
  if (p && L0u.mfo.N > 0) {   // FP64 only, as in level_launch
    if constexpr (std::is_same<T, double>::value)
      launch(k_mfv_start<T>, mfop_grid<T>(L0u.mfo.N), 128, 0, s, L0u.mfo, in_u, p, (const T*)L0u.dinv,
             (T)L0u.ch.c0, L0u.b, L0u.d, L0u.x);
  } else if (p) {
    SpmvArgs<T> a;
    a.x = p; a.y = L0u.b; a.z = in_u; a.alpha = -1; a.beta = 1;
    a.d = L0u.d; a.dinv = L0u.dinv; a.xo = L0u.x; a.c2 = (T)L0u.ch.c0;
    sell_launch(pr.op.Bt, MODE_INIT, a, s);
  } else {
    const int n2 = 2 * P.nU;
    launch(k_cheb_first<T>, nblk(n2, 256), 256, 0, s, n2, in_u, L0u.dinv, (T)L0u.ch.c0, L0u.d, L0u.x, (T)1, L0u.b);
  }
  SpmvArgs<T> fin;
  fin.acc = acc; fin.omega = omega;
  bool fused = false;
  vcycle(pr.mgU, 0, s, out_u, acc ? &fin : (const SpmvArgs<T>*)nullptr, &fused);
  if (acc && !fused) {
    const size_t n2 = 2 * (size_t)P.nU;
    launch(k_axpy<T>, nblk(n2, 256), 256, 0, s, n2, omega, (const T*)out_u, acc);
  }
}

// One application of the Stokes approximation to (in_u, in_p): the pressure
// part, then the velocity part with B^T p.  With split = true the pressure
// part runs on stream s4 beside the velocity part and the B^T p term is
// dropped (block-diagonal).
template <class T>
static void stokes_apply(Problem& P, Prec<T>& pr, const T* in_u, const T* in_p, T* out_u, T* out_p, cudaStream_t s,
                         bool split) {
  if (split) {
    CK(cudaEventRecord(P.ev_fork2, s));
    CK(cudaStreamWaitEvent(P.s4, P.ev_fork2, 0));
    stokes_pressure(P, pr, in_p, out_p, P.s4);
    CK(cudaEventRecord(P.ev_join2, P.s4));
    stokes_velocity(P, pr, in_u, (const T*)nullptr, out_u, s);
    CK(cudaStreamWaitEvent(s, P.ev_join2, 0));
  } else {
    stokes_pressure(P, pr, in_p, out_p, s);
    stokes_velocity(P, pr, in_u, (const T*)out_p, out_u, s);
  }
}

// Residual of the Stokes block at pr.zw for the right-hand side (vu, vp) into
// pr.t; with start, the pressure rows also start their V-cycle.
template <class T>
static void stokes_res_launch(Problem& P, Prec<T>& pr, const T* vu, const T* vp, bool start, cudaStream_t s) {
  MGLevel<T>& L = pr.mgP.lv[0];
  const T* dinv = start ? L.dinv : nullptr;
  T *b = start ? L.b : nullptr, *d = start ? L.d : nullptr, *x = start ? L.x : nullptr;
  if (pr.mf.N > 0) {
    const unsigned gU = mfop_grid<T>(pr.mf.N);
    launch(k_mf_stokes_res<T>, gU + nblk((size_t)P.nP * (3 / mfop_prows<T>()), 128), 128, 0, s, pr.mf, (int)gU, P.nU, P.nP, pr.zw, vu, vp, pr.t, dinv,
           (T)L.ch.c0, b, d, x);
  } else {
    launch(k_stokes_res<T>, pr.op.gU + pr.op.gP, 128, 0, s, pr.op, pr.zw, vu, vp, pr.t, dinv, (T)L.ch.c0, b, d, x);
  }
}

// y = alpha A x + beta z for the full operator; with Z, x is also stored as its
// column ctl->j.
template <class T, class TY>
static void full_launch(const Prec<T>& pr, const T* x, TY* y, const TY* z, TY alpha, TY beta, T* Z, size_t zld,
                        const Ctl* ctl, cudaStream_t s) {
  const FullOp<T>& op = pr.op;
  if (pr.mf.N > 0) {
    const unsigned gU = mfop_grid<T>(pr.mf.N), gP = nblk((size_t)op.nP * (3 / mfop_prows<T>()), 128);
    launch(k_fullmv_mf<T, TY>, gU + gP + op.gS, 128, 0, s, op, pr.mf, (int)gU, (int)gP, x, y, z, alpha, beta, Z, zld,
           ctl);
  } else {
    launch(k_fullmv<T, T, TY>, op.gU + op.gP + op.gS, 128, 0, s, op, x, y, z, alpha, beta, Z, zld, ctl);
  }
}

// One application z = P^-1 v of the block preconditioner (Section 5), input
// pr.vin, output pr.zw.
//   precond 0: diag(A_11, A_22)                      (block-diagonal)
//   precond 1: [[A_11, 0], [A_21, A_22]]             (block lower-triangular)
//   precond 2: [[A_11, A_12], [0, A_22]]             (block upper-triangular:
//              the solid block first, then the fluid with v_u - C_f^T z_l)
//   precond 3: as 2, velocity and pressure parts of A_11^-1 side by side.
// A_11^-1 is stokes_its steps of Richardson on the Stokes block, each step one
// application of stokes_apply (one step = the plain one-shot approximation).
template <class T>
static void precond_launch(Problem& P, Prec<T>& pr, cudaStream_t s) {
  const int pc = P.prm.precond;
  T* vp = pr.vin + P.offP;
  T* zp = pr.zw + P.offP;
  const bool split = (pc == 3);
  // the solid block does not depend on the fluid for precond 0, 2 and 3: run
  // it on a parallel branch (its kernels are small and latency-bound)
  if (pc != 1) {
    CK(cudaEventRecord(P.ev_fork, s));
    CK(cudaStreamWaitEvent(P.s3, P.ev_fork, 0));
    solid_launch(P, pr, P.s3);
    CK(cudaEventRecord(P.ev_join, P.s3));
  }
  const T* vu = pr.vin;
  if (pc == 2) {
    // the pressure part of the first Stokes application needs only v_p: it
    // runs beside the solid branch, and only the velocity part waits for z_l
    stokes_pressure(P, pr, vp, zp, s);
    CK(cudaStreamWaitEvent(s, P.ev_join, 0));
    launch(k_cft_sub<T>, nblk(P.nU, 128), 128, 0, s, P.nU, P.cft_ptr, P.cft_col, pr.op.cft_val, pr.zw + P.offL, pr.vin,
                                                  pr.ru);
    vu = pr.ru;
    stokes_velocity(P, pr, vu, (const T*)zp, pr.zw, s);
  } else {
    if (pc == 3) {
      CK(cudaStreamWaitEvent(s, P.ev_join, 0));
      launch(k_cft_sub<T>, nblk(P.nU, 128), 128, 0, s, P.nU, P.cft_ptr, P.cft_col, pr.op.cft_val, pr.zw + P.offL,
             pr.vin, pr.ru);
      vu = pr.ru;
    }
    stokes_apply(P, pr, vu, vp, pr.zw, zp, s, split);
  }
  const size_t nf = 2 * (size_t)P.nU + 3 * (size_t)P.nP;
  MGLevel<T>& L0p = pr.mgP.lv[0];
  for (int it = 1; it < pr.stokes_its; ++it) {
    if (split) {
      stokes_res_launch<T>(P, pr, vu, vp, false, s);
      stokes_apply(P, pr, pr.t, pr.t + P.offP, pr.dz, pr.dz + P.offP, s, split);
      launch(k_axpy<T>, nblk(nf, 256), 256, 0, s, nf, pr.stokes_omega, pr.dz, pr.zw);
    } else if (L0p.mf && pr.mgU.lv[0].mf && (double)pr.stokes_omega == 1.0) {
      // the Stokes residual formed inside the finest down launches: the
      // pressure correction from v_p - (-B) z_u, added to z_p; then, since
      // z_p then holds the corrected pressure (omega = 1), the velocity
      // correction from v_u - A_f z_u - (-B^T) z_p, which is the upper
      // triangular step's right-hand side t_u - (-B^T) dz_p
      stokes_pressure(P, pr, vp, pr.dz + P.offP, s, false, pr.zw + P.offP, pr.stokes_omega, (const T*)pr.zw);
      stokes_velocity(P, pr, vu, (const T*)(pr.zw + P.offP), pr.dz, s, pr.zw, pr.stokes_omega, (const T*)pr.zw);
    } else {
      // residual (starting the pressure smoother), then the pressure and
      // velocity corrections, each added to z by its own last kernel
      stokes_res_launch<T>(P, pr, vu, vp, !L0p.mf, s);
      stokes_pressure(P, pr, pr.t + P.offP, pr.dz + P.offP, s, true, pr.zw + P.offP, pr.stokes_omega);
      stokes_velocity(P, pr, pr.t, (const T*)(pr.dz + P.offP), pr.dz, s, pr.zw, pr.stokes_omega);
    }
  }
  if (pc == 1) solid_launch(P, pr, s);
  if (pc == 0) CK(cudaStreamWaitEvent(s, P.ev_join, 0));
}

// --------------------------------------------------------- Krylov kernels
// Reductions over the n unknowns use a fixed grid of nb CTAs of 256 threads;
// CTA b owns the sub-chunks b, b + nb, ... of CH rows, and the per-CTA partials
// are summed in a fixed order, so every result is deterministic.  n is even
// (three of the four segments are pairs and N is even), so every column of V
// starts on a 16-byte boundary and rows are taken in pairs.
//
// On GB300 these kernels are bound by the FP64 pipe (2 DFMA per clock per SM)
// when n is large, and by their chain of dependent round trips when it is
// small.  The multi-dot gives each warp whole vectors (eight 16-byte loads in
// flight per lane, one shuffle reduction per four vectors and CH rows).  At
// most kRedMaxBlocks CTAs write partials, so the last CTA sums at most 32
// values per lane and vector; with one partial per 512 rows that sum alone
// took 40 of the 186 us of pass 1 at N = 512.
constexpr int kRedMaxBlocks = 1024;
constexpr int kChunkSmall = 512;     // rows per sub-chunk up to 2^19 unknowns
constexpr int kChunkLarge = 1024;    // beyond: half as many shuffle reductions
static inline int red_chunk(size_t n) { return n <= ((size_t)1 << 19) ? kChunkSmall : kChunkLarge; }
static inline int red_grid(size_t n) {
  const size_t nsub = (n + red_chunk(n) - 1) / red_chunk(n);
  const size_t rounds = (nsub + kRedMaxBlocks - 1) / kRedMaxBlocks;
  return (int)((nsub + rounds - 1) / rounds);
}

// Sums of a, b, c, d over the warp, in lanes 0, 8, 16, 24: the four share the
// steps of one butterfly (6 additions, where four separate sums take 20; an
// FP64 instruction holds its pipe for 64 cycles on this part).
__device__ __forceinline__ double warp_sum4(double a, double b, double c, double d) {
  const int lane = threadIdx.x & 31;
  const bool hi = lane & 16, h8 = lane & 8;
  const double s0 = (hi ? c : a) + __shfl_xor_sync(0xffffffffu, hi ? a : c, 16);
  const double s1 = (hi ? d : b) + __shfl_xor_sync(0xffffffffu, hi ? b : d, 16);
  double s = (h8 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, h8 ? s0 : s1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// this lane's part of V[i] . ws over CH rows (nrow of them in the last chunk)
template <int CH>
__device__ __forceinline__ double dot_part(const double* __restrict__ v, const double* __restrict__ ws, int nrow) {
  const int lane = threadIdx.x & 31;
  const double2* __restrict__ v2 = reinterpret_cast<const double2*>(v);
  const double2* __restrict__ w2 = reinterpret_cast<const double2*>(ws);
  double a0 = 0, a1 = 0;
  if (nrow == CH) {
#pragma unroll
    for (int h = 0; h < CH / 512; ++h) {
      double2 x[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = v2[lane + 32 * (8 * h + q)];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const double2 w = w2[lane + 32 * (8 * h + q)];
        a0 += x[q].x * w.x;
        a1 += x[q].y * w.y;
      }
    }
  } else {
    for (int r = lane; 2 * r < nrow; r += 32) {
      const double2 x = v2[r], w = w2[r];
      a0 += x.x * w.x;
      a1 += x.y * w.y;
    }
  }
  return a0 + a1;
}

// acc[i] += V[i] . ws over the nrow rows from r0 (ws: nrow values in shared
// memory); warp w of the eight takes the vectors w, w + 8, ..., and only it
// touches their acc[i]
template <int CH>
__device__ __forceinline__ void mdot_warps(const double* __restrict__ V, size_t ld, int cnt,
                                           const double* __restrict__ ws, size_t r0, int nrow,
                                           double* __restrict__ acc) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  for (int i = wp; i < cnt; i += 32) {
    double a[4] = {0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i + 8 * q < cnt) a[q] = dot_part<CH>(V + (size_t)(i + 8 * q) * ld + r0, ws, nrow);
    const double s = warp_sum4(a[0], a[1], a[2], a[3]);
    const int mine = i + (lane & 24);
    if ((lane & 7) == 0 && mine < cnt) acc[mine] += s;
  }
}

// out[i] = sum over the nb CTAs of part[i nb + b]
__device__ __forceinline__ void finalize_warps(const double* __restrict__ part, int nb, int cnt,
                                               double* __restrict__ out) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  for (int i = wp; i < cnt; i += 32) {
    const double* __restrict__ p = part + (size_t)i * nb;
    double a[4] = {0, 0, 0, 0};
#pragma unroll 4
    for (int b = lane; b < nb; b += 32) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (i + 8 * q < cnt) a[q] += p[(size_t)(8 * q) * nb + b];
    }
    const double s = warp_sum4(a[0], a[1], a[2], a[3]);
    const int mine = i + (lane & 24);
    if ((lane & 7) == 0 && mine < cnt) out[mine] = s;
  }
}

// w - sum_i V[i] h[i] at the row pair r2 (rows 2 r2, 2 r2 + 1), eight columns
// in flight
__device__ __forceinline__ double2 gs_update(const double* __restrict__ V, size_t ld, int cnt, const double* hs,
                                             double2 w, size_t r2) {
  const double2* __restrict__ v = reinterpret_cast<const double2*>(V) + r2;
  const size_t l2 = ld >> 1;
  double s0 = 0, s1 = 0, t0 = 0, t1 = 0;
  int i = 0;
  for (; i + 7 < cnt; i += 8) {
    double2 x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = v[(size_t)(i + q) * l2];
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      s0 += x[q].x * hs[i + q];
      s1 += x[q].y * hs[i + q];
      t0 += x[q + 1].x * hs[i + q + 1];
      t1 += x[q + 1].y * hs[i + q + 1];
    }
  }
  if (i < cnt) {   // up to seven more, still all in flight at once
    double2 x[8];
#pragma unroll
    for (int q = 0; q < 7; ++q)
      if (i + q < cnt) x[q] = v[(size_t)(i + q) * l2];
#pragma unroll
    for (int q = 0; q < 7; ++q)
      if (i + q < cnt) {
        s0 += x[q].x * hs[i + q];
        s1 += x[q].y * hs[i + q];
      }
  }
  w.x -= s0 + t0;
  w.y -= s1 + t1;
  return w;
}

struct KrylovArgs {
  int n;
  int chunk;     // rows per sub-chunk of the reductions (red_chunk)
  size_t ld;
  const double* V;
  double* w;
  double* part;  // part[i * nb + block]
  double* h1;
  double* h2;
  double* H;
  double* cs;
  double* sn;
  double* g;
  Ctl* ctl;
  cudaGraphConditionalHandle cond;        // Arnoldi loop
  cudaGraphConditionalHandle cond_outer;  // restart / refinement loop
};

// Classical Gram-Schmidt with one refinement pass when needed (Daniel,
// Gragg, Kaufman and Stewart 1976; the "refine if needed" rule of PETSc's
// GMRES): pass 1 forms h1 = V^T w and ||w||; pass 2 updates w -= V h1, forms
// ||w|| and already the second projection h2 = V^T w, while the CTA's part
// of V is still in its L1; if the norm fell below ||w|| / sqrt(2), pass 3
// subtracts w -= V h2 (it returns at once otherwise).  Forming h2 in pass 2
// replaces a pass of its own (launch, reduction and a third read of V) in
// the refined steps, which a preconditioner that works makes the common ones:
// A z_j is then close to v_j and most of w cancels.

// Hessenberg column j, Givens rotation, residual estimate and the stop
// decision of the Arnoldi loop, by one whole CTA.  An FP64 instruction of a
// warp holds its pipe for 64 cycles here whatever its active lanes, so what
// does not depend on the recurrence runs on all lanes at once: of the earlier
// rotations only a' = c b - s a is a chain (one multiply-add per rotation, the
// products c b formed before, the rotated entries after), the two square roots
// share one instruction sequence and so do the three quotients.  Written for
// one thread with every step a global read, a hypot and three divisions, this
// made pass 2 15 us at N = 16, where its data is nothing.  Pass 1 / pass 2 or 4
// / the least squares at j = 10 went from 10.7 / 15.3 / 10 to 7.2 / 13 / 2.7 us
// at N = 24 (pass 2 now with the second projection), from 186 / 138 / - to 119 /
// 228 us at N = 512, where the former pass 3 took 159.
struct ArnoldiShared {
  double h[256], cb[256], ns[256], a[256];   // column, c b, -s, partly rotated a
};
// this thread's inputs of the Givens step, read by every CTA while it waits
// for its rows anyway: only one CTA needs them, at the very end
struct ArnoldiIn {
  double h1 = 0, cs = 0, sn = 0, g = 0;
};
__device__ __forceinline__ ArnoldiIn arnoldi_load(const KrylovArgs& k, int j) {
  const int t = threadIdx.x;   // j < 250 <= the CTA's threads
  ArnoldiIn in;
  if (t <= j) in.h1 = k.h1[t];
  if (t < j) {
    in.cs = k.cs[t];
    in.sn = k.sn[t];
  }
  if (t == 0) in.g = k.g[j];
  return in;
}

__device__ __forceinline__ void arnoldi_finish(const KrylovArgs& k, ArnoldiShared& sh, const ArnoldiIn& in, int j,
                                               const double* h2s, double s2) {
  Ctl* c = k.ctl;
  const int m1 = c->m + 1, t = threadIdx.x;
  const double cst = in.cs, snt = in.sn;
  if (t <= j) sh.h[t] = in.h1 + (h2s ? h2s[t] : 0.0);
  if (t < j) sh.ns[t] = -snt;
  __syncthreads();
  if (t < j) sh.cb[t] = cst * sh.h[t + 1];
  __syncthreads();
  if (t < 32) {
    double a = sh.h[0];
    for (int i = 0; i < j; ++i) {
      if (t == 0) sh.a[i] = a;
      a = fma(sh.ns[i], a, sh.cb[i]);
    }
    // r = sqrt(a^2 + ||w||^2) in lane 0, ||w|| in lane 1
    const double root = sqrt(t == 0 ? fma(a, a, s2) : s2);
    const double r = __shfl_sync(0xffffffffu, root, 0), nrm = __shfl_sync(0xffffffffu, root, 1);
    // a / r, ||w|| / r, 1 / ||w||
    const double quo = (t == 0 ? a : (t == 1 ? nrm : 1.0)) / (t <= 1 ? r : nrm);
    const double q0 = __shfl_sync(0xffffffffu, quo, 0), q1 = __shfl_sync(0xffffffffu, quo, 1);
    const double q2 = __shfl_sync(0xffffffffu, quo, 2);
    if (t == 0) {
      const double gj = in.g;
      const double cc = (r > 0) ? q0 : 1.0, ss = (r > 0) ? q1 : 0.0;
      k.cs[j] = cc;
      k.sn[j] = ss;
      const double gn = -ss * gj;
      k.g[j + 1] = gn;
      k.g[j] = cc * gj;
      k.H[(size_t)j * m1 + j] = r;
      k.H[(size_t)j * m1 + j + 1] = 0.0;
      const double res = fabs(gn);
      const int its = c->its + 1;
      c->its = its;
      c->res = res;
      bool stop = false;
      if (!(res == res) || !(nrm == nrm)) { c->flags |= FLAG_NAN; stop = true; c->j = j; }
      else if (r == 0.0) { c->flags |= FLAG_BREAKDOWN; stop = true; c->j = j; }
      else {
        c->j = j + 1;
        if (res <= c->cycle_tol || j + 1 >= c->m || its >= c->max_it || nrm == 0.0) stop = true;
      }
      c->scale = (nrm > 0.0) ? q2 : 0.0;
      c->cyc_active = stop ? 0 : 1;
      if (k.cond) cudaGraphSetConditional(k.cond, stop ? 0u : 1u);
    }
  }
  __syncthreads();
  if (t < j) k.H[(size_t)j * m1 + t] = cst * sh.a[t] + snt * sh.h[t + 1];
}

// rows of sub-chunk `sub` into ws (shared); the number of rows
template <int CH>
__device__ __forceinline__ int load_chunk(const KrylovArgs& k, int sub, double* ws) {
  const size_t r0 = (size_t)sub * CH;
  const int nrow = (int)min((size_t)CH, (size_t)k.n - r0);
  const double2* __restrict__ w = reinterpret_cast<const double2*>(k.w + r0);
  for (int r = threadIdx.x; 2 * r < nrow; r += blockDim.x) reinterpret_cast<double2*>(ws)[r] = w[r];
  return nrow;
}

// pass 1: h1 = V[0..j]^T w and ||w||^2
template <int CH>
__global__ void __launch_bounds__(kRedThreads, 3) k_gs1(KrylovArgs k) {
  pdl_begin();
  __shared__ __align__(16) double ws[CH];
  __shared__ double acc[256 + 1];
  const int cnt = k.ctl->j + 1, nb = gridDim.x;
  for (int i = threadIdx.x; i <= cnt; i += blockDim.x) acc[i] = 0;
  const int nsub = (k.n + CH - 1) / CH, lane = threadIdx.x & 31;
  for (int sub = blockIdx.x; sub < nsub; sub += nb) {
    __syncthreads();
    const int nrow = load_chunk<CH>(k, sub, ws);
    __syncthreads();
    if (threadIdx.x >= kRedThreads - 32) {   // the last warp (fewest vectors): w . w
      double a = 0;
      for (int r = lane; r < nrow; r += 32) a += ws[r] * ws[r];
      a = warp_sum(a);
      if (lane == 0) acc[cnt] += a;
    }
    mdot_warps<CH>(k.V, k.ld, cnt, ws, (size_t)sub * CH, nrow, acc);
  }
  __syncthreads();
  for (int i = threadIdx.x; i <= cnt; i += blockDim.x) k.part[(size_t)i * nb + blockIdx.x] = acc[i];
  if (last_block(&k.ctl->counter[0])) {
    finalize_warps(k.part, nb, cnt + 1, k.h1);
    if (threadIdx.x == 0) k.ctl->counter[0] = 0;
  }
}

// pass 2: w -= V h1, ||w||^2 and h2 = V^T w; finish the step or ask for the
// refinement (h1[cnt] is ||w||^2 of pass 1)
template <int CH>
__global__ void __launch_bounds__(kRedThreads, 3) k_gs2(KrylovArgs k) {
  pdl_begin();
  __shared__ __align__(16) double ws[CH];
  __shared__ double hs[256], acc[256], sm[32];
  __shared__ ArnoldiShared ash;
  __shared__ double s2s;
  const int j = k.ctl->j, cnt = j + 1, nb = gridDim.x;
  const ArnoldiIn in = arnoldi_load(k, j);
  const double wn2 = threadIdx.x == 0 ? k.h1[cnt] : 0.0;
  if (threadIdx.x < cnt) {
    hs[threadIdx.x] = in.h1;
    acc[threadIdx.x] = 0;
  }
  const int nsub = (k.n + CH - 1) / CH;
  double nacc = 0;
  for (int sub = blockIdx.x; sub < nsub; sub += nb) {
    __syncthreads();
    const size_t r0 = (size_t)sub * CH;
    const int nrow = (int)min((size_t)CH, (size_t)k.n - r0);
    double2* w2 = reinterpret_cast<double2*>(k.w + r0);
    for (int r = threadIdx.x; 2 * r < nrow; r += blockDim.x) {
      const double2 v = gs_update(k.V, k.ld, cnt, hs, w2[r], (r0 >> 1) + r);
      w2[r] = v;
      reinterpret_cast<double2*>(ws)[r] = v;
      nacc += v.x * v.x + v.y * v.y;
    }
    __syncthreads();
    mdot_warps<CH>(k.V, k.ld, cnt, ws, r0, nrow, acc);
  }
  const double bs = block_sum(nacc, sm);
  if (threadIdx.x == 0) k.part[(size_t)cnt * nb + blockIdx.x] = bs;
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) k.part[(size_t)i * nb + blockIdx.x] = acc[i];
  if (last_block(&k.ctl->counter[1])) {
    finalize_warps(k.part, nb, cnt + 1, k.h2);
    __syncthreads();
    if (threadIdx.x == 0) {
      Ctl* c = k.ctl;
      c->counter[1] = 0;
      const double s2 = k.h2[cnt];
      c->refine = (s2 < 0.5 * wn2) ? 1 : 0;
      if (c->refine) c->refines += 1;
      s2s = c->refine ? -1.0 : s2;
    }
    __syncthreads();
    // -1 marks the refinement; a NaN norm is not below any bound and finishes here
    if (s2s != -1.0) arnoldi_finish(k, ash, in, j, nullptr, s2s);
  }
}

// pass 3 (refinement only): w -= V h2, ||w||^2, finish the step
template <int CH>
__global__ void __launch_bounds__(kRedThreads, 3) k_gs3(KrylovArgs k) {
  pdl_begin();
  __shared__ double hs[256], sm[32];
  __shared__ ArnoldiShared ash;
  __shared__ double s2s;
  const int refine = k.ctl->refine, j = k.ctl->j, cnt = j + 1, nb = gridDim.x;
  if (!refine) return;
  const ArnoldiIn in = arnoldi_load(k, j);
  if (threadIdx.x < cnt) hs[threadIdx.x] = k.h2[threadIdx.x];
  __syncthreads();
  const int nsub = (k.n + CH - 1) / CH;
  double nacc = 0;
  for (int sub = blockIdx.x; sub < nsub; sub += nb) {
    const size_t r0 = (size_t)sub * CH;
    const int nrow = (int)min((size_t)CH, (size_t)k.n - r0);
    double2* w2 = reinterpret_cast<double2*>(k.w + r0);
    for (int r = threadIdx.x; 2 * r < nrow; r += blockDim.x) {
      const double2 v = gs_update(k.V, k.ld, cnt, hs, w2[r], (r0 >> 1) + r);
      w2[r] = v;
      nacc += v.x * v.x + v.y * v.y;
    }
  }
  const double bs = block_sum(nacc, sm);
  if (threadIdx.x == 0) k.part[blockIdx.x] = bs;
  if (last_block(&k.ctl->counter[2])) {
    double a = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) a += k.part[b];
    const double s2 = block_sum(a, sm);
    if (threadIdx.x == 0) {
      k.ctl->counter[2] = 0;
      s2s = s2;
    }
    __syncthreads();
    arnoldi_finish(k, ash, in, j, hs, s2s);
  }
}

// The next basis vector V[j] = w * scale (j already advanced, or 0 at the
// start of a cycle), and with it the preconditioner's input in its precision.
template <class T>
__global__ void k_basis(int n2, double* __restrict__ V, size_t ld, const double* __restrict__ w, T* __restrict__ vin,
                        const Ctl* ctl) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n2) return;
  const double sc = ctl->scale;
  double2 v = reinterpret_cast<const double2*>(w)[i];
  v.x *= sc;
  v.y *= sc;
  reinterpret_cast<double2*>(V + (size_t)ctl->j * ld)[i] = v;
  typename Vec2<T>::type o;
  o.x = (T)v.x;
  o.y = (T)v.y;
  reinterpret_cast<typename Vec2<T>::type*>(vin)[i] = o;
}

// The whole orthogonalisation of a small problem in one launch: a cluster of 16
// CTAs holds w in registers, sums its dots through distributed shared memory,
// and goes through the same passes (h1 and ||w||, the update with h2, the
// refinement if needed, the Givens step, the next basis vector) with cluster
// barriers between them.  As launches, the passes of a 7400-unknown problem take
// 33 us, nearly all of it launch boundaries, last-block hand-overs and the
// FP64 latency of their reductions; 16 SMs hold the FP64 work of up to 512 rows
// each (kGsClusterRows) in about the time the hand-overs take, in short cycles.
// Rows are worked by four warps, one per SM quarter: an FP64 instruction holds
// a quarter's pipe for 64 cycles, so more warps would only repeat the butterflies.
constexpr int kGsCluster = 16;
constexpr int kGsWorkers = 128;                       // threads that own row pairs
constexpr int kGsPairs = 2;                           // row pairs of one of them, at most
constexpr int kGsClusterRows = 2 * kGsWorkers * kGsPairs;

struct GsClusterShared {
  double red[4][260];          // per-warp sums
  double part[3][260];         // this CTA's sums, read by the whole cluster
  double h1[256], h2[260];     // the cluster's sums
  double scale;
};

// sums of v over the cluster's CTAs: out[i] = sum_r part_r[i], i < cnt
__device__ __forceinline__ void gs_cluster_gather(cg::cluster_group& cl, double* part, int cnt, double* out) {
  const int r = threadIdx.x & 15;
  const double* remote = cl.map_shared_rank(part, r);
  for (int i0 = threadIdx.x >> 4; i0 - (int)(threadIdx.x >> 4) < cnt; i0 += 2 * (kRedThreads / 16)) {
    const int i1 = i0 + kRedThreads / 16;
    double a = i0 < cnt ? remote[i0] : 0.0, b = i1 < cnt ? remote[i1] : 0.0;
    // two sums share the butterfly over 16 lanes: a in lanes 0-7, b in 8-15
    const bool hi = r & 8;
    double s = (hi ? b : a) + __shfl_xor_sync(0xffffffffu, hi ? a : b, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (r == 0 && i0 < cnt) out[i0] = s;
    if (r == 8 && i1 < cnt) out[i1] = s;
  }
}

// dots of this CTA's rows with V[0 .. cnt-1] and their sum of squares (entry
// cnt), into part; every thread of the CTA calls it
__device__ __forceinline__ void gs_cluster_dots(const double2* __restrict__ v0, size_t l2, int cnt, int np,
                                                const double2* w, GsClusterShared& sh, double* part, bool dots) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (threadIdx.x < kGsWorkers) {
    double nn = 0;
#pragma unroll
    for (int u = 0; u < kGsPairs; ++u) {
      nn = fma(w[u].x, w[u].x, nn);
      nn = fma(w[u].y, w[u].y, nn);
    }
    for (int i = 0; i < (dots ? cnt : 0) + 1; i += 4) {   // one slot past the vectors: the sum of squares
      double a[4] = {0, 0, 0, 0};
      const int nv = dots ? cnt : 0;
#pragma unroll
      for (int u = 0; u < kGsPairs; ++u) {
        const int r = threadIdx.x + kGsWorkers * u;
        if (r >= np) break;
        double2 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (i + q < nv) x[q] = v0[(size_t)(i + q) * l2 + r];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (i + q < nv) a[q] = fma(x[q].y, w[u].y, fma(x[q].x, w[u].x, a[q]));
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (i + q == nv) a[q] = nn;
      const double s = warp_sum4(a[0], a[1], a[2], a[3]);
      const int mine = i + (lane >> 3);
      if ((lane & 7) == 0 && mine <= nv) sh.red[wp][mine] = s;
    }
  }
  __syncthreads();
  const int nv = dots ? cnt : 0;
  for (int i = threadIdx.x; i <= nv; i += kRedThreads)
    part[i] = (sh.red[0][i] + sh.red[1][i]) + (sh.red[2][i] + sh.red[3][i]);
}

template <class T>
__global__ void __launch_bounds__(kRedThreads) k_gs_cluster(KrylovArgs k, double* __restrict__ V, T* __restrict__ vin) {
  pdl_begin();
  __shared__ GsClusterShared sh;
  __shared__ ArnoldiShared ash;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), t = threadIdx.x;
  const int j = k.ctl->j, cnt = j + 1;
  const ArnoldiIn in = [&] {
    ArnoldiIn v;
    if (rank == 0) {
      if (t < j) {
        v.cs = k.cs[t];
        v.sn = k.sn[t];
      }
      if (t == 0) v.g = k.g[j];
    }
    return v;
  }();
  const int n2 = k.n / 2, per = (n2 + kGsCluster - 1) / kGsCluster;   // row pairs of a CTA
  const int p0 = min(n2, rank * per), np = min(n2, p0 + per) - p0;
  const size_t l2 = k.ld >> 1;
  const double2* __restrict__ v0 = reinterpret_cast<const double2*>(k.V) + p0;
  double2 w[kGsPairs];
#pragma unroll
  for (int u = 0; u < kGsPairs; ++u) {
    const int r = t + kGsWorkers * u;
    w[u].x = w[u].y = 0;
    if (t < kGsWorkers && r < np) w[u] = reinterpret_cast<const double2*>(k.w)[p0 + r];
  }
  auto update = [&](const double* h) {
    if (t >= kGsWorkers) return;
    for (int i = 0; i < cnt; i += 4) {
#pragma unroll
      for (int u = 0; u < kGsPairs; ++u) {
        const int r = t + kGsWorkers * u;
        if (r >= np) break;
        double2 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (i + q < cnt) x[q] = v0[(size_t)(i + q) * l2 + r];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (i + q < cnt) {
            w[u].x = fma(-h[i + q], x[q].x, w[u].x);
            w[u].y = fma(-h[i + q], x[q].y, w[u].y);
          }
      }
    }
  };
  gs_cluster_dots(v0, l2, cnt, np, w, sh, sh.part[0], true);
  cl.sync();
  gs_cluster_gather(cl, sh.part[0], cnt + 1, sh.h2);
  __syncthreads();
  const double wn2 = sh.h2[cnt];
  if (t < cnt) sh.h1[t] = sh.h2[t];
  __syncthreads();
  update(sh.h1);
  gs_cluster_dots(v0, l2, cnt, np, w, sh, sh.part[1], true);
  cl.sync();
  gs_cluster_gather(cl, sh.part[1], cnt + 1, sh.h2);
  __syncthreads();
  double s2 = sh.h2[cnt];
  const bool refine = s2 < 0.5 * wn2;   // the same numbers in every CTA
  if (refine) {
    update(sh.h2);
    gs_cluster_dots(v0, l2, cnt, np, w, sh, sh.part[2], false);
    cl.sync();
    gs_cluster_gather(cl, sh.part[2], 1, sh.h2 + 258);
    __syncthreads();
    s2 = sh.h2[258];
  }
  if (t == 0) {
    const double nrm = sqrt(s2);
    sh.scale = (nrm > 0.0) ? 1.0 / nrm : 0.0;
  }
  __syncthreads();
  if (t < kGsWorkers) {
    const double sc = sh.scale;
    using T2 = typename Vec2<T>::type;
    double2* vn = reinterpret_cast<double2*>(V + (size_t)(j + 1) * k.ld) + p0;
#pragma unroll
    for (int u = 0; u < kGsPairs; ++u) {
      const int r = t + kGsWorkers * u;
      if (r >= np) break;
      double2 x = w[u];
      x.x *= sc;
      x.y *= sc;
      vn[r] = x;
      T2 o;
      o.x = (T)x.x;
      o.y = (T)x.y;
      reinterpret_cast<T2*>(vin)[p0 + r] = o;
    }
  }
  if (rank == 0) {
    if (t == 0) {
      k.ctl->refine = refine ? 1 : 0;
      if (refine) k.ctl->refines += 1;
    }
    ArnoldiIn a = in;
    if (t <= j) a.h1 = sh.h1[t];
    arnoldi_finish(k, ash, a, j, refine ? sh.h2 : nullptr, s2);
  }
  cl.sync();   // no CTA leaves while another may still read its sums
}

// start of a cycle: beta = ||w|| with w = b - A x already formed
__global__ void __launch_bounds__(kRedThreads) k_cycle_start(KrylovArgs k) {
  pdl_begin();
  __shared__ double sm[32];
  double acc = 0;
  for (size_t r0 = (size_t)blockIdx.x * k.chunk; r0 < (size_t)k.n; r0 += (size_t)gridDim.x * k.chunk)
    for (size_t r = r0 + threadIdx.x; r < min((size_t)k.n, r0 + k.chunk); r += blockDim.x) acc += k.w[r] * k.w[r];
  acc = block_sum(acc, sm);
  if (threadIdx.x == 0) k.part[blockIdx.x] = acc;
  if (last_block(&k.ctl->counter[3])) {
    double a = 0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) a += k.part[b];
    const double s2 = block_sum(a, sm);
    if (threadIdx.x == 0) {
      Ctl* c = k.ctl;
      c->counter[3] = 0;
      const double beta = sqrt(s2);
      c->beta = beta;
      c->j = 0;
      c->cycles += 1;
      k.g[0] = beta;
      c->last_true = (c->bnorm > 0) ? beta / c->bnorm : beta;
      bool stop = false;
      if (!(beta == beta)) { c->flags |= FLAG_NAN; stop = true; }
      c->converged = (beta <= c->target) ? 1 : 0;
      if (c->converged || c->its >= c->max_it || c->cycles > c->max_cycles ||
          (c->flags & (FLAG_NAN | FLAG_BREAKDOWN)) || c->aflags)
        stop = true;
      c->stop = stop ? 1 : 0;
      c->cycle_tol = fmax(c->inner_rtol * beta, c->target);
      c->scale = (beta > 0) ? 1.0 / beta : 0.0;
      c->res = beta;
      c->cyc_active = stop ? 0 : 1;
      if (k.cond) cudaGraphSetConditional(k.cond, stop ? 0u : 1u);
      if (k.cond_outer) cudaGraphSetConditional(k.cond_outer, stop ? 0u : 1u);
    }
  }
}

// ||b||, the target, and reset of the per-solve counters
__global__ void __launch_bounds__(kRedThreads) k_solve_begin(KrylovArgs k, const double* __restrict__ b, double rtol,
                                                             double inner_rtol, int max_it, int m, int max_cycles) {
  pdl_begin();
  __shared__ double sm[32];
  double acc = 0;
  for (size_t r0 = (size_t)blockIdx.x * k.chunk; r0 < (size_t)k.n; r0 += (size_t)gridDim.x * k.chunk)
    for (size_t r = r0 + threadIdx.x; r < min((size_t)k.n, r0 + k.chunk); r += blockDim.x) acc += b[r] * b[r];
  acc = block_sum(acc, sm);
  if (threadIdx.x == 0) k.part[blockIdx.x] = acc;
  if (last_block(&k.ctl->counter[4])) {
    double a = 0;
    for (int bb = threadIdx.x; bb < (int)gridDim.x; bb += blockDim.x) a += k.part[bb];
    const double s2 = block_sum(a, sm);
    if (threadIdx.x == 0) {
      Ctl* c = k.ctl;
      c->counter[4] = 0;
      c->bnorm = sqrt(s2);
      c->target = rtol * c->bnorm;
      c->inner_rtol = inner_rtol;
      c->its = 0; c->cycles = 0; c->j = 0; c->flags = 0; c->refines = 0; c->refine = 0;
      c->converged = 0; c->stop = 0;
      c->max_it = max_it; c->m = m; c->max_cycles = max_cycles;
    }
  }
}

// least squares on the rotated Hessenberg matrix: y = R^-1 g by one warp.
// Column-oriented back substitution: lane l holds the right-hand sides l,
// l + 32, ... and the reciprocals of their diagonals (all taken at once); each
// solved entry is broadcast and its column, the next one already loading,
// subtracted from the entries above.  So a step is one multiplication and one
// multiply-add deep.  (One thread walking the rows, with a dependent global
// read per entry and a division per row, took 10 us at 10 entries.)
constexpr int kLsqRows = 8;   // 32 * 8 >= the largest restart
__global__ void __launch_bounds__(32) k_lsq(const double* __restrict__ H, const double* __restrict__ g,
                                            double* __restrict__ y, const Ctl* ctl) {
  pdl_begin();
  const int lane = threadIdx.x;
  const int kk = ctl->j, m1 = ctl->m + 1;
  double v[kLsqRows], inv[kLsqRows], c[kLsqRows];
#pragma unroll
  for (int q = 0; q < kLsqRows; ++q) {
    const int r = lane + 32 * q;
    v[q] = inv[q] = c[q] = 0.0;
    if (32 * q < kk) {
      if (r < kk) {
        v[q] = g[r];
        inv[q] = 1.0 / H[(size_t)r * m1 + r];
        if (r < kk - 1) c[q] = H[(size_t)(kk - 1) * m1 + r];
      }
    }
  }
#pragma unroll
  for (int b = kLsqRows - 1; b >= 0; --b) {
    for (int i = min(kk, 32 * b + 32) - 1; i >= 32 * b; --i) {
      double d[kLsqRows];   // the next column, above its diagonal
#pragma unroll
      for (int q = 0; q <= b; ++q) {
        const int r = lane + 32 * q;
        d[q] = r < i - 1 ? H[(size_t)(i - 1) * m1 + r] : 0.0;
      }
      const double yi = __shfl_sync(0xffffffffu, v[b] * inv[b], i & 31);
#pragma unroll
      for (int q = 0; q <= b; ++q) {
        v[q] -= c[q] * yi;   // zero at and below the diagonal
        c[q] = d[q];
      }
      if (lane == (i & 31)) y[i] = yi;
    }
  }
}

// x += Z y (right preconditioning: the update lives in span{Z}), two rows per
// thread, eight columns in flight
template <class T>
__global__ void __launch_bounds__(256) k_xupdate(int n2, double* __restrict__ x, const T* __restrict__ Z, size_t ld,
                                                 const double* __restrict__ y, const Ctl* ctl) {
  pdl_begin();
  using T2 = typename Vec2<T>::type;
  __shared__ double ys[256];
  const int kk = ctl->j;
  for (int l = threadIdx.x; l < kk; l += blockDim.x) ys[l] = y[l];
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n2) return;
  const T2* __restrict__ z = reinterpret_cast<const T2*>(Z) + i;
  const size_t l2 = ld >> 1;
  double2 v = reinterpret_cast<double2*>(x)[i];
  int l = 0;
  for (; l + 7 < kk; l += 8) {
    T2 q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) q[u] = z[(size_t)(l + u) * l2];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v.x += (double)q[u].x * ys[l + u];
      v.y += (double)q[u].y * ys[l + u];
    }
  }
  for (; l < kk; ++l) {
    const T2 q = z[(size_t)l * l2];
    v.x += (double)q.x * ys[l];
    v.y += (double)q.y * ys[l];
  }
  reinterpret_cast<double2*>(x)[i] = v;
}

// nodal velocities on the lattice -> node order, as u^n and as the iterate
__global__ void k_state_in(size_t nlat, const int* __restrict__ l2n, const double* __restrict__ u,
                           double* __restrict__ uold, double* __restrict__ x) {
  pdl_begin();
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= nlat) return;
  const int k = l2n[i];
  if (k < 0) return;   // the walls keep their data
  const double2 v = reinterpret_cast<const double2*>(u)[i];
  reinterpret_cast<double2*>(uold)[k] = v;
  reinterpret_cast<double2*>(x)[k] = v;
}

// node order -> lattice, wall values included
__global__ void k_state_out(size_t nlat, const int* __restrict__ l2n, const double* __restrict__ wall,
                            const double* __restrict__ x, double* __restrict__ u) {
  pdl_begin();
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= nlat) return;
  const int k = l2n[i];
  reinterpret_cast<double2*>(u)[i] = k >= 0 ? reinterpret_cast<const double2*>(x)[k] : reinterpret_cast<const double2*>(wall)[i];
}

// zero mean of the constant pressure coefficients (p in L^2_0)
__global__ void __launch_bounds__(kRedThreads) k_pmean(int nP, double* __restrict__ p, double* __restrict__ part,
                                                       Ctl* ctl) {
  pdl_begin();
  __shared__ double sm[32];
  double acc = 0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nP; c += gridDim.x * blockDim.x) acc += p[3 * (size_t)c];
  acc = block_sum(acc, sm);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
  if (last_block(&ctl->counter[5])) {
    if (threadIdx.x == 0) {
      double s = 0;
      for (int b = 0; b < (int)gridDim.x; ++b) s += part[b];
      ctl->counter[5] = 0;
      ctl->pmean = s / nP;
    }
  }
}

__global__ void k_psub(int nP, double* __restrict__ p, const Ctl* ctl) {
  pdl_begin();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < nP) p[3 * (size_t)c] -= ctl->pmean;
}

// ------------------------------------------------------------------ setup
static void check_params(const fsi_params& p, int n_nodes, int n_tris) {
  if (p.N < 2 || p.N > 4096 || (p.N & 1)) throw std::invalid_argument("N must be even, 2..4096");
  int Nc = p.N;
  while (Nc % 2 == 0 && Nc > 4) Nc /= 2;
  if (Nc > 8) throw std::invalid_argument("N must be c * 2^k with c <= 8");
  if (!(p.dt > 0) || !(p.rho_f > 0) || !(p.nu > 0) || !(p.kappa >= 0)) throw std::invalid_argument("bad material");
  if (p.precond < 0 || p.precond > 3) throw std::invalid_argument("precond");
  if (p.precision != 0 && p.precision != 1) throw std::invalid_argument("precision");
  if (p.solid_elem != 0 && p.solid_elem != 1) throw std::invalid_argument("solid_elem");
  if (n_nodes < (p.solid_elem == 1 ? 4 : 3) || n_tris < 1) throw std::invalid_argument("solid mesh");
  if (p.solid_elem == 1 && (p.coupling != 0 || p.solid_law != 0))
    throw std::invalid_argument("the Q1 solid takes the point rule and the linear law");
  if (p.mg_cluster < -1) throw std::invalid_argument("mg_cluster");
  if (p.mg_fused != 0 && p.mg_fused != -1) throw std::invalid_argument("mg_fused");
  if (p.mg_coarse > 32) throw std::invalid_argument("mg_coarse must be at most 32");
  if (p.mg_coarse_p > 32) throw std::invalid_argument("mg_coarse_p must be at most 32");
  if (p.coupling != 0 && p.coupling != 1) throw std::invalid_argument("coupling");
  if (p.solid_law != 0 && p.solid_law != 1) throw std::invalid_argument("solid_law");
  if (p.autotune != 0 && p.autotune != 1) throw std::invalid_argument("autotune");
  if (p.solid_law == 1 && !(p.gamma > 0 && p.eta > 0)) throw std::invalid_argument("gamma, eta");
  // the Givens kernels hold one Hessenberg column in shared memory (256 doubles)
  if (p.restart > 250) throw std::invalid_argument("restart must be <= 250");
  if (p.stokes_its > 16) throw std::invalid_argument("stokes_its must be <= 16");
}

// Node ids per solid element and rule points per element (P1: the 6-point
// triangle rule; Q1: 3 x 3 Gauss).
static int elem_nodes(const fsi_params& p) { return p.solid_elem == 1 ? 4 : 3; }
static int elem_points(const fsi_params& p) { return p.solid_elem == 1 ? 9 : 6; }

static fsi_params with_defaults(fsi_params p) {
  if (p.restart <= 0) p.restart = 200;
  if (!(p.rtol > 0)) p.rtol = 1e-8;
  if (p.max_it <= 0) p.max_it = 1000;
  if (p.mg_degree <= 0) p.mg_degree = 2;
  // Q1: D^-1 C_s has a wider interval ([1/4, 9/4] on squares against [1/2, 2]
  // for P1), so about 1.6 x the Chebyshev steps for the same reduction
  if (p.cs_degree <= 0) p.cs_degree = (p.precision == 1) ? (p.solid_elem == 1 ? 20 : 12) : (p.solid_elem == 1 ? 26 : 16);
  if (!(p.inner_rtol > 0)) p.inner_rtol = 1e-5;
  if (p.max_refine <= 0) p.max_refine = 30;
  if (p.stokes_its <= 0) p.stokes_its = 1;
  if (!(p.stokes_omega > 0)) p.stokes_omega = 1.0;
  if (!(p.newton_tol > 0)) p.newton_tol = 1e-6;
  if (p.newton_max <= 0) p.newton_max = 20;
  // coarsest grid 16 cells: one dense product (a 15 MB FP32 inverse, held in
  // L2) in place of the 16-cell level's two launches and the 8-cell solve
  if (p.mg_coarse <= 0) p.mg_coarse = 16;
  if (p.mg_coarse_p <= 0) p.mg_coarse_p = p.mg_coarse;
  return p;
}

// The four hierarchies' plans and coarsest solves, before the memory of the levels,
// the operators and the basis is taken: the full inverses that the creation needs go
// back before the rest comes.
static void build_hierarchies(Problem& P) {
  const bool mixed = P.prm.precision == 1;
  // the FP64 levels are matrix-free products launch by launch (the FP32 ones
  // take the fused kernels); mg_fused = -1 keeps the stored matrices
  const bool mfree = P.prm.mg_fused == 0;
  // With the matrix-free levels the automatic choice leaves the cluster out:
  // two fused launches per level measured faster than the cluster launch of
  // the same levels in FP32 (10.8 against 9.7 steps/s on the 128 x 128
  // cavity), and in FP64 the pressure cluster from 32 cells down takes 42 us
  // where its levels launch by launch take 20.
  int cl_max = P.prm.mg_cluster;
  if (cl_max == 0 && mfree) cl_max = 8;
  for (bool pressure : {false, true}) {
    MG<double>& m64 = pressure ? P.p64.mgP : P.p64.mgU;
    MG<float>& m32 = pressure ? P.p32.mgP : P.p32.mgU;
    plan_mg<double>(P.hs, pressure, P.prm.mg_degree, m64, mfree);
    if (mixed) plan_mg<float>(P.hs, pressure, P.prm.mg_degree, m32, false);
    build_coarse(P.ar, P.hs, pressure, m64, mixed ? &m32 : nullptr, cl_max, P.stream);
    if (mixed) select_mf<float>(m32, P.hs, P.prm.mg_fused, P.ar.count_only);
  }
  // mg_fused = -1 also keeps the stored fluid rows of the operator and of the
  // Stokes residual: the assembled form that the matrix-free one is tested against
  if (mfree && P.N >= kMfo64MinNFull) P.p64.mf = make_mfop<double>(P.hs.levels[0]);
  if (mfree && mixed) P.p32.mf = make_mfop<float>(P.hs.levels[0]);
}

template <class T>
static void build_prec(Problem& P, Prec<T>& pr, const FullOp<T>& op) {
  Arena& ar = P.ar;
  alloc_mg<T>(ar, P.hs, pr.mgU, P.prm.autotune == 1, P.stream);
  alloc_mg<T>(ar, P.hs, pr.mgP, P.prm.autotune == 1, P.stream);
  pr.op = op;
  pr.As = upload_sell<T>(ar, to_sell(P.hs.As));
  if (P.prm.solid_law == 1) {
    pr.KT.nrows = P.nS; pr.KT.BR = 2; pr.KT.BC = 2; pr.KT.NV = 4; pr.KT.kron = false;
    pr.KT.soff = op.Ssol.soff; pr.KT.len = op.Ssol.len; pr.KT.col = op.Ssol.col;
    if constexpr (std::is_same<T, double>::value) pr.KT.val = P.kt64;
    else pr.KT.val = P.kt32;
  }
  pr.mpinv = upload_as<T>(ar, P.hs.mp_inv);
  pr.csdinv = upload_as<T>(ar, P.hs.cs_dinv);
  pr.vin = ar.alloc<T>(P.n);
  pr.zw = ar.alloc<T>(P.n);
  const size_t n2 = 2 * (size_t)P.nS;
  pr.sb = ar.alloc<T>(n2); pr.sx = ar.alloc<T>(n2); pr.sx2 = ar.alloc<T>(n2); pr.sd = ar.alloc<T>(n2);
  pr.cs_k = P.prm.cs_degree;
  pr.chs = cheb_coeffs(P.hs.cs_lo, P.hs.cs_hi, pr.cs_k);
  const size_t nf = 2 * (size_t)P.nU + 3 * (size_t)P.nP;
  pr.ru = ar.alloc<T>(2 * (size_t)P.nU);
  pr.t = ar.alloc<T>(nf);
  pr.dz = ar.alloc<T>(nf);
  pr.stokes_its = P.prm.stokes_its;
  pr.stokes_omega = (T)P.prm.stokes_omega;
}

// The operator's structure; the stored fluid rows only where they are read
// (pr.mf: not by the products; -B^T also starts the velocity V-cycle of a finest
// level that is neither fused nor matrix-free).
template <class T>
static FullOp<T> make_op(Problem& P, const Prec<T>& pr, const T* cfv, const T* cftv) {
  Arena& ar = P.ar;
  FullOp<T> op;
  op.nU = P.nU; op.nP = P.nP; op.nS = P.nS;
  op.gU = nblk(P.nU, 32); op.gP = nblk(P.nP, 32); op.gS = nblk(P.nS, 32);
  const MGLevel<T>& L0 = pr.mgU.lv[0];
  if (pr.mf.N == 0) {
    op.Af = upload_sell<T>(ar, to_sell(P.hs.levels[0].A));
    op.Bneg = upload_sell<T>(ar, to_sell(P.hs.Bneg));
  } else {
    ar.spared += (long long)(sell_bytes<T>(P.hs.levels[0].A) + sell_bytes<T>(P.hs.Bneg));
  }
  if (pr.mf.N == 0 || !(L0.mf || L0.mfo.N > 0)) op.Bt = upload_sell<T>(ar, to_sell(P.hs.Bt));
  op.Ssol = upload_sell<T>(ar, to_sell(P.hs.Ssol));
  op.cft_ptr = P.cft_ptr; op.cft_col = P.cft_col; op.cft_val = cftv;
  op.cf_len = P.cf_len; op.cf_col = P.cf_col; op.cf_val = cfv; op.cf_cap = P.cf_cap;
  op.inv_dt = (T)(1.0 / P.prm.dt);
  if (P.prm.solid_law == 1) {
    if constexpr (std::is_same<T, double>::value) op.kt = P.kt64;
    else op.kt = P.kt32;
  }
  return op;
}

static KrylovArgs krylov_args(Problem& P, cudaGraphConditionalHandle h) {
  KrylovArgs k{};
  k.n = (int)P.n;
  k.chunk = red_chunk(P.n);
  k.ld = P.n;
  k.V = P.V;
  k.w = P.w;
  k.part = P.part;
  k.h1 = P.y + (P.m + 2);       // scratch after y (m+2 entries each)
  k.h2 = P.y + 2 * (P.m + 2);
  k.H = P.H; k.cs = P.cs; k.sn = P.sn; k.g = P.g;
  k.ctl = P.ctl;
  k.cond = h;
  return k;
}

// S4 by the exact rule: the pairs of small triangles (when there is room for them),
// then the C_f rows.
static void exact_rule_launch(Problem& P, cudaStream_t s) {
  if (P.pairs)
    launch(k_exact_pairs, nblk((size_t)kExactCells * P.nTri, 128), 128, 0, s, P.nTri, P.N, P.tris, P.Xold, P.area, P.pairs);
  launch(k_cf_rows_exact, nblk(P.nS, kCfWarps), 32 * kCfWarps, 0, s, P.nS, P.N, P.ntp, P.nt, P.tris, P.Xold, P.area,
         P.l2n, P.wall, P.cf_cap, P.cf_len, P.cf_col, P.cf_val, P.cf_val32, P.cflift, &P.ctl->aflags, P.pairs, P.nTri);
}

// S2 + S4 by the point rule: locate the rule points, then the C_f rows.
static void point_rule_launch(Problem& P, cudaStream_t s) {
  if (elem_nodes(P.prm) == 4) {
    launch(k_locate<4>, nblk(P.nPts, 256), 256, 0, s, P.nPts, P.N, P.tris, P.Xold, P.cell, P.xi, P.eta,
           &P.ctl->aflags);
    launch(k_cf_rows<4>, nblk(P.nS, kCfWarps), 32 * kCfWarps, 0, s, P.nS, P.N, P.ntp, P.nt, P.area, P.cell, P.xi,
           P.eta, P.l2n, P.wall, P.cf_cap, P.cf_len, P.cf_col, P.cf_val, P.cf_val32, P.cflift, &P.ctl->aflags);
  } else {
    launch(k_locate<3>, nblk(P.nPts, 256), 256, 0, s, P.nPts, P.N, P.tris, P.Xold, P.cell, P.xi, P.eta,
           &P.ctl->aflags);
    launch(k_cf_rows<3>, nblk(P.nS, kCfWarps), 32 * kCfWarps, 0, s, P.nS, P.N, P.ntp, P.nt, P.area, P.cell, P.xi,
           P.eta, P.l2n, P.wall, P.cf_cap, P.cf_len, P.cf_col, P.cf_val, P.cf_val32, P.cflift, &P.ctl->aflags);
  }
}

static void assemble_launch(Problem& P, cudaStream_t s) {
  CK(cudaMemsetAsync(&P.ctl->aflags, 0, sizeof(int), s));
  if (P.prm.coupling == 1) {  // the paper's exact rule: mesh intersection
    exact_rule_launch(P, s);
  } else {                    // located points of the point rule
    point_rule_launch(P, s);
  }
  CK(cudaMemsetAsync(P.cft_cnt, 0, sizeof(int) * P.nU, s));
  const size_t nslot = (size_t)P.nS * P.cf_cap;
  launch(k_cft_count, nblk(nslot, 256), 256, 0, s, P.nS, P.cf_cap, P.cf_len, P.cf_col, P.cft_cnt);
  const int nb = (int)nblk(P.nU, kScanBlock);
  launch(k_scan_partial, nb, kScanBlock, 0, s, P.nU, P.cft_cnt, P.scan_bsum);
  launch(k_scan_top, 1, kScanBlock, 0, s, nb, P.scan_bsum);
  launch(k_scan_final, nb, kScanBlock, 0, s, P.nU, P.cft_cnt, P.scan_bsum, P.cft_ptr, P.cft_cur);
  launch(k_cft_scatter, nblk(nslot, 256), 256, 0, s, P.nS, P.cf_cap, P.cf_len, P.cf_col, P.cf_val, P.cft_cur,
                                                 P.cft_col, P.cft_val);
  launch(k_cft_sort, nblk(P.nU, 128), 128, 0, s, P.nU, P.cft_ptr, P.cft_col, P.cft_val, P.cft_val32);
  // S1: g1 = (rho/dt) M u^n - K_ID u_D ;  g2 = -(1/dt) C_s X^n - C_D u_D
  sell_launch(P.M64, MODE_AXPBY, axpby<double>(P.uold, P.b, P.lift_u, P.prm.rho_f / P.prm.dt, 1.0), s);
  sell_launch(P.Cs64, MODE_AXPBY, axpby<double>(P.Xold, P.b + P.offL, P.cflift, -1.0 / P.prm.dt, -1.0), s);
}

// Gram-Schmidt of w against V[0..j], the Givens step and the next basis vector
template <int CH, class T>
static void orthogonalise_launch(Problem& P, Prec<T>& pr, const KrylovArgs& k, cudaStream_t s) {
  launch(k_gs1<CH>, P.red_blocks, kRedThreads, 0, s, k);
  launch(k_gs2<CH>, P.red_blocks, kRedThreads, 0, s, k);
  launch(k_gs3<CH>, P.red_blocks, kRedThreads, 0, s, k);
  launch(k_basis<T>, nblk(P.n / 2, 256), 256, 0, s, (int)(P.n / 2), P.V, P.n, P.w, pr.vin, P.ctl);
}

template <class T>
static cudaLaunchConfig_t gs_cluster_config(cudaLaunchAttribute* at, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kGsCluster);
  cfg.blockDim = dim3(kRedThreads);
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kGsCluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// Whether the problem's orthogonalisation runs as one cluster: its rows fit, and
// the device schedules a cluster of this (non-portable) size.  A row pair more per
// worker makes each basis vector dearer (0.77, 1.22, 1.68 and 2.13 us a vector at
// one to four pairs, 0.7 to 0.85 as separate launches), so the line lies where the
// cycles of a precision still gain, in us an iteration with j vectors, cluster
// against launches:
//   FP64, cycles as long as the solve, one pair (n <= 4096): n = 3366 86 / 98 at
//     j = 10, 96 / 99 at 24, 162 / 167 at 112, 248 / 259 at 220; but n = 5110
//     104 / 110 at 10, 138 / 136 at 40, 230 / 206 at 112, 360 / 287 at 220;
//   mixed, cycles of some 10 vectors (inner_rtol), two pairs (n <= 8192): n = 7014
//     54.4 / 56.4 at 10, 70.7 / 68.9 at 24; but n = 16054 75 / 68 at 10, 143 / 88 at
//     40, and FP64 n = 9726 103 / 104 at 10, 156 / 133 at 40.
template <class T>
static bool gs_cluster_fits(size_t n) {
  if (n > (size_t)kGsCluster * kGsClusterRows / (sizeof(T) == 8 ? 2 : 1)) return false;
  if (cudaFuncSetAttribute(k_gs_cluster<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg = gs_cluster_config<T>(at, nullptr);
  int num = 0;
  if (cudaOccupancyMaxActiveClusters(&num, k_gs_cluster<T>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return num > 0;
}

template <class T>
static void gs_cluster_launch(Problem& P, Prec<T>& pr, const KrylovArgs& k, cudaStream_t s) {
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = gs_cluster_config<T>(at, s);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_gs_cluster<T>, k, P.V, pr.vin);
  if (e != cudaSuccess) throw CudaError(e, "cudaLaunchKernelEx (cluster orthogonalisation)");
}

// One Arnoldi iteration; pr.vin holds v_j on entry (k_basis of the previous
// iteration or of the cycle's start wrote it).
template <class T>
static void iteration_launch(Problem& P, Prec<T>& pr, const KrylovArgs& k, cudaStream_t s) {
  precond_launch(P, pr, s);
  full_launch<T, double>(pr, pr.zw, P.w, nullptr, 1.0, 0.0, (T*)P.Z, P.n, P.ctl, s);
  if (P.gs_cluster) gs_cluster_launch<T>(P, pr, k, s);
  else if (k.chunk == kChunkSmall) orthogonalise_launch<kChunkSmall>(P, pr, k, s);
  else orthogonalise_launch<kChunkLarge>(P, pr, k, s);
}

template <class T>
static void cycle_start_launch(Problem& P, Prec<T>& pr, const KrylovArgs& k, cudaStream_t s) {
  full_launch<double, double>(P.p64, P.x, P.w, P.b, -1.0, 1.0, nullptr, 0, nullptr, s);
  launch(k_cycle_start, P.red_blocks, kRedThreads, 0, s, k);
  launch(k_basis<T>, nblk(P.n / 2, 256), 256, 0, s, (int)(P.n / 2), P.V, P.n, P.w, pr.vin, P.ctl);
}

template <class T>
static void cycle_end_launch(Problem& P, cudaStream_t s) {
  launch(k_lsq, 1, 32, 0, s, P.H, P.g, P.y, P.ctl);
  launch(k_xupdate<T>, nblk(P.n / 2, 256), 256, 0, s, (int)(P.n / 2), P.x, (const T*)P.Z, P.n, P.y, P.ctl);
}

static int count_kernel_nodes(cudaGraph_t g) {
  size_t n = 0;
  CK(cudaGraphGetNodes(g, nullptr, &n));
  std::vector<cudaGraphNode_t> nodes(n);
  CK(cudaGraphGetNodes(g, nodes.data(), &n));
  int k = 0;
  for (auto nd : nodes) {
    cudaGraphNodeType t;
    CK(cudaGraphNodeGetType(nd, &t));
    if (t == cudaGraphNodeTypeKernel) ++k;
  }
  return k;
}

// The whole solve as one graph: an outer WHILE node over restart/refinement
// cycles whose body computes the true FP64 residual (k_cycle_start sets both
// conditions), runs the Arnoldi loop as an inner WHILE node (k_gs2/k_gs3 set
// its condition) and updates x.  No host round trip inside a solve.
template <class T>
static void build_cycle_graph(Problem& P, Prec<T>& pr) {
  cudaGraph_t g = nullptr;
  CK(cudaGraphCreate(&g, 0));
  cudaGraphConditionalHandle h_out;
  CK(cudaGraphConditionalHandleCreate(&h_out, g, 1, cudaGraphCondAssignDefault));
  cudaGraphNodeParams op = {};
  op.type = cudaGraphNodeTypeConditional;
  op.conditional.handle = h_out;
  op.conditional.type = cudaGraphCondTypeWhile;
  op.conditional.size = 1;
  cudaGraphNode_t onode;
  CK(cudaGraphAddNode(&onode, g, nullptr, nullptr, 0, &op));
  cudaGraph_t obody = op.conditional.phGraph_out[0];
  cudaStream_t s = P.s2;
  CK(cudaStreamBeginCaptureToGraph(s, obody, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
  cudaGraphConditionalHandle h_in;
  CK(cudaGraphConditionalHandleCreate(&h_in, obody, 0, 0));
  KrylovArgs k = krylov_args(P, h_in);
  k.cond_outer = h_out;
  cycle_start_launch(P, pr, k, s);
  cudaStreamCaptureStatus st;
  cudaGraph_t cg = nullptr;
  const cudaGraphNode_t* deps = nullptr;
  size_t ndeps = 0;
  CK(cudaStreamGetCaptureInfo(s, &st, nullptr, &cg, &deps, nullptr, &ndeps));
  cudaGraphNodeParams ip = {};
  ip.type = cudaGraphNodeTypeConditional;
  ip.conditional.handle = h_in;
  ip.conditional.type = cudaGraphCondTypeWhile;
  ip.conditional.size = 1;
  cudaGraphNode_t inode;
  CK(cudaGraphAddNode(&inode, cg, deps, nullptr, ndeps, &ip));
  CK(cudaStreamUpdateCaptureDependencies(s, &inode, nullptr, 1, cudaStreamSetCaptureDependencies));
  cudaGraph_t ibody = ip.conditional.phGraph_out[0];
  CK(cudaStreamBeginCaptureToGraph(P.s5, ibody, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
  KrylovArgs ki = k;
  ki.cond_outer = 0;
  iteration_launch(P, pr, ki, P.s5);
  CK(cudaStreamEndCapture(P.s5, &ibody));
  P.kn_body = count_kernel_nodes(ibody);
  cycle_end_launch<T>(P, s);
  CK(cudaStreamEndCapture(s, &obody));
  P.kn_cycle = count_kernel_nodes(obody);
  P.gr_cycle = g;
  CK(cudaGraphInstantiate(&P.g_cycle, P.gr_cycle, 0));
}

template <class T>
static void build_host_loop_graphs(Problem& P, Prec<T>& pr) {
  cudaStream_t s = P.stream;
  KrylovArgs k = krylov_args(P, 0);
  CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  cycle_start_launch(P, pr, k, s);
  CK(cudaStreamEndCapture(s, &P.gr_cstart));
  CK(cudaGraphInstantiate(&P.g_cstart, P.gr_cstart, 0));
  CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  iteration_launch(P, pr, k, s);
  CK(cudaStreamEndCapture(s, &P.gr_body));
  CK(cudaGraphInstantiate(&P.g_body, P.gr_body, 0));
  CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  cycle_end_launch<T>(P, s);
  CK(cudaStreamEndCapture(s, &P.gr_cend));
  CK(cudaGraphInstantiate(&P.g_cend, P.gr_cend, 0));
  P.kn_body = count_kernel_nodes(P.gr_body);
}

static void build_graphs(Problem& P) {
  cudaStream_t s = P.stream;
  // assemble
  CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  assemble_launch(P, s);
  CK(cudaStreamEndCapture(s, &P.gr_assemble));
  CK(cudaGraphInstantiate(&P.g_assemble, P.gr_assemble, 0));
  // begin: ||b|| and counters
  CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  {
    KrylovArgs k = krylov_args(P, 0);
    const double inner = (P.prm.precision == 1) ? P.prm.inner_rtol : 0.0;
    const int max_cycles = (P.prm.precision == 1) ? P.prm.max_refine + 1 : (1 << 30);
    launch(k_solve_begin, P.red_blocks, kRedThreads, 0, s, k, P.b, P.prm.rtol, inner, P.prm.max_it, P.m, max_cycles);
  }
  CK(cudaStreamEndCapture(s, &P.gr_begin));
  CK(cudaGraphInstantiate(&P.g_begin, P.gr_begin, 0));
  P.gs_cluster = P.prm.precision == 1 ? gs_cluster_fits<float>(P.n) : gs_cluster_fits<double>(P.n);
  // cycle
  const char* hl = getenv("FSI_HOST_LOOP");
  P.host_loop = hl && hl[0] == '1';
  if (P.host_loop) {
    if (P.prm.precision == 1) build_host_loop_graphs<float>(P, P.p32);
    else build_host_loop_graphs<double>(P, P.p64);
  } else {
    if (P.prm.precision == 1) build_cycle_graph<float>(P, P.p32);
    else build_cycle_graph<double>(P, P.p64);
  }
  // finish: zero-mean pressure
  CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  launch(k_pmean, std::min(64, (int)nblk(P.nP, kRedThreads)), kRedThreads, 0, s, P.nP, P.x + P.offP, P.part, P.ctl);
  launch(k_psub, nblk(P.nP, 256), 256, 0, s, P.nP, P.x + P.offP, P.ctl);
  CK(cudaStreamEndCapture(s, &P.gr_finish));
  CK(cudaGraphInstantiate(&P.g_finish, P.gr_finish, 0));
  P.kn_assemble = count_kernel_nodes(P.gr_assemble);
  P.kn_begin = count_kernel_nodes(P.gr_begin);
  if (P.host_loop) P.kn_cycle = count_kernel_nodes(P.gr_cstart) + count_kernel_nodes(P.gr_cend);
  P.kn_finish = count_kernel_nodes(P.gr_finish);
}

static void allocate_problem(Problem& P, const double* ref_xy, const int* tris_h) {
  Arena& ar = P.ar;
  const HostSetup& hs = P.hs;
  const int npe = elem_nodes(P.prm);
  P.tris = ar.upload(std::vector<int>(tris_h, tris_h + npe * (size_t)P.nTri));
  P.area = ar.upload(npe == 4 ? hs.pt_w : hs.tri_area);
  P.ntp = ar.upload(hs.node_tri_ptr);
  P.nt = ar.upload(hs.node_tri);
  P.l2n = ar.upload(hs.lattice_to_node);
  P.wall = ar.upload(hs.wall_u);
  P.cell = ar.alloc<int>(P.nPts);
  P.xi = ar.alloc<double>(P.nPts);
  P.eta = ar.alloc<double>(P.nPts);
  // capacity of a coupling row: the fluid lattice nodes of the cells that the
  // triangles around one solid node overlap in the reference configuration
  // (at least 64, at most the assembly window); a row that outgrows it later
  // raises FSI_ERR_CAPACITY
  {
    int need = 64;
    for (int l = 0; l < P.nS; ++l) {
      double lo[2] = {1e300, 1e300}, hi[2] = {-1e300, -1e300};
      for (int k = hs.node_tri_ptr[l]; k < hs.node_tri_ptr[l + 1]; ++k) {
        const int t = hs.node_tri[k] / npe;
        for (int v = 0; v < npe; ++v)
          for (int c = 0; c < 2; ++c) {
            const double x = ref_xy[2 * (size_t)tris_h[npe * (size_t)t + v] + c];
            lo[c] = std::min(lo[c], x);
            hi[c] = std::max(hi[c], x);
          }
      }
      if (hi[0] < lo[0]) continue;
      const int cw = (int)std::floor(hi[0] * P.N) - (int)std::floor(lo[0] * P.N) + 1;
      const int ch = (int)std::floor(hi[1] * P.N) - (int)std::floor(lo[1] * P.N) + 1;
      need = std::max(need, (2 * cw + 1) * (2 * ch + 1));
    }
    P.cf_cap = std::min(need, kCfWindow);
  }
  if (P.prm.solid_law == 1) {
    std::vector<double> tg(6 * (size_t)P.nTri);
    for (int t = 0; t < P.nTri; ++t) {
      const double* p0 = ref_xy + 2 * (size_t)tris_h[3 * t];
      const double* p1 = ref_xy + 2 * (size_t)tris_h[3 * t + 1];
      const double* p2 = ref_xy + 2 * (size_t)tris_h[3 * t + 2];
      const double d1x = p1[0] - p0[0], d1y = p1[1] - p0[1], d2x = p2[0] - p0[0], d2y = p2[1] - p0[1];
      const double det = d1x * d2y - d1y * d2x;
      const double g1x = d2y / det, g1y = -d2x / det, g2x = -d1y / det, g2y = d1x / det;
      const double v[6] = {-(g1x + g2x), -(g1y + g2y), g1x, g1y, g2x, g2y};
      for (int q = 0; q < 6; ++q) tg[6 * (size_t)t + q] = v[q];
    }
    P.tgrad = ar.upload(tg);
    const SellHost ss = to_sell(hs.Ssol);
    const size_t nslot = (size_t)ss.soff[ss.nslices];
    P.kt64 = ar.alloc<double>(4 * nslot);
    P.kt32 = ar.alloc<float>(4 * nslot);
  }
  const size_t cfslots = (size_t)nblk(P.nS, 32) * 32 * P.cf_cap;
  P.cf_len = ar.alloc<int>(P.nS);
  P.cf_col = ar.alloc<int>(cfslots);
  P.cf_val = ar.alloc<double>(cfslots);
  P.cf_val32 = ar.alloc<float>(cfslots);
  P.cflift = ar.alloc<double>(2 * (size_t)P.nS);
  const size_t tcap = (size_t)P.nS * P.cf_cap;
  P.cft_ptr = ar.alloc<int>(P.nU + 1);
  P.cft_col = ar.alloc<int>(tcap);
  P.cft_val = ar.alloc<double>(tcap);
  P.cft_val32 = ar.alloc<float>(tcap);
  P.cft_cnt = ar.alloc<int>(P.nU);
  P.cft_cur = ar.alloc<int>(P.nU);
  P.scan_bsum = ar.alloc<int>(nblk(P.nU, kScanBlock) + 1);
  P.x = ar.alloc<double>(P.n);
  P.b = ar.alloc<double>(P.n);
  P.w = ar.alloc<double>(P.n);
  P.uold = ar.alloc<double>(2 * (size_t)P.nU);
  P.Xold = ar.alloc<double>(2 * (size_t)P.nS);
  P.lift_u = ar.upload(hs.lift_u);
  P.M64 = upload_sell<double>(ar, to_sell(hs.M));
  P.Cs64 = upload_sell<double>(ar, to_sell(hs.Cs));
  build_hierarchies(P);
  const int m = P.m;
  P.V = ar.alloc<double>((size_t)(m + 1) * P.n);
  if (P.prm.precision == 1) P.Z = ar.alloc<float>((size_t)m * P.n);
  else P.Z = ar.alloc<double>((size_t)m * P.n);
  P.H = ar.alloc<double>((size_t)(m + 1) * m);
  P.cs = ar.alloc<double>(m + 1);
  P.sn = ar.alloc<double>(m + 1);
  P.g = ar.alloc<double>(m + 2);
  P.y = ar.alloc<double>(3 * (size_t)(m + 2));
  P.red_blocks = red_grid(P.n);
  P.part = ar.alloc<double>((size_t)std::max(P.red_blocks, 64) * (m + 2));
  P.ctl = ar.alloc<Ctl>(1);
  P.op64 = make_op<double>(P, P.p64, P.cf_val, P.cft_val);
  build_prec<double>(P, P.p64, P.op64);
  if (P.prm.precision == 1) {
    P.op32 = make_op<float>(P, P.p32, P.cf_val32, P.cft_val32);
    build_prec<float>(P, P.p32, P.op32);
  }
  // FP32 first: a mixed problem's solves take it
  if (P.prm.precision == 1) setup_mass_solves<float>(P, P.p32, ref_xy);
  setup_mass_solves<double>(P, P.p64, ref_xy);
  // The pairs of the exact rule live in the Krylov basis, idle while C_f is
  // assembled; where it is too short (few vectors, a body much finer than the grid)
  // they take memory spared elsewhere, or each row forms its own.
  if (P.prm.coupling == 1) {
    const size_t np = 27 * (size_t)kExactCells * P.nTri;
    if ((size_t)(P.m + 1) * P.n >= np) {
      P.pairs = P.V;
    } else if ((long long)Arena::size<double>(np) <= ar.spared) {
      ar.spared -= Arena::size<double>(np);
      P.pairs = ar.alloc<double>(np);
    }
  }
}


// ----------------------------------------------------------- timing hook
template <class T>
static double fullop_bytes(Problem& P, bool mf, double cfnnz, size_t xbytes, size_t ybytes) {
  const HostSetup& hs = P.hs;
  double b = sell_bytes<T>(hs.Ssol);   // matrix-free fluid rows read no stored blocks
  if (!mf) b += sell_bytes<T>(hs.levels[0].A) + sell_bytes<T>(hs.Bt) + sell_bytes<T>(hs.Bneg);
  b += 2.0 * cfnnz * (sizeof(T) + sizeof(int)) + (P.nU + 1) * 4.0 + P.nS * 4.0;
  b += (double)P.n * (xbytes + ybytes);
  return b;
}

__global__ void k_flush(size_t n, uint4* __restrict__ buf, unsigned v) {
  pdl_begin();
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    buf[i] = make_uint4(v, v, v, v);
}

}  // namespace fsi

// ================================================================== C ABI
using namespace fsi;

struct fsi_problem {
  Problem P;
};

static int map_exception() {
  try {
    throw;
  } catch (const std::bad_alloc&) {
    return FSI_ERR_OOM;
  } catch (const std::invalid_argument&) {
    return FSI_ERR_INVALID;
  } catch (const CudaError& e) {
    if (e.code == cudaErrorMemoryAllocation) return FSI_ERR_OOM;
    return FSI_ERR_CUDA;
  } catch (...) {
    return FSI_ERR_CUDA;
  }
}

// State in and out.  The caller's nodal arrays cross in one copy each, to and
// from a scratch area on the device (the Krylov basis, idle between solves: it
// holds at least two vectors of n, more than the lattice's 2 (2N+1)^2 for every
// N >= 2), and two kernels permute between lattice and node order there.  On the
// host the same took an index loop over the nodes, a second upload and, on the
// way out, a zeroed copy of the whole vector.
static void upload_state(Problem& P, const double* u, const double* X) {
  const size_t nlat = (size_t)(2 * P.N + 1) * (2 * P.N + 1);
  if (u) {
    CK(cudaMemcpyAsync(P.V, u, 2 * nlat * 8, cudaMemcpyHostToDevice, P.stream));
    launch(k_state_in, nblk(nlat, 256), 256, 0, P.stream, nlat, P.l2n, (const double*)P.V, P.uold, P.x);
  }
  if (X) {
    CK(cudaMemcpyAsync(P.Xold, X, 2 * (size_t)P.nS * 8, cudaMemcpyHostToDevice, P.stream));
    CK(cudaMemcpyAsync(P.x + P.offX, P.Xold, 2 * (size_t)P.nS * 8, cudaMemcpyDeviceToDevice, P.stream));
  }
  if (u || X) CK(cudaStreamSynchronize(P.stream));
}

// by_counts: the mesh stands for every mesh of its counts
static size_t footprint_impl(const fsi_params& prm0, int n_nodes, int n_tris, const double* ref_xy,
                             const int* tris, bool by_counts) {
  fsi_params prm = with_defaults(prm0);
  check_params(prm, n_nodes, n_tris);
  Problem P;
  P.prm = prm;
  P.ar.count_only = true;
  P.by_counts = by_counts;
  P.N = prm.N;
  VNum vn(prm.N);
  P.nU = vn.n; P.nP = prm.N * prm.N; P.nS = n_nodes; P.nTri = n_tris; P.nPts = elem_points(prm) * n_tris;
  P.offP = 2 * (size_t)P.nU; P.offX = P.offP + 3 * (size_t)P.nP; P.offL = P.offX + 2 * (size_t)P.nS;
  P.n = P.offL + 2 * (size_t)P.nS;
  P.m = prm.restart;
  SetupParams sp{prm.N, prm.rho_f, prm.nu, prm.kappa, prm.dt, prm.lid_u};
  sp.npe = elem_nodes(prm);
  sp.coarse_max = prm.mg_coarse;
  sp.coarse_max_p = prm.mg_coarse_p;
  build_setup(sp, n_nodes, n_tris, ref_xy, tris, P.hs);
  allocate_problem(P, ref_xy, tris);
  return P.ar.peak;
}

extern "C" {

size_t fsi_footprint_bytes(const fsi_params* params, int n_solid_nodes, int n_tris) {
  if (!params || n_solid_nodes < 3 || n_tris < 1) return 0;
  try {
    // a synthetic solid with the same counts: matrix sizes depend on counts only
    // up to the solid adjacency, which is bounded by a small ring patch
    std::vector<double> xy(2 * (size_t)n_solid_nodes);
    std::vector<int> tr(3 * (size_t)n_tris);
    for (int i = 0; i < n_solid_nodes; ++i) { xy[2 * i] = 0.5 + 1e-3 * (i % 7); xy[2 * i + 1] = 0.5 + 1e-3 * (i / 7 % 7); }
    for (int t = 0; t < n_tris; ++t) { tr[3 * t] = 0; tr[3 * t + 1] = 1 + t % (n_solid_nodes - 2); tr[3 * t + 2] = 2 + t % (n_solid_nodes - 2); }
    // solid matrices only need a valid orientation; use a fan of unit triangles
    for (int i = 0; i < n_solid_nodes; ++i) {
      const double a = 6.283185307179586 * i / n_solid_nodes;
      xy[2 * i] = 0.5 + 0.1 * std::cos(a);
      xy[2 * i + 1] = 0.5 + 0.1 * std::sin(a);
    }
    xy[0] = 0.5; xy[1] = 0.5;
    if (params->solid_elem == 1) {
      if (n_solid_nodes < 4) return 0;  // a quadrilateral needs 4 nodes
      tr.assign(4 * (size_t)n_tris, 0);
      if (n_solid_nodes < 8) {
        // a ladder of m quadrilaterals-wide strip: nodes j (bottom) and m + j (top)
        const int m = n_solid_nodes / 2;
        for (int j = 0; j < m; ++j) {
          xy[2 * j] = xy[2 * (m + j)] = 0.3 + 0.4 * j / (m - 1);
          xy[2 * j + 1] = 0.45;
          xy[2 * (m + j) + 1] = 0.55;
        }
        for (int t = 0; t < n_tris; ++t) {
          const int j = t % (m - 1);
          tr[4 * t] = j; tr[4 * t + 1] = j + 1; tr[4 * t + 2] = m + j + 1; tr[4 * t + 3] = m + j;
        }
        return footprint_impl(*params, n_solid_nodes, n_tris, xy.data(), tr.data(), true);
      }
      // quadrilaterals (centre, three consecutive ring nodes): convex and
      // counter-clockwise while three ring steps span less than half a turn
      for (int t = 0; t < n_tris; ++t) {
        const int a = 1 + t % (n_solid_nodes - 1);
        const int b = 1 + (a % (n_solid_nodes - 1));
        const int c = 1 + (b % (n_solid_nodes - 1));
        tr[4 * t] = 0; tr[4 * t + 1] = a; tr[4 * t + 2] = b; tr[4 * t + 3] = c;
      }
      return footprint_impl(*params, n_solid_nodes, n_tris, xy.data(), tr.data(), true);
    }
    if (n_solid_nodes < 5) {
      // too few ring nodes for a fan (its closing triangle would span half a
      // turn): one triangle, or a strip of two-triangle cells (nodes j bottom,
      // m + j top), counter-clockwise
      const int m = n_solid_nodes / 2;
      if (n_solid_nodes == 3) {
        const double p3[6] = {0.45, 0.45, 0.55, 0.45, 0.5, 0.55};
        for (int i = 0; i < 6; ++i) xy[i] = p3[i];
      } else {
        for (int j = 0; j < m; ++j) {
          xy[2 * j] = xy[2 * (m + j)] = 0.3 + 0.4 * j / (m - 1);
          xy[2 * j + 1] = 0.45;
          xy[2 * (m + j) + 1] = 0.55;
        }
      }
      for (int t = 0; t < n_tris; ++t) {
        if (n_solid_nodes == 3) { tr[3 * t] = 0; tr[3 * t + 1] = 1; tr[3 * t + 2] = 2; continue; }
        const int c = t % (2 * (m - 1)), j = c / 2;
        if (c % 2 == 0) { tr[3 * t] = j; tr[3 * t + 1] = j + 1; tr[3 * t + 2] = m + j + 1; }
        else { tr[3 * t] = j; tr[3 * t + 1] = m + j + 1; tr[3 * t + 2] = m + j; }
      }
      return footprint_impl(*params, n_solid_nodes, n_tris, xy.data(), tr.data(), true);
    }
    for (int t = 0; t < n_tris; ++t) {
      const int a = 1 + t % (n_solid_nodes - 1);
      const int b = 1 + (a % (n_solid_nodes - 1));
      tr[3 * t] = 0; tr[3 * t + 1] = a; tr[3 * t + 2] = b;
    }
    return footprint_impl(*params, n_solid_nodes, n_tris, xy.data(), tr.data(), true);
  } catch (...) {
    return 0;
  }
}

int fsi_create_problem_budget(const fsi_params* params, const fsi_solid_mesh* mesh, const double* u0,
                              const double* X0, void* cuda_stream, size_t budget_bytes, fsi_problem** out) {
  if (!params || !mesh || !out || !mesh->ref_xy || !mesh->tris) return FSI_ERR_INVALID;
  *out = nullptr;
  fsi_problem* h = nullptr;
  try {
    fsi_params prm = with_defaults(*params);
    check_params(prm, mesh->n_nodes, mesh->n_tris);
    for (size_t i = 0; i < (size_t)elem_nodes(prm) * mesh->n_tris; ++i)
      if (mesh->tris[i] < 0 || mesh->tris[i] >= mesh->n_nodes) return FSI_ERR_INVALID;
    if (budget_bytes > 0) {
      const size_t need = footprint_impl(prm, mesh->n_nodes, mesh->n_tris, mesh->ref_xy, mesh->tris, false);
      if (need > budget_bytes) return FSI_ERR_BUDGET;
    }
    h = new fsi_problem();
    Problem& P = h->P;
    P.prm = prm;
    CK(cudaGetDevice(&P.device));
    if (cuda_stream) {
      P.stream = (cudaStream_t)cuda_stream;
    } else {
      CK(cudaStreamCreateWithFlags(&P.stream, cudaStreamNonBlocking));
      P.own_stream = true;
    }
    CK(cudaStreamCreateWithFlags(&P.s2, cudaStreamNonBlocking));
    CK(cudaStreamCreateWithFlags(&P.s3, cudaStreamNonBlocking));
    CK(cudaStreamCreateWithFlags(&P.s4, cudaStreamNonBlocking));
    CK(cudaStreamCreateWithFlags(&P.s5, cudaStreamNonBlocking));
    CK(cudaEventCreateWithFlags(&P.ev_join2, cudaEventDisableTiming));
    CK(cudaEventCreateWithFlags(&P.ev_fork2, cudaEventDisableTiming));
    CK(cudaEventCreateWithFlags(&P.ev_fork, cudaEventDisableTiming));
    CK(cudaEventCreateWithFlags(&P.ev_join, cudaEventDisableTiming));
    P.N = prm.N;
    VNum vn(prm.N);
    P.nU = vn.n; P.nP = prm.N * prm.N; P.nS = mesh->n_nodes; P.nTri = mesh->n_tris; P.nPts = elem_points(prm) * mesh->n_tris;
    P.offP = 2 * (size_t)P.nU; P.offX = P.offP + 3 * (size_t)P.nP; P.offL = P.offX + 2 * (size_t)P.nS;
    P.n = P.offL + 2 * (size_t)P.nS;
    P.m = prm.restart;
    SetupParams sp{prm.N, prm.rho_f, prm.nu, prm.kappa, prm.dt, prm.lid_u};
    sp.npe = elem_nodes(prm);
    sp.coarse_max = prm.mg_coarse;
  sp.coarse_max_p = prm.mg_coarse_p;
    build_setup(sp, P.nS, P.nTri, mesh->ref_xy, mesh->tris, P.hs);
    {
      double lam[6][3], w[6];
      triangle_rule(lam, w);
      CK(cudaMemcpyToSymbol(c_rule_lam, lam, sizeof(lam)));
      CK(cudaMemcpyToSymbol(c_rule_w, w, sizeof(w)));
      // Radon's 7-point rule (exact to degree 5) from its closed form: the
      // centroid, weight 9/40; orbits (a, a, 1-2a), a = (6 -/+ sqrt 15)/21,
      // weights (155 -/+ sqrt 15)/1200
      double rl[7][3], rw[7];
      const double r15 = std::sqrt(15.0);
      rl[0][0] = rl[0][1] = rl[0][2] = 1.0 / 3.0;
      rw[0] = 9.0 / 40.0;
      const double oa[2] = {(6.0 - r15) / 21.0, (6.0 + r15) / 21.0};
      const double ow[2] = {(155.0 - r15) / 1200.0, (155.0 + r15) / 1200.0};
      for (int o = 0; o < 2; ++o)
        for (int k = 0; k < 3; ++k) {
          for (int c = 0; c < 3; ++c) rl[1 + 3 * o + k][c] = (c == k) ? 1.0 - 2.0 * oa[o] : oa[o];
          rw[1 + 3 * o + k] = ow[o];
        }
      CK(cudaMemcpyToSymbol(c_radon_lam, rl, sizeof(rl)));
      CK(cudaMemcpyToSymbol(c_radon_w, rw, sizeof(rw)));
      // Q1: (s, t, s t) of the 3 x 3 Gauss points and the shape functions there
      double qs[9], qt[9], qst[9], qw[9], qp[9][3], qc[9][4];
      quad_rule(qs, qt, qst, qw);
      for (int q = 0; q < 9; ++q) {
        qp[q][0] = qs[q]; qp[q][1] = qt[q]; qp[q][2] = qst[q];
        q1_shape(qs[q], qt[q], qc[q]);
      }
      CK(cudaMemcpyToSymbol(c_q1_pt, qp, sizeof(qp)));
      CK(cudaMemcpyToSymbol(c_q1_chi, qc, sizeof(qc)));
    }
    allocate_problem(P, mesh->ref_xy, mesh->tris);
    CK(cudaMemset(P.ctl, 0, sizeof(Ctl)));
    CK(cudaMemset(P.cf_len, 0, sizeof(int) * P.nS));
    CK(cudaMemset(P.cft_ptr, 0, sizeof(int) * (P.nU + 1)));
    CK(cudaMemset(P.cflift, 0, sizeof(double) * 2 * P.nS));
    CK(cudaMemset(P.x, 0, P.n * 8));
    CK(cudaMemset(P.b, 0, P.n * 8));
    CK(cudaMemcpy(P.b + P.offP, P.hs.lift_p.data(), P.hs.lift_p.size() * 8, cudaMemcpyHostToDevice));
    CK(cudaMallocHost((void**)&P.ctl_host, sizeof(Ctl)));
    std::vector<double> u(2 * (size_t)(2 * P.N + 1) * (2 * P.N + 1));
    if (u0) std::copy(u0, u0 + u.size(), u.begin());
    upload_state(P, u.data(), X0 ? X0 : mesh->ref_xy);
    build_graphs(P);
    CK(cudaDeviceSynchronize());
    *out = h;
    return FSI_OK;
  } catch (...) {
    const int code = map_exception();
    if (h) fsi_destroy(h);
    return code;
  }
}

int fsi_create_problem(const fsi_params* params, const fsi_solid_mesh* mesh, const double* u0, const double* X0,
                       void* cuda_stream, fsi_problem** out) {
  return fsi_create_problem_budget(params, mesh, u0, X0, cuda_stream, 0, out);
}

int fsi_assemble_step(fsi_problem* h) {
  if (!h) return FSI_ERR_INVALID;
  try {
    CK(cudaGraphLaunch(h->P.g_assemble, h->P.stream));
    h->P.assembled = true;
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

static int status_from_ctl(const Ctl& c) {
  if (c.aflags & FLAG_OUT_OF_DOMAIN) return FSI_ERR_OUT_OF_DOMAIN;
  if (c.aflags & FLAG_CAPACITY) return FSI_ERR_CAPACITY;
  if (c.flags & FLAG_NAN) return FSI_ERR_NAN;
  if (c.flags & FLAG_BREAKDOWN) return FSI_ERR_BREAKDOWN;
  if (!c.converged) return FSI_ERR_NOT_CONVERGED;
  return FSI_OK;
}

static int fill_info(const Problem& P, fsi_solve_info* info) {
  const Ctl& c = *P.ctl_host;
  const int st = status_from_ctl(c);
  if (info) {
    info->iterations = c.its;
    info->restarts = std::max(0, c.cycles - 2);
    info->refinements = (P.prm.precision == 1) ? std::max(0, c.cycles - 1) : 0;
    info->status = st;
    info->rel_residual = c.last_true;
    info->rel_residual_est = (c.bnorm > 0) ? c.res / c.bnorm : c.res;
  }
  return st;
}

// queue S5-S8 (and the pressure normalisation) without waiting
static void enqueue_solve(Problem& P) {
  if (!P.assembled) CK(cudaGraphLaunch(P.g_assemble, P.stream));
  P.assembled = false;
  CK(cudaGraphLaunch(P.g_begin, P.stream));
  CK(cudaGraphLaunch(P.g_cycle, P.stream));
  CK(cudaGraphLaunch(P.g_finish, P.stream));
  CK(cudaMemcpyAsync(P.ctl_host, P.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, P.stream));
}

static void enqueue_advance(Problem& P) {
  CK(cudaMemcpyAsync(P.uold, P.x, 2 * (size_t)P.nU * 8, cudaMemcpyDeviceToDevice, P.stream));
  CK(cudaMemcpyAsync(P.Xold, P.x + P.offX, 2 * (size_t)P.nS * 8, cudaMemcpyDeviceToDevice, P.stream));
}

// One linear solve of the assembled block system (S5-S8) from the current
// iterate P.x.
static int solve_linear(Problem& P, fsi_solve_info* info) {
  {
    if (!P.host_loop) {
      enqueue_solve(P);
      CK(cudaStreamSynchronize(P.stream));
      return fill_info(P, info);
    }
    if (!P.assembled) CK(cudaGraphLaunch(P.g_assemble, P.stream));
    P.assembled = false;
    CK(cudaGraphLaunch(P.g_begin, P.stream));
    const int max_cycles = (P.prm.precision == 1) ? P.prm.max_refine + 1 : 1000000;
    Ctl& c = *P.ctl_host;
    for (int cyc = 0; cyc < max_cycles; ++cyc) {
      CK(cudaGraphLaunch(P.g_cstart, P.stream));
      CK(cudaMemcpyAsync(P.ctl_host, P.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, P.stream));
      CK(cudaStreamSynchronize(P.stream));
      while (c.cyc_active) {
        CK(cudaGraphLaunch(P.g_body, P.stream));
        CK(cudaMemcpyAsync(P.ctl_host, P.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, P.stream));
        CK(cudaStreamSynchronize(P.stream));
      }
      CK(cudaGraphLaunch(P.g_cend, P.stream));
      CK(cudaMemcpyAsync(P.ctl_host, P.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, P.stream));
      CK(cudaStreamSynchronize(P.stream));
      if (c.stop || c.aflags) break;
    }
    CK(cudaGraphLaunch(P.g_finish, P.stream));
    CK(cudaMemcpyAsync(P.ctl_host, P.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, P.stream));
    CK(cudaStreamSynchronize(P.stream));
    return fill_info(P, info);
  }
}

// Newton's method for the nonlinear solid law (Section 4: a nonlinear P(F)
// is handled by a Newton iteration): from X_0 = X^n, each iteration puts the
// tangent K_T(X_k) in place of A_s and K_T X_k - S(X_k) in the solid rows of
// the right-hand side, and solves the block system from the current iterate.
// Stops when max |X_{k+1} - X_k| <= newton_tol * max |X_{k+1} - X^n| (floor
// 1e-13).
static int solve_newton(Problem& P, fsi_solve_info* info) {
  const size_t n2 = 2 * (size_t)P.nS;
  std::vector<double> xk(n2), xn(n2), xo(n2);
  CK(cudaMemcpyAsync(P.x + P.offX, P.Xold, n2 * 8, cudaMemcpyDeviceToDevice, P.stream));
  CK(cudaMemcpyAsync(xo.data(), P.Xold, n2 * 8, cudaMemcpyDeviceToHost, P.stream));
  CK(cudaStreamSynchronize(P.stream));
  xk = xo;
  int total_its = 0, st = FSI_OK;
  fsi_solve_info last{};
  for (int it = 0; it < P.prm.newton_max; ++it) {
    launch(k_solid_tangent, nblk(P.nS, 128), 128, 0, P.stream, P.nS, P.ntp, P.nt, P.tris, P.area, P.tgrad,
           (const double*)(P.x + P.offX), P.prm.gamma, P.prm.eta, P.op64.Ssol.soff, P.op64.Ssol.len,
           P.op64.Ssol.col, P.kt64, P.kt32, P.b + P.offX, &P.ctl->aflags);
    st = solve_linear(P, &last);
    total_its += last.iterations;
    if (st != FSI_OK) break;
    CK(cudaMemcpyAsync(xn.data(), P.x + P.offX, n2 * 8, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaStreamSynchronize(P.stream));
    double dx = 0.0, disp = 0.0;
    for (size_t i = 0; i < n2; ++i) {
      dx = std::max(dx, std::fabs(xn[i] - xk[i]));
      disp = std::max(disp, std::fabs(xn[i] - xo[i]));
    }
    xk.swap(xn);
    last.newton_iterations = it + 1;
    if (dx <= std::max(P.prm.newton_tol * disp, 1e-13)) break;
    if (it + 1 == P.prm.newton_max) st = FSI_ERR_NOT_CONVERGED;
    P.assembled = true;  // C_f(X^n) and the linear right-hand side stay as assembled
  }
  P.assembled = false;
  last.iterations = total_its;
  last.status = st;
  if (info) *info = last;
  return st;
}

int fsi_solve_step(fsi_problem* h, fsi_solve_info* info) {
  if (!h) return FSI_ERR_INVALID;
  Problem& P = h->P;
  try {
    if (info) info->newton_iterations = 0;
    if (P.prm.solid_law == 1) return solve_newton(P, info);
    return solve_linear(P, info);
  } catch (...) {
    return map_exception();
  }
}

int fsi_step_async(fsi_problem* h) {
  if (!h || h->P.host_loop || h->P.prm.solid_law != 0) return FSI_ERR_INVALID;
  Problem& P = h->P;
  try {
    P.assembled = false;
    enqueue_solve(P);
    enqueue_advance(P);
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_step_poll(fsi_problem* h, fsi_solve_info* info) {
  if (!h) return FSI_ERR_INVALID;
  Problem& P = h->P;
  const cudaError_t q = cudaStreamQuery(P.stream);
  if (q == cudaErrorNotReady) return 1;
  if (q != cudaSuccess) return FSI_ERR_CUDA;
  fill_info(P, info);
  return 0;
}

int fsi_step_batch(fsi_problem* const* problems, int count, fsi_solve_info* infos) {
  if (!problems || count < 0) return FSI_ERR_INVALID;
  for (int i = 0; i < count; ++i)
    if (!problems[i] || problems[i]->P.host_loop || problems[i]->P.prm.solid_law != 0) return FSI_ERR_INVALID;
  int first_err = FSI_OK;
  try {
    // queue every instance's whole step on its own stream, then wait for all
    for (int i = 0; i < count; ++i) {
      Problem& P = problems[i]->P;
      P.assembled = false;
      enqueue_solve(P);
      enqueue_advance(P);
    }
    for (int i = 0; i < count; ++i) {
      Problem& P = problems[i]->P;
      CK(cudaStreamSynchronize(P.stream));
      const int st = fill_info(P, infos ? &infos[i] : nullptr);
      if (st != FSI_OK && first_err == FSI_OK) first_err = st;
    }
    return first_err;
  } catch (...) {
    return map_exception();
  }
}

int fsi_advance(fsi_problem* h) {
  if (!h) return FSI_ERR_INVALID;
  Problem& P = h->P;
  try {
    CK(cudaMemcpyAsync(P.uold, P.x, 2 * (size_t)P.nU * 8, cudaMemcpyDeviceToDevice, P.stream));
    CK(cudaMemcpyAsync(P.Xold, P.x + P.offX, 2 * (size_t)P.nS * 8, cudaMemcpyDeviceToDevice, P.stream));
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_step(fsi_problem* h, fsi_solve_info* info) {
  int st = fsi_assemble_step(h);
  if (st != FSI_OK) return st;
  st = fsi_solve_step(h, info);
  if (st != FSI_OK) return st;
  return fsi_advance(h);
}

int fsi_get_state(fsi_problem* h, double* u, double* pr, double* X, double* lam) {
  if (!h) return FSI_ERR_INVALID;
  Problem& P = h->P;
  try {
    const size_t nlat = (size_t)(2 * P.N + 1) * (2 * P.N + 1);
    if (u) {
      launch(k_state_out, nblk(nlat, 256), 256, 0, P.stream, nlat, P.l2n, P.wall, (const double*)P.x, P.V);
      CK(cudaMemcpyAsync(u, P.V, 2 * nlat * 8, cudaMemcpyDeviceToHost, P.stream));
    }
    if (pr) CK(cudaMemcpyAsync(pr, P.x + P.offP, 3 * (size_t)P.nP * 8, cudaMemcpyDeviceToHost, P.stream));
    if (X) CK(cudaMemcpyAsync(X, P.x + P.offX, 2 * (size_t)P.nS * 8, cudaMemcpyDeviceToHost, P.stream));
    if (lam) CK(cudaMemcpyAsync(lam, P.x + P.offL, 2 * (size_t)P.nS * 8, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaStreamSynchronize(P.stream));
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_set_state(fsi_problem* h, const double* u, const double* X) {
  if (!h) return FSI_ERR_INVALID;
  try {
    upload_state(h->P, u, X);
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_sizes(const fsi_problem* h, int* n_u, int* n_p, int* n_x, int* n_total) {
  if (!h) return FSI_ERR_INVALID;
  const Problem& P = h->P;
  if (n_u) *n_u = 2 * P.nU;
  if (n_p) *n_p = 3 * P.nP;
  if (n_x) *n_x = 2 * P.nS;
  if (n_total) *n_total = (int)P.n;
  return FSI_OK;
}

int fsi_get_points(fsi_problem* h, int* cell, double* xi, double* eta) {
  if (!h) return FSI_ERR_INVALID;
  Problem& P = h->P;
  if (P.prm.coupling != 0) return FSI_ERR_INVALID;  // the exact rule locates no points
  try {
    if (cell) CK(cudaMemcpyAsync(cell, P.cell, (size_t)P.nPts * 4, cudaMemcpyDeviceToHost, P.stream));
    if (xi) CK(cudaMemcpyAsync(xi, P.xi, (size_t)P.nPts * 8, cudaMemcpyDeviceToHost, P.stream));
    if (eta) CK(cudaMemcpyAsync(eta, P.eta, (size_t)P.nPts * 8, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaStreamSynchronize(P.stream));
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_get_coupling(fsi_problem* h, int* nnz, int* rows, int* lattice_cols, double* vals) {
  if (!h || !nnz) return FSI_ERR_INVALID;
  Problem& P = h->P;
  try {
    const size_t nslot = (size_t)nblk(P.nS, 32) * 32 * P.cf_cap;
    std::vector<int> len(P.nS), col(nslot);
    std::vector<double> val(nslot);
    CK(cudaMemcpyAsync(len.data(), P.cf_len, (size_t)P.nS * 4, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaMemcpyAsync(col.data(), P.cf_col, nslot * 4, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaMemcpyAsync(val.data(), P.cf_val, nslot * 8, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaStreamSynchronize(P.stream));
    int total = 0;
    for (int l = 0; l < P.nS; ++l) total += len[l];
    if (!rows) { *nnz = total; return FSI_OK; }
    if (*nnz < total) return FSI_ERR_INVALID;
    int q = 0;
    for (int l = 0; l < P.nS; ++l)
      for (int k = 0; k < len[l]; ++k) {
        const size_t slot = (size_t)(l >> 5) * 32 * P.cf_cap + (size_t)k * 32 + (l & 31);
        rows[q] = l;
        if (lattice_cols) lattice_cols[q] = P.hs.interior_lattice[col[slot]];
        if (vals) vals[q] = val[slot];
        ++q;
      }
    *nnz = total;
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_apply_operator(fsi_problem* h, const double* xh, double* yh, int precision) {
  if (!h || !xh || !yh) return FSI_ERR_INVALID;
  Problem& P = h->P;
  if (precision == 1 && P.prm.precision != 1) return FSI_ERR_INVALID;
  try {
    double* tmp = P.V;  // first basis vector as scratch
    CK(cudaMemcpyAsync(tmp, xh, P.n * 8, cudaMemcpyHostToDevice, P.stream));
    if (precision == 1) {
      launch(k_convert<double, float>, nblk(P.n, 256), 256, 0, P.stream, P.n, tmp, P.p32.vin);
      full_launch<float, double>(P.p32, P.p32.vin, P.w, nullptr, 1.0, 0.0, nullptr, 0, nullptr, P.stream);
    } else {
      full_launch<double, double>(P.p64, tmp, P.w, nullptr, 1.0, 0.0, nullptr, 0, nullptr, P.stream);
    }
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(yh, P.w, P.n * 8, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaStreamSynchronize(P.stream));
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_apply_preconditioner(fsi_problem* h, const double* vh, double* zh, int precision) {
  if (!h || !vh || !zh) return FSI_ERR_INVALID;
  Problem& P = h->P;
  if (precision == 1 && P.prm.precision != 1) return FSI_ERR_INVALID;
  try {
    double* tmp = P.V;
    CK(cudaMemcpyAsync(tmp, vh, P.n * 8, cudaMemcpyHostToDevice, P.stream));
    if (precision == 1) {
      launch(k_convert<double, float>, nblk(P.n, 256), 256, 0, P.stream, P.n, tmp, P.p32.vin);
      precond_launch(P, P.p32, P.stream);
      launch(k_convert<float, double>, nblk(P.n, 256), 256, 0, P.stream, P.n, P.p32.zw, P.w);
    } else {
      launch(k_copy<double>, nblk(P.n, 256), 256, 0, P.stream, P.n, tmp, P.p64.vin);
      precond_launch(P, P.p64, P.stream);
      launch(k_copy<double>, nblk(P.n, 256), 256, 0, P.stream, P.n, P.p64.zw, P.w);
    }
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(zh, P.w, P.n * 8, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaStreamSynchronize(P.stream));
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_graph_kernel_counts(const fsi_problem* h, int* counts) {
  if (!h || !counts) return FSI_ERR_INVALID;
  const Problem& P = h->P;
  counts[0] = P.kn_assemble; counts[1] = P.kn_begin; counts[2] = P.kn_cycle;
  counts[3] = P.kn_body; counts[4] = P.kn_finish;
  return FSI_OK;
}

int fsi_time_kernel(fsi_problem* h, int which, int reps, double* avg_ms, double* bytes) {
  if (!h || !avg_ms || !bytes || reps <= 0) return FSI_ERR_INVALID;
  Problem& P = h->P;
  if ((which == 0 || which == 2 || (which >= 4 && which <= 7) || (which >= 10 && which <= 13)) &&
      P.prm.precision != 1)
    return FSI_ERR_INVALID;
  if (which == 8 && P.prm.coupling != 0) return FSI_ERR_INVALID;  // would overwrite the exact rows
  if (which == 9 && P.prm.coupling != 1) return FSI_ERR_INVALID;
  if (which == 3 && P.p64.mgU.lv.empty()) return FSI_ERR_INVALID;  // no FP64 hierarchy in mixed mode
  try {
    // total C_f entries of the last assembly
    std::vector<int> len(P.nS);
    CK(cudaMemcpy(len.data(), P.cf_len, (size_t)P.nS * 4, cudaMemcpyDeviceToHost));
    double cfnnz = 0;
    for (int v : len) cfnnz += v;
    const size_t flush_n = (size_t)(256u << 20) / sizeof(uint4);
    uint4* fl = nullptr;
    CK(cudaMalloc(&fl, flush_n * sizeof(uint4)));
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    double total = 0;
    cudaStream_t s = P.stream;
    const HostBlockMatrix& A0 = P.hs.levels[0].A;
    // the stored matrix of the smoothing steps, for the timing alone
    struct Held : Arena {
      ~Held() { release(); }
    } held;
    Sell<float> A2;
    Sell<double> A3;
    if (which == 2 || (which == 3 && P.p64.mgU.lv[0].mfo.N == 0)) {
      const SellHost sa = to_sell(A0);
      if (which == 2) A2 = upload_sell<float>(held, sa);
      else A3 = upload_sell<double>(held, sa);
      if (P.prm.autotune == 1) {
        if (which == 2) autotune_sell<float>(A2, sa.soff[sa.nslices]);
        else autotune_sell<double>(A3, sa.soff[sa.nslices]);
      }
    }
    for (int r = 0; r < reps + 1; ++r) {
      if (which < 4 || which >= 10) launch(k_flush, 2 * 152, 512, 0, s, flush_n, fl, (unsigned)r);
      CK(cudaEventRecord(e0, s));
      switch (which) {
        case 0:  // full operator, FP32 (mixed inner iteration)
          full_launch<float, double>(P.p32, P.p32.zw, P.w, nullptr, 1.0, 0.0, nullptr, 0, nullptr, s);
          *bytes = fullop_bytes<float>(P, P.p32.mf.N > 0, cfnnz, sizeof(float), sizeof(double));
          break;
        case 1:  // full operator, FP64 (residual / FP64 iteration)
          full_launch<double, double>(P.p64, P.x, P.w, P.b, -1.0, 1.0, nullptr, 0, nullptr, s);
          *bytes = fullop_bytes<double>(P, P.p64.mf.N > 0, cfnnz, 16, 8);
          break;
        case 2: {  // finest velocity Chebyshev step on the stored matrix, FP32
          MGLevel<float>& L = P.p32.mgU.lv[0];
          SpmvArgs<float> a;
          a.x = L.x; a.y = L.x2; a.z = L.b; a.d = L.d; a.dinv = L.dinv; a.c1 = 0.5f; a.c2 = 0.5f;
          sell_launch(A2, MODE_CHEB, a, s);
          *bytes = sell_bytes<float>(A0) + 6.0 * L.n * sizeof(float);
          break;
        }
        case 3: {  // finest velocity Chebyshev step as the FP64 V-cycle runs it
          MGLevel<double>& L = P.p64.mgU.lv[0];
          SpmvArgs<double> a;
          a.x = L.x; a.y = L.x2; a.z = L.b; a.d = L.d; a.dinv = L.dinv; a.c1 = 0.5; a.c2 = 0.5;
          if (L.mfo.N > 0) level_launch(L, MODE_CHEB, a, s);
          else sell_launch(A3, MODE_CHEB, a, s);
          *bytes = (L.mfo.N > 0 ? 0.0 : sell_bytes<double>(A0)) + 6.0 * L.n * sizeof(double);
          break;
        }
        case 4:    // one V-cycle on the Q2 velocity hierarchy, FP32
        case 5: {  // one V-cycle on the pressure Laplacian hierarchy, FP32
          MG<float>& mg = (which == 4) ? P.p32.mgU : P.p32.mgP;
          vcycle<float>(mg, 0, s, mg.lv[0].mf ? mg.lv[0].x : mg.lv[0].x2);
          *bytes = vcycle_work<float>(P.hs, mg, which == 5).bytes;
          break;
        }
        case 8:    // C_f rows by the point rule at located points (S2 + S4)
          point_rule_launch(P, s);
          *bytes = 0;
          break;
        case 9:    // C_f rows by the exact rule (mesh intersection)
          exact_rule_launch(P, s);
          *bytes = 0;
          break;
        case 10:   // fused finest-level launches, FP32: velocity down / up,
        case 11:   // pressure down / up (the level's current vectors)
        case 12:
        case 13: {
          MG<float>& mg = (which <= 11) ? P.p32.mgU : P.p32.mgP;
          MGLevel<float>& L = mg.lv[0];
          if (!L.mf) {
            cudaFree(fl);
            return FSI_ERR_INVALID;
          }
          MGLevel<float>& C = mg.lv[1];
          const bool up = (which & 1) != 0;
          if (up) mf_up_launch(mg, 0, L.b, C.x, L.x, nullptr, s);
          else mf_down_launch(mg, 0, L.b, s);
          *bytes = mf_work(P.hs, 0, which >= 12, up, mg.degree, sizeof(float)).bytes;
          break;
        }
        case 6:    // the cluster launch of the velocity coarse levels alone, FP32
        case 7: {  // the same for the pressure Laplacian
          MG<float>& mg = (which == 6) ? P.p32.mgU : P.p32.mgP;
          if (!mg.cl.on) {
            cudaFree(fl);
            return FSI_ERR_INVALID;
          }
          MGLevel<float>& L = mg.lv[mg.cl.lc];
          cluster_launch<float>(mg, L.b, L.x, s);
          *bytes = 0;
          break;
        }
        default:
          cudaFree(fl);
          return FSI_ERR_INVALID;
      }
      CK(cudaEventRecord(e1, s));
      CK(cudaEventSynchronize(e1));
      float ms = 0;
      CK(cudaEventElapsedTime(&ms, e0, e1));
      if (r > 0) total += ms;  // first launch is a warm-up
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(fl);
    *avg_ms = total / reps;
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

int fsi_kernel_flops(fsi_problem* h, int which, double* flops) {
  if (!h || !flops) return FSI_ERR_INVALID;
  Problem& P = h->P;
  if (P.prm.precision != 1) return FSI_ERR_INVALID;
  if (which == 4 || which == 5) {
    *flops = vcycle_work<float>(P.hs, which == 4 ? P.p32.mgU : P.p32.mgP, which == 5).flops;
    return FSI_OK;
  }
  if (which < 10 || which > 13) return FSI_ERR_INVALID;
  const MG<float>& mg = (which <= 11) ? P.p32.mgU : P.p32.mgP;
  if (mg.lv.empty() || !mg.lv[0].mf) return FSI_ERR_INVALID;
  *flops = mf_work(P.hs, 0, which >= 12, (which & 1) != 0, mg.degree, sizeof(float)).flops;
  return FSI_OK;
}

int fsi_interior_nodes(const fsi_problem* h, int* lattice_ids) {
  if (!h || !lattice_ids) return FSI_ERR_INVALID;
  std::copy(h->P.hs.interior_lattice.begin(), h->P.hs.interior_lattice.end(), lattice_ids);
  return FSI_OK;
}

int fsi_get_rhs(fsi_problem* h, double* bh) {
  if (!h || !bh) return FSI_ERR_INVALID;
  Problem& P = h->P;
  try {
    CK(cudaMemcpyAsync(bh, P.b, P.n * 8, cudaMemcpyDeviceToHost, P.stream));
    CK(cudaStreamSynchronize(P.stream));
    return FSI_OK;
  } catch (...) {
    return map_exception();
  }
}

void fsi_destroy(fsi_problem* h) {
  if (!h) return;
  Problem& P = h->P;
  cudaGraphExec_t ex[7] = {P.g_assemble, P.g_begin, P.g_cycle, P.g_finish, P.g_cstart, P.g_body, P.g_cend};
  cudaGraph_t gr[7] = {P.gr_assemble, P.gr_begin, P.gr_cycle, P.gr_finish, P.gr_cstart, P.gr_body, P.gr_cend};
  if (P.stream) cudaStreamSynchronize(P.stream);
  for (auto e : ex) if (e) cudaGraphExecDestroy(e);
  for (auto g : gr) if (g) cudaGraphDestroy(g);
  P.ar.release();
  if (P.ctl_host) cudaFreeHost(P.ctl_host);
  if (P.s2) cudaStreamDestroy(P.s2);
  if (P.s3) cudaStreamDestroy(P.s3);
  if (P.s4) cudaStreamDestroy(P.s4);
  if (P.s5) cudaStreamDestroy(P.s5);
  if (P.ev_join2) cudaEventDestroy(P.ev_join2);
  if (P.ev_fork2) cudaEventDestroy(P.ev_fork2);
  if (P.ev_fork) cudaEventDestroy(P.ev_fork);
  if (P.ev_join) cudaEventDestroy(P.ev_join);
  if (P.own_stream && P.stream) cudaStreamDestroy(P.stream);
  delete h;
}

const char* fsi_status_str(int s) {
  switch (s) {
    case FSI_OK: return "ok";
    case FSI_ERR_INVALID: return "invalid argument";
    case FSI_ERR_OOM: return "device out of memory";
    case FSI_ERR_BUDGET: return "footprint above budget";
    case FSI_ERR_OUT_OF_DOMAIN: return "solid point outside the fluid domain";
    case FSI_ERR_NOT_CONVERGED: return "not converged";
    case FSI_ERR_BREAKDOWN: return "Krylov breakdown";
    case FSI_ERR_NAN: return "NaN or Inf in the residual";
    case FSI_ERR_TIMEOUT: return "bounded device wait ran out";
    case FSI_ERR_CAPACITY: return "coupling row over capacity";
    case FSI_ERR_CUDA: return "CUDA error";
    default: return "unknown status";
  }
}

}  // extern "C"
