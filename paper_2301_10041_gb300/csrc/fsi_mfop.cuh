// Matrix-free operators of the uniform grid: one thread per Q2 node and pressure
// cell in FP32, per component in FP64, the stencils of fsi_mgfused.cuh as kernel parameters.
//
// They replace the sliced-ELL products (k_sell, k_fullmv, k_stokes_res) where
// the grid has its stencils (N >= 4) and the caller does not ask for the
// per-level sparse kernels:
//
//  * the fluid rows of the full operator, in both precisions.  The sparse form
//    reads 36 (FP32: 20) bytes per 2x2 block, 600 MB per FP32 product at
//    N = 512; the matrix-free form reads the vectors only;
//  * the FP64 multigrid levels.  An FP64 instruction of a warp holds its pipe
//    for 64 cycles however few lanes are active, and the sparse kernel spends 30
//    of them on 8 rows (16 products, 4 reduction steps, an epilogue with one lane
//    in four): 120 per 32 rows.  A thread per component takes 60: the blocks of
//    A = (rho/dt) M + K are symmetric with equal off-diagonal entries, and these
//    vanish when the two nodes share a grid line (the mixed derivative of a
//    product basis), which the host checks on the assembled rows (MfOp).
#pragma once
#include "fsi_kernels.cuh"
#include "fsi_mgfused.cuh"

namespace fsi {

// A: (xx, xy = yx, yy) per [node type][dy+2][dx+2]; divB as in MfRes.
template <class T>
struct MfOp {
  int N = 0;          // 0: no stencils, the sparse kernels run
  T c[4][5][5][3];
  T divB[3][9][2];
};

// Values per thread: both components of a node in FP32, one in FP64, where
// the pipe makes every product 64 cycles deep and a corner node has 82 of them.
template <class T>
struct MfLanes {
  static constexpr int C = sizeof(T) == 8 ? 1 : 2;   // components per thread
  static constexpr int S = 2 / C;                    // threads per node
};

// Velocity nodes are numbered by type, each type row by row; a warp takes 32 / S
// consecutive nodes of one type.
__host__ __device__ __forceinline__ int mfop_count(int N, int t) {
  return ((t & 1) ? N : N - 1) * ((t >> 1) ? N : N - 1);
}
template <class T>
inline unsigned mfop_grid(int N) {   // CTAs of 4 warps
  int w = 0;
  for (int t = 0; t < 4; ++t) w += (MfLanes<T>::S * mfop_count(N, t) + 31) / 32;
  return (unsigned)((w + 3) / 4);
}

// this thread's C values of vector v at entry r = 2 id + d
template <class T, int C>
__device__ __forceinline__ void mfop_ld(const T* __restrict__ v, size_t r, T o[C]) {
  if constexpr (C == 2) {
    const typename Vec2<T>::type q = *reinterpret_cast<const typename Vec2<T>::type*>(v + r);
    o[0] = q.x;
    o[1] = q.y;
  } else {
    o[0] = v[r];
  }
}
template <class T, int C>
__device__ __forceinline__ void mfop_st(T* __restrict__ v, size_t r, const T o[C]) {
  if constexpr (C == 2) {
    typename Vec2<T>::type q;
    q.x = o[0];
    q.y = o[1];
    *reinterpret_cast<typename Vec2<T>::type*>(v + r) = q;
  } else {
    v[r] = o[0];
  }
}

// s = (A x) at the interior node (ix, iy) of type TAU, component d (FP64) or
// both; x in node order, absent (wall) neighbours are zero
template <int TAU, class T>
__device__ __forceinline__ void mfop_vel(const MfOp<T>& op, const T* __restrict__ x, int ix, int iy, int d,
                                         T s[MfLanes<T>::C]) {
  using T2 = typename Vec2<T>::type;
  constexpr int PX = TAU & 1, PY = TAU >> 1, C = MfLanes<T>::C;
  constexpr int RX = PX ? 1 : 2, RY = PY ? 1 : 2;
  const int N = op.N;
  const bool xl = ix - RX >= 1, xr = ix + RX <= 2 * N - 1, yl = iy - RY >= 1, yr = iy + RY <= 2 * N - 1;
  T a0 = 0, a1 = 0, b0 = 0, b1 = 0;
#pragma unroll
  for (int dy = -RY; dy <= RY; ++dy) {
    T2 v[2 * RX + 1];
#pragma unroll
    for (int dx = -RX; dx <= RX; ++dx) {
      const bool in = (dx > -RX || xl) && (dx < RX || xr) && (dy > -RY || yl) && (dy < RY || yr);
      v[dx + RX].x = v[dx + RX].y = 0;
      if (in) {
        constexpr int kType[2][2] = {{0, 1}, {2, 3}};
        const int t2 = kType[(PY + dy) & 1][(PX + dx) & 1];
        const int jx = ix + dx, jy = iy + dy;
        const int id = t2 == 0 ? mf_vnode_t<0>(N, jx, jy)
                               : (t2 == 1 ? mf_vnode_t<1>(N, jx, jy)
                                          : (t2 == 2 ? mf_vnode_t<2>(N, jx, jy) : mf_vnode_t<3>(N, jx, jy)));
        v[dx + RX] = reinterpret_cast<const T2*>(x)[id];
      }
    }
#pragma unroll
    for (int dx = -RX; dx <= RX; ++dx) {
      const T* c = op.c[TAU][dy + 2][dx + 2];
      const T2 q = v[dx + RX];
      if constexpr (C == 2) {
        a0 = fma(c[0], q.x, a0);
        a1 = fma(c[2], q.y, a1);
        if (dx != 0 && dy != 0) {
          b0 = fma(c[1], q.y, b0);
          b1 = fma(c[1], q.x, b1);
        }
      } else {
        a0 = fma(d ? c[2] : c[0], d ? q.y : q.x, a0);
        if (dx != 0 && dy != 0) b0 = fma(c[1], d ? q.x : q.y, b0);
      }
    }
  }
  s[0] = a0 + b0;
  if constexpr (C == 2) s[1] = a1 + b1;
}

// s += -B^T p at a node (p: three values per cell of the whole grid)
template <int TAU, class T>
__device__ __forceinline__ void mfop_btp(const MfOp<T>& op, const T* __restrict__ p, int ix, int iy, int d,
                                         T s[MfLanes<T>::C]) {
  constexpr int PX = TAU & 1, PY = TAU >> 1, C = MfLanes<T>::C;
#pragma unroll
  for (int j = 0; j < (PY ? 1 : 2); ++j)
#pragma unroll
    for (int i = 0; i < (PX ? 1 : 2); ++i) {
      const int aa = PX ? 1 : (i == 0 ? 2 : 0), ab = PY ? 1 : (j == 0 ? 2 : 0);
      const int cx = (ix - aa) >> 1, cy = (iy - ab) >> 1, al = 3 * ab + aa;
      const T* __restrict__ q = p + 3 * ((size_t)cy * op.N + cx);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if constexpr (C == 2) {
          s[0] = fma(op.divB[k][al][0], q[k], s[0]);
          s[1] = fma(op.divB[k][al][1], q[k], s[1]);
        } else {
          s[0] = fma(d ? op.divB[k][al][1] : op.divB[k][al][0], q[k], s[0]);
        }
      }
    }
}

// y = rows k0 .. k0 + K - 1 of -B u at cell c
template <int K, class T>
__device__ __forceinline__ void mfop_bu(const MfOp<T>& op, const T* __restrict__ u, int c, int k0, T y[K]) {
  using T2 = typename Vec2<T>::type;
  const int N = op.N, cx = c % N, cy = c / N;
  T2 v[9];
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const int jx = 2 * cx + b % 3, jy = 2 * cy + b / 3;
    v[b].x = v[b].y = 0;
    if (mf_vinterior(N, jx, jy)) {
      constexpr int kTau[9] = {0, 1, 0, 2, 3, 2, 0, 1, 0};
      const int id = kTau[b] == 0 ? mf_vnode_t<0>(N, jx, jy)
                                  : (kTau[b] == 1 ? mf_vnode_t<1>(N, jx, jy)
                                                  : (kTau[b] == 2 ? mf_vnode_t<2>(N, jx, jy) : mf_vnode_t<3>(N, jx, jy)));
      v[b] = reinterpret_cast<const T2*>(u)[id];
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    y[k] = 0;
#pragma unroll
    for (int b = 0; b < 9; ++b) {
      T bx, by;
      if constexpr (K == 3) {
        bx = op.divB[k][b][0];
        by = op.divB[k][b][1];
      } else {   // the row is a value: pick its entries off the FP64 pipe
        bx = k0 == 0 ? op.divB[0][b][0] : (k0 == 1 ? op.divB[1][b][0] : op.divB[2][b][0]);
        by = k0 == 0 ? op.divB[0][b][1] : (k0 == 1 ? op.divB[1][b][1] : op.divB[2][b][1]);
      }
      y[k] = fma(by, v[b].y, fma(bx, v[b].x, y[k]));
    }
  }
}
// pressure rows of a cell per thread
template <class T>
__host__ __device__ constexpr int mfop_prows() { return sizeof(T) == 8 ? 1 : 3; }

// fn(type, node id, ix, iy, d) for this warp's nodes; `warp` counts over the grid
template <class T, class F>
__device__ __forceinline__ void mfop_nodes(int N, int warp, F&& fn) {
  constexpr int S = MfLanes<T>::S;
  const int lane = threadIdx.x & 31;
  int w = warp, base = 0;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int cnt = mfop_count(N, t), nw = (S * cnt + 31) / 32;
    if (w >= 0 && w < nw) {
      const int e = 32 * w + lane, k = e / S, d = e - S * k;
      if (k < cnt) {
        const int wd = (t & 1) ? N : N - 1, r = k / wd, q = k - r * wd;
        const int ix = (t & 1) ? 2 * q + 1 : 2 * q + 2, iy = (t >> 1) ? 2 * r + 1 : 2 * r + 2;
        switch (t) {
          case 0: fn(std::integral_constant<int, 0>(), base + k, ix, iy, d); break;
          case 1: fn(std::integral_constant<int, 1>(), base + k, ix, iy, d); break;
          case 2: fn(std::integral_constant<int, 2>(), base + k, ix, iy, d); break;
          default: fn(std::integral_constant<int, 3>(), base + k, ix, iy, d); break;
        }
      }
    }
    w -= nw;
    base += cnt;
  }
}

// One velocity level product with the epilogues of k_sell (the modes the
// velocity hierarchy uses): AXPBY, CHEB, CHEB0 (with the Richardson update).
template <class T, int MODE>
__global__ void __launch_bounds__(128) k_mfv(const __grid_constant__ MfOp<T> op, const __grid_constant__ SpmvArgs<T> a) {
  constexpr int C = MfLanes<T>::C;
  pdl_begin();
  mfop_nodes<T>(op.N, blockIdx.x * 4 + (threadIdx.x >> 5), [&](auto tc, int id, int ix, int iy, int dd) {
    const size_t r = 2 * (size_t)id + dd;
    T z[C] = {}, d[C] = {}, dv[C] = {}, x[C] = {}, s[C], y[C];
    if (a.z) mfop_ld<T, C>(a.z, r, z);
    if (MODE == MODE_CHEB) mfop_ld<T, C>(a.d, r, d);
    if (MODE != MODE_AXPBY) {
      mfop_ld<T, C>(a.dinv, r, dv);
      mfop_ld<T, C>(a.x, r, x);
    }
    mfop_vel<decltype(tc)::value, T>(op, a.x, ix, iy, dd, s);
    if (MODE == MODE_AXPBY) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        y[c] = a.alpha * s[c];
        if (a.z) y[c] = fma(a.beta, z[c], y[c]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        d[c] = a.c1 * d[c] + a.c2 * dv[c] * (z[c] - s[c]);
        y[c] = x[c] + d[c];
      }
      mfop_st<T, C>(a.d, r, d);
      if (a.acc) {
        T o[C];
        mfop_ld<T, C>(a.acc, r, o);
#pragma unroll
        for (int c = 0; c < C; ++c) o[c] = fma(a.omega, y[c], o[c]);
        mfop_st<T, C>(a.acc, r, o);
      }
    }
    mfop_st<T, C>(a.y, r, y);
  });
}

// t = z - (-B^T) p, the velocity smoother's input and its start d = x = c0 D^-1 t
template <class T>
__global__ void __launch_bounds__(128) k_mfv_start(const __grid_constant__ MfOp<T> op, const T* __restrict__ z,
                                                   const T* __restrict__ p, const T* __restrict__ dinv, T c0,
                                                   T* __restrict__ t, T* __restrict__ d, T* __restrict__ x) {
  constexpr int C = MfLanes<T>::C;
  pdl_begin();
  mfop_nodes<T>(op.N, blockIdx.x * 4 + (threadIdx.x >> 5), [&](auto tc, int id, int ix, int iy, int dd) {
    const size_t r = 2 * (size_t)id + dd;
    T b[C], s[C] = {}, di[C];
    mfop_ld<T, C>(z, r, b);
    mfop_ld<T, C>(dinv, r, di);
    mfop_btp<decltype(tc)::value, T>(op, p, ix, iy, dd, s);
#pragma unroll
    for (int c = 0; c < C; ++c) b[c] -= s[c];
    mfop_st<T, C>(t, r, b);
#pragma unroll
    for (int c = 0; c < C; ++c) b[c] *= c0 * di[c];
    mfop_st<T, C>(d, r, b);
    mfop_st<T, C>(x, r, b);
  });
}

// One pressure level product: CHEB and CHEB0 with the Cahouet-Chabard epilogue
// of k_sell, a thread per row.  The rows of the 3x3 blocks come from the level's
// stencil table (fsi_mgfused.cuh) through L1: 27 FP64 multiply-adds take far
// longer than their loads.
template <class T, int MODE>
__global__ void __launch_bounds__(96) k_mfp(int N, const T* __restrict__ tab, const __grid_constant__ SpmvArgs<T> a) {
  pdl_begin();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= 3 * N * N) return;
  const int c = r / 3, k = r - 3 * c, cx = c % N, cy = c / N;
  const T z = a.z[r], x = a.x[r], dv = a.dinv[r], d = MODE == MODE_CHEB ? a.d[r] : (T)0;
  const T smp = a.sout ? a.smp[r] : (T)0, sv = a.sout ? a.sv[r] : (T)0, acc = a.acc ? a.acc[r] : (T)0;
  const T* __restrict__ blk = tab + kMfPresVar * mf_variant(N, cx, cy) + 3 * k;
  T s[3] = {0, 0, 0};
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy) {
#pragma unroll
    for (int dx = -1; dx <= 1; ++dx) {
      if (!mf_cin(N, cx + dx, cy + dy)) continue;
      const T* __restrict__ xn = a.x + 3 * ((size_t)(cy + dy) * N + cx + dx);
      const T* __restrict__ b = blk + kMfPresBlk * (3 * (dy + 1) + dx + 1);
      s[dy + 1] = fma(b[2], xn[2], fma(b[1], xn[1], fma(b[0], xn[0], s[dy + 1])));
    }
  }
  const T dn = a.c1 * d + a.c2 * dv * (z - ((s[0] + s[1]) + s[2]));
  a.d[r] = dn;
  const T y = x + dn;
  a.y[r] = y;
  T o = y;
  if (a.sout) {
    o = -(a.snu * smp * sv + a.srdt * y);
    a.sout[r] = o;
  }
  if (a.acc) a.acc[r] = fma(a.omega, o, acc);
}

// Residual of the Stokes block, as k_stokes_res: t_u = r_u - A z_u - (-B^T) z_p,
// t_p = r_p - (-B) z_u, the pressure rows also starting their V-cycle.
template <class T>
__global__ void __launch_bounds__(128) k_mf_stokes_res(const __grid_constant__ MfOp<T> op, int gU, int nU, int nP,
                                                       const T* __restrict__ z, const T* __restrict__ ru,
                                                       const T* __restrict__ rp, T* __restrict__ t,
                                                       const T* __restrict__ pdinv, T pc0, T* __restrict__ pb,
                                                       T* __restrict__ pd, T* __restrict__ px) {
  constexpr int C = MfLanes<T>::C, K = mfop_prows<T>();
  pdl_begin();
  const size_t offP = 2 * (size_t)nU;
  if ((int)blockIdx.x < gU) {
    mfop_nodes<T>(op.N, blockIdx.x * 4 + (threadIdx.x >> 5), [&](auto tc, int id, int ix, int iy, int d) {
      const size_t r = 2 * (size_t)id + d;
      T s[C], o[C];
      mfop_ld<T, C>(ru, r, o);
      mfop_vel<decltype(tc)::value, T>(op, z, ix, iy, d, s);
      mfop_btp<decltype(tc)::value, T>(op, z + offP, ix, iy, d, s);
#pragma unroll
      for (int c = 0; c < C; ++c) o[c] -= s[c];
      mfop_st<T, C>(t, r, o);
    });
    return;
  }
  const int e = (blockIdx.x - gU) * blockDim.x + threadIdx.x;
  const int c = e / (3 / K), k0 = e - c * (3 / K);
  if (c >= nP) return;
  T s[K];
  mfop_bu<K, T>(op, z, c, k0, s);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const size_t i = 3 * (size_t)c + k0 + k;
    const T tv = rp[i] - s[k];
    t[offP + i] = tv;
    if (pd) {
      pb[i] = tv;
      const T v = pc0 * pdinv[i] * tv;
      pd[i] = v;
      px[i] = v;
    }
  }
}

// y = alpha A x + beta z for the block operator, as k_fullmv with the fluid
// rows matrix-free: a thread per node (its C_f^T row four entries at a time),
// a thread per cell, and the solid rows as there.
template <class T, class TY>
__global__ void __launch_bounds__(128) k_fullmv_mf(const __grid_constant__ FullOp<T> op, const __grid_constant__ MfOp<T> mf,
                                                   int gU, int gP, const T* __restrict__ x, TY* __restrict__ y,
                                                   const TY* __restrict__ z, TY alpha, TY beta, T* __restrict__ Z,
                                                   size_t zld, const Ctl* __restrict__ ctl) {
  using T2 = typename Vec2<T>::type;
  constexpr int C = MfLanes<T>::C, K = mfop_prows<T>();
  pdl_begin();
  const int b = blockIdx.x;
  const size_t offP = 2 * (size_t)op.nU, offX = offP + 3 * (size_t)op.nP, offL = offX + 2 * (size_t)op.nS;
  T* Zc = Z ? Z + (size_t)ctl->j * zld : nullptr;
  if (b < gU) {
    mfop_nodes<T>(mf.N, b * 4 + (threadIdx.x >> 5), [&](auto tc, int id, int ix, int iy, int d) {
      const size_t r = 2 * (size_t)id + d;
      T own[C], s[C];
      if (Zc) {
        mfop_ld<T, C>(x, r, own);
        mfop_st<T, C>(Zc, r, own);
      }
      const int k1 = op.cft_ptr[id + 1];
      int k = op.cft_ptr[id];
      mfop_vel<decltype(tc)::value, T>(mf, x, ix, iy, d, s);
      mfop_btp<decltype(tc)::value, T>(mf, x + offP, ix, iy, d, s);
      const T2* __restrict__ lam = reinterpret_cast<const T2*>(x + offL);
      for (; k < k1; k += 4) {
        T v[4];
        T2 l[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          v[u] = l[u].x = l[u].y = 0;
          if (k + u < k1) {   // an absent entry reads nothing: 0 times an infinity would not be 0
            v[u] = op.cft_val[k + u];
            l[u] = lam[op.cft_col[k + u]];
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if constexpr (C == 2) {
            s[0] = fma(v[u], l[u].x, s[0]);
            s[1] = fma(v[u], l[u].y, s[1]);
          } else {
            s[0] = fma(v[u], d ? l[u].y : l[u].x, s[0]);
          }
        }
      }
      TY o[C], zv[C];
      if (z) mfop_ld<TY, C>(z, r, zv);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        o[c] = alpha * (TY)s[c];
        if (z) o[c] += beta * zv[c];
      }
      mfop_st<TY, C>(y, r, o);
    });
  } else if (b < gU + gP) {
    const int e = (b - gU) * 128 + threadIdx.x;
    const int c = e / (3 / K), k0 = e - c * (3 / K);
    if (c >= op.nP) return;
    T s[K];
    mfop_bu<K, T>(mf, x, c, k0, s);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const size_t i = offP + 3 * (size_t)c + k0 + k;
      TY o = alpha * (TY)s[k];
      if (z) o += beta * z[i];
      y[i] = o;
      if (Zc) Zc[i] = x[i];
    }
  } else {
    fullmv_solid_rows<T, T, TY>(op, b - gU - gP, x, y, z, alpha, beta);
    if (Zc) {
      const int c = 64 * (b - gU - gP) + (threadIdx.x & 63);
      const size_t o = (threadIdx.x < 64 ? offX : offL) + c;
      if (c < 2 * op.nS) Zc[o] = x[o];
    }
  }
}

}  // namespace fsi
