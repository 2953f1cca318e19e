// Block factorisation of the block-tridiagonal s I - L, one factorisation per
// shift reused by every later solve (Sec. III.A).
//
// With the unknowns ordered by streamwise column, s I - L has diagonal blocks
// D_i, sub-diagonal blocks A_i = -L_{i,i-1} and super-diagonal blocks
// C_i = -L_{i,i+1} (b x b, A_i and C_i with at most 3q entries per row).  The
// block LU runs from both ends to the middle column m = nx / 2 at once, so that
// the chain of dependent blocks is half as long and every launch has twice the
// problems (half 0: columns 0, 1, .. m - 1; half 1: nx - 1, nx - 2, .. m + 1):
//     S_0 = D_0,  G_i = S_i^{-1},  X_i = G_i C_i,  S_{i+1} = D_{i+1} - A_{i+1} X_i
//     S_{nx-1} = D_{nx-1},  X_i = G_i A_i,  S_{i-1} = D_{i-1} - C_{i-1} X_i
//     S_m = D_m - A_m X_{m-1} - C_m X_{m+1}.
// Work buffers hold both halves: problem f of half h at index h F + f.  Measured
// against the same kernels run from one end, factorisation and solves: two
// frequencies of 128 x 64 points 13.5 ms instead of 25.5, six of 512 x 256 points
// 401 instead of 619; in FP64 four of 128 x 64 points and their gradient 75
// instead of 101.
// G_i is formed explicitly, so every later solve is a dense block product
// instead of a pair of triangular solves.  This file holds the Schur update and
// the Gauss-Jordan inversion used for FP64 factors and for the FP32 shapes that
// the slab form (factor_w.cu) does not take; both pivot implicitly (rows never
// move; rowpiv[r] is the column row r pivoted for, pivslot[c] the row that
// pivoted column c).  Per panel K of 16 columns:
//   panel  : one cluster of CTAs per problem applies the previous panel's
//            transformation to K and runs the 16 eliminations
//            (gjp_panel_kernel);
//   gather : B = M[P, :], P the panel's pivot rows, saved before they change;
//   update : M[r, m] += M[r, K] B[:, m] (r not in P), M[P, m] = M[P, K] B[:, m]
//            for the columns m outside K and the next panel, on all SMs beside
//            the next panel (gjp_update_kernel).
#include <cuda.h>

#include <algorithm>

#include "rr_internal.cuh"
#include "tc.cuh"

namespace {

__device__ __forceinline__ int slotx(int dx, int dy) { return (dx + 1) * 3 + (dy + 1); }

// M = D_i + L_{i,i+dx} X_{i+dx} (dx = -1 in half 0, +1 in half 1; no X for the end
// columns), i.e. S_i = D_i - A_i X_{i-1} and its mirror image; with add, M +=
// L_{i,i+dx} X_{i+dx} only (the middle column's second neighbour).  One CTA per
// (SCHUR_Y grid points in y = SCHUR_Y * q rows, column tile, problem): the rows of
// X its rows couple to (the y neighbours, SCHUR_Y + 2
// points) are staged once in shared memory, so every X row is read from
// memory about once instead of once per coupled row; a row's stencil
// coefficients are uniform across the CTA (broadcast loads).
// one thread per column of the tile: the block has CB threads
constexpr int SCHUR_Y = 8;
template <typename T> struct SchurCfg { static constexpr int CB = sizeof(T) == 4 ? 256 : 128; };
template <typename T>
__host__ __device__ constexpr size_t schur_smem(int q) {
  return (size_t)(SCHUR_Y + 2) * q * SchurCfg<T>::CB * sizeof(C_t<T>);
}

template <typename T>
__global__ void __launch_bounds__(SchurCfg<T>::CB)
schur_kernel(OpView op, const double2* __restrict__ shifts, int nh, int col0, int col1, int dx0,
             int add, const C_t<T>* __restrict__ Xprev, C_t<T>* __restrict__ M) {
  using C = C_t<T>;
  constexpr int CB = SchurCfg<T>::CB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* Xs = reinterpret_cast<C*>(smem_raw);  // [(SCHUR_Y + 2) * q][CB]
  const int b = op.b, q = op.q, ny = op.ny;
  const int nt = gridDim.x / nh, half = blockIdx.x / nt;
  const int f = blockIdx.z, pf = half * gridDim.z + f;
  const int i = half ? col1 : col0, dx = half ? -dx0 : dx0;
  const int y0 = (blockIdx.x - half * nt) * SCHUR_Y;
  const int c0 = blockIdx.y * CB;
  const C sh = mk((T)shifts[f].x, (T)shifts[f].y);
  const C* Xp = Xprev ? Xprev + (size_t)pf * b * b : nullptr;
  C* Mf = M + (size_t)pf * b * b;
  const int ny_blk = min(SCHUR_Y, ny - y0);
  // stage X rows of y points y0 - 1 .. y0 + ny_blk (slot k <-> point y0 - 1 + k)
  if (Xp) {
    const int nslots = (ny_blk + 2) * q;
    for (int e = threadIdx.x; e < nslots * CB; e += CB) {
      const int sl = e / CB, cc = e - sl * CB;
      const int pt = sl / q, comp = sl - pt * q;
      // point y0 - 1 + pt, wrapped when y is periodic (outside the grid
      // otherwise: never read, its coupling coefficient is absent)
      const int yy = op.periodic ? (y0 - 1 + pt + ny) % ny : y0 - 1 + pt;
      const int c = c0 + cc;
      C v = czero<C>();
      if (c < b && yy >= 0 && yy < ny) v = Xp[(size_t)(yy * q + comp) * b + c];
      Xs[sl * CB + cc] = v;
    }
    __syncthreads();
  }
  // The CTA's rows (ny_blk points x q variables) share their stencil
  // coefficients: stage them once, with the neighbour point of every y
  // offset (-1: a Dirichlet ghost), so the per-entry loop reads shared
  // memory only.
  __shared__ T cA[SCHUR_Y * 4][12];  // coupling to column i + dx, term (dy, cp)
  __shared__ T cD[SCHUR_Y * 4][12];  // diagonal block D_i (slot dx = 0)
  __shared__ int jyt[SCHUR_Y][3];    // neighbour y of point y0 + ly at dy = -1, 0, 1
  const int nt3 = 3 * q;
  for (int e = threadIdx.x; e < ny_blk * q * nt3; e += blockDim.x) {
    const int lr = e / nt3, t = e - lr * nt3;
    const int ly = lr / q, comp = lr - ly * q;
    const int iy = y0 + ly, dy = t / q - 1, cp = t - (t / q) * q;
    const int jy = nbr_y(iy, dy, ny, op.periodic);
    const size_t cf = ((size_t)i * b + iy * q + comp) * op.S;
    cA[lr][t] = (jy >= 0 && Xp) ? coefv<T>(op, cf + slotx(dx, dy) * q + cp) : (T)0;
    cD[lr][t] = jy >= 0 ? coefv<T>(op, cf + slotx(0, dy) * q + cp) : (T)0;
  }
  for (int e = threadIdx.x; e < ny_blk * 3; e += blockDim.x)
    jyt[e / 3][e % 3] = nbr_y(y0 + e / 3, e % 3 - 1, ny, op.periodic);
  __syncthreads();
  const int c = c0 + threadIdx.x;
  if (c >= b) return;
  const int jc = c / q, cc = c - jc * q;  // column c = variable cc of point jc
  for (int ly = 0; ly < ny_blk; ++ly) {
    const int iy = y0 + ly;
    for (int comp = 0; comp < q; ++comp) {
      const int r = iy * q + comp, lr = ly * q + comp;
      C val = add ? Mf[(size_t)r * b + c] : (r == c) ? sh : czero<C>();
      // D_i: the row's entries at column c (one per y offset landing on jc)
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
        if (!add && jyt[ly][dy] == jc) val.x -= cD[lr][dy * q + cc];
      if (Xp) {
#pragma unroll
        for (int t = 0; t < 12; ++t) {  // 3 y neighbours x q <= 4 variables
          if (t >= nt3) break;
          const T av = cA[lr][t];
          // slot of point iy + dy: ly + 1 + dy (periodic wrap stays in the
          // staged range because the staged points are y0 - 1 .. y0 + ny_blk)
          const int dy = t / q - 1, cp = t - (t / q) * q;
          if (av != (T)0) val = crfma(av, Xs[((ly + 1 + dy) * q + cp) * CB + threadIdx.x], val);
        }
      }
      Mf[(size_t)r * b + c] = val;
    }
  }
}

// ------------------------------------------------------------------- panel
constexpr int GP_NB = 16;       // panel width
constexpr int GP_LPR = 4;       // lanes of a row
constexpr int GP_CPL = GP_NB / GP_LPR;
constexpr int GP_MAXW = 16;     // warps of a CTA: 8 rows each
constexpr int GP_CLMAX = 8;

// 16-byte pieces of a candidate row and of 1 / pivot
template <typename T> __host__ __device__ constexpr int gp_pieces() { return GP_NB * (int)sizeof(C_t<T>) / 16; }
// a candidate slot: the row, then 1 / pivot in one 16-byte piece
template <typename T> __host__ __device__ constexpr int gp_slot() { return (gp_pieces<T>() + 1) * 16; }

// pivot magnitude as an integer that orders like it (without its lowest five
// bits): |x|^2 in FP32, the larger of |re| and |im| in FP64, whose high words
// need no FP64 arithmetic (its rate is a sixty-fourth of the integer rate)
__device__ __forceinline__ unsigned gp_mag(float2 x) {
  return __float_as_uint(x.x * x.x + x.y * x.y) & ~31u;
}
__device__ __forceinline__ unsigned gp_mag(double2 x) {
  return max((unsigned)__double2hiint(x.x) & 0x7fffffffu, (unsigned)__double2hiint(x.y) & 0x7fffffffu) &
         ~31u;
}
// magnitudes below which a pivot counts as zero, because its square vanishes (2^-538;
// FP32: a square of 2^-144), and below which 1 / square may overflow (2^-511; 2^-126)
template <typename T> __device__ __forceinline__ constexpr unsigned gp_zero() {
  return sizeof(T) == 8 ? 0x1e500000u : 32u;
}
template <typename T> __device__ __forceinline__ constexpr unsigned gp_small() {
  return sizeof(T) == 8 ? 0x20000000u : 0x00800000u;
}
// a magnitude above this is not a number
template <typename T> __device__ __forceinline__ constexpr unsigned gp_inf() {
  return sizeof(T) == 8 ? 0x7ff00000u : 0x7f800000u;
}
__device__ __forceinline__ float2 gp_shfl(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ double2 gp_shfl(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

struct PanelArgs {
  int b, k0, nbk, kp0, rpc, CL, F;
  int* rowpiv;    // [F][b]
  int* pivslot;   // [F][b]
  int* flag;      // [F] singular flags
  int* err;       // wait timeout
  uint32_t tries;
};

template <typename T>
constexpr size_t panel_smem(int rpc, int CL) {
  return (size_t)2 * CL * gp_slot<T>() + (size_t)2 * GP_MAXW * gp_slot<T>() +
         (size_t)rpc * (GP_NB + 1) * sizeof(C_t<T>) + (size_t)GP_NB * GP_NB * sizeof(C_t<T>);
}

// Eliminates the columns K = [k0, k0 + nbk) of every row of M; CTA rank r of the
// problem's cluster holds the rows r, r + CL, ... with four columns of K per
// lane.  When kp0 >= 0 the panel [kp0, kp0 + 16) was factored last and its
// transformation has reached every column but its own and K; it is applied to K
// first, x += M[r, Kp] B (x = M[r, Kp] B in its pivot rows).  Per step: the CTA's
// best eligible row (warp reductions and a barrier), whose warp forms 1 / pivot;
// it goes to every CTA of the cluster (st.async, see gjw_slab_kernel for the
// buffers' reuse); each warp picks the best of the CL candidates and eliminates.
// Outputs: the columns K of M, rowpiv of the rows pivoted here, pivslot.
// Bound (FP64): 20 FP64 instructions per warp and step at 64 cycles of its
// quarter of the SM, and the step's chain.  192 rows, four problems: 1.5 us a
// step; one CTA per problem took 243 us a panel.
template <typename T>
__global__ void __launch_bounds__(GP_MAXW * 32) gjp_panel_kernel(PanelArgs g, C_t<T>* __restrict__ Mall) {
  using C = C_t<T>;
  constexpr int NB = GP_NB, LPR = GP_LPR, CPL = GP_CPL, NP = gp_pieces<T>(), SLOT = gp_slot<T>();
  constexpr int CS = sizeof(C), PPL = CPL * CS / 16;  // pieces of a lane
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t mbar[2];
  __shared__ unsigned wkey[2][32];
  const int CL = g.CL, b = g.b, nbk = g.nbk;
  unsigned char* cand = smem_raw;                       // [2][CL][SLOT], slot CL - 1 - rank
  unsigned char* wst = cand + (size_t)2 * CL * SLOT;    // [2][GP_MAXW][SLOT], slot 15 - warp
  C* As = reinterpret_cast<C*>(wst + (size_t)2 * GP_MAXW * SLOT);  // [rpc][NB + 1]
  C* Bp = As + (size_t)g.rpc * (NB + 1);                // [NB][NB]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
  const int rank = (int)tc::cluster_rank();
  const int f = blockIdx.x / CL;  // problem of a half
  const int nrows = max(0, (b - rank + CL - 1) / CL);
  C* M = Mall + (size_t)f * b * b;
  int* rowpiv = g.rowpiv + (size_t)f * b;
  const int* pivslot = g.pivslot + (size_t)f * b;
  const int prow = tid / LPR, cg = (tid % LPR) * CPL;
  const bool live = prow < nrows;
  const int grow = prow * CL + rank;

  if (tid < 2) tc::mbar_init(&mbar[tid], 1);
  for (int e = tid; e < 64; e += nthr) wkey[e >> 5][e & 31] = 0u;  // (a CTA may be one warp)
  const int rp = live && g.k0 > 0 ? rowpiv[grow] : -1;
  const bool prevpiv = g.kp0 >= 0 && rp >= g.kp0 && rp < g.kp0 + NB;
  C x[CPL];
#pragma unroll
  for (int c = 0; c < CPL; ++c)
    x[c] = live && !prevpiv && cg + c < nbk ? M[(size_t)grow * b + g.k0 + cg + c] : czero<C>();
  if (g.kp0 >= 0) {
    for (int e = tid; e < nrows * NB; e += nthr) {
      const int r = e / NB, j = e - r * NB;
      As[r * (NB + 1) + j] = M[(size_t)(r * CL + rank) * b + g.kp0 + j];
    }
    for (int e = tid; e < NB * NB; e += nthr) {
      const int j = e / NB, c = e - j * NB;
      Bp[e] = c < nbk ? M[(size_t)pivslot[g.kp0 + j] * b + g.k0 + c] : czero<C>();
    }
  }
  // barriers initialised, and every CTA's reads of M done before any CTA writes
  tc::cluster_sync();
  if (g.kp0 >= 0 && live) {
    C u[CPL];  // summed on its own: one rounding against x (gjp_update_kernel)
#pragma unroll
    for (int c = 0; c < CPL; ++c) u[c] = czero<C>();
#pragma unroll 4
    for (int j = 0; j < NB; ++j) {
      const C a = As[prow * (NB + 1) + j];
#pragma unroll
      for (int c = 0; c < CPL; ++c) u[c] = cfma(a, Bp[j * NB + cg + c], u[c]);
    }
#pragma unroll
    for (int c = 0; c < CPL; ++c) x[c] = cadd(x[c], u[c]);
  }
  bool elig = live && rp < 0;
  int mypiv = -1;
  bool singular = false, ok = true;

  // the CTA's candidate: warp w sends its pieces to the CTAs w, w + W, ...
  const int myslot = CL - 1 - rank;
  const uint32_t cand_a = tc::smem_u32(cand) + (uint32_t)myslot * SLOT;
  const uint32_t mbar_a = tc::smem_u32(&mbar[0]);
  const uint32_t cbytes = (uint32_t)CL * SLOT;
  const unsigned row_id = 31u - (unsigned)(lane / LPR);
  unsigned char* my_wst = wst + (size_t)(GP_MAXW - 1 - warp) * SLOT + cg * CS;
#pragma unroll 1
  for (int jb = 0; jb < LPR; ++jb) {
    const int src_lane = (lane & ~(LPR - 1)) | jb;
    const bool mycol = cg == jb * CPL;
#pragma unroll
    for (int s = 0; s < CPL; ++s) {
      const int j = jb * CPL + s, buf = s & 1;
      if (j >= nbk) break;
      const C xs = gp_shfl(x[s], src_lane);
      const unsigned kmax = __reduce_max_sync(0xffffffffu, (elig ? gp_mag(xs) : 0u) | row_id);
      const bool wrow = ((kmax ^ row_id) & 31u) == 0u;  // the warp's best row
      if (wrow) {
        if (cg == 0) wkey[buf][warp] = kmax;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
          // (a warp without an eligible row: zero in the pivot's place)
          const C v = c == s && mycol && kmax < 32u ? czero<C>() : x[c];
          *reinterpret_cast<C*>(my_wst + (size_t)buf * GP_MAXW * SLOT + c * CS) = v;
        }
      }
      __syncthreads();
      const unsigned wk = (wkey[buf][lane] & ~31u) | ((15u - lane) & 31u);
      const unsigned cw = __reduce_max_sync(0xffffffffu, wk) & 15u;  // 15 - warp
      const unsigned char* src = wst + ((size_t)buf * GP_MAXW + cw) * SLOT;
      if (cw + warp == 15u) {  // 1 / pivot, by the warp that holds the candidate
        C pv = *reinterpret_cast<const C*>(src + j * CS);
        if (gp_mag(pv) < gp_zero<T>()) pv = mk(sizeof(T) == 8 ? (T)1e-150 : (T)1e-18, (T)0);
        const T pd = pv.x * pv.x + pv.y * pv.y;
        alignas(16) C pi[16 / CS] = {};
        if (gp_mag(pv) < gp_small<T>()) {
          pi[0] = mk(pv.x / pd, -pv.y / pd);
        } else {
          const T rd = (T)1 / pd;
          pi[0] = mk(pv.x * rd, -pv.y * rd);
        }
        const float4 val = *reinterpret_cast<const float4*>(pi);
        if (lane < CL)
          tc::st_async16(tc::cluster_map(cand_a + (uint32_t)(buf * CL * SLOT + NP * 16), lane), val,
                         tc::cluster_map(mbar_a + buf * 8, lane));
      }
      {
        const int W = nthr >> 5, per = 32 / NP;  // receivers of one warp instruction
        const float4 val = *reinterpret_cast<const float4*>(src + (lane % NP) * 16);
        for (int d0 = warp * per; d0 < CL; d0 += W * per) {
          const int d = d0 + lane / NP;
          if (d < CL)
            tc::st_async16(tc::cluster_map(cand_a + (uint32_t)(buf * CL * SLOT + (lane % NP) * 16), d),
                           val, tc::cluster_map(mbar_a + buf * 8, d));
        }
      }
      if (tid == 0) tc::mbar_expect_tx(&mbar[buf], cbytes);
      if (ok) ok = tc::cluster_wait(&mbar[buf], (s >> 1) & 1, g.tries);
      const unsigned char* cb = cand + (size_t)buf * CL * SLOT;
      const int sl = min(lane, CL - 1);
      const unsigned cmax = __reduce_max_sync(
          0xffffffffu, gp_mag(*reinterpret_cast<const C*>(cb + (size_t)sl * SLOT + j * CS)) | sl);
      singular |= cmax < gp_zero<T>() || (cmax & ~31u) > gp_inf<T>();
      const int pc = (int)(cmax & 31u);
      src = cb + (size_t)pc * SLOT;
      const C pinv = *reinterpret_cast<const C*>(src + NP * 16);
      C q[CPL];
#pragma unroll
      for (int u = 0; u < PPL; ++u)
        reinterpret_cast<float4*>(q)[u] = *reinterpret_cast<const float4*>(src + cg * CS + u * 16);
      C m = cneg(cmul(xs, pinv));
      if (pc == myslot && cw + warp == 15u) {  // (the whole warp)
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
          x[c].x = wrow ? (T)0 : x[c].x;
          x[c].y = wrow ? (T)0 : x[c].y;
        }
        m.x = wrow ? pinv.x : m.x;
        m.y = wrow ? pinv.y : m.y;
        elig = elig && !wrow;
        mypiv = wrow ? j : mypiv;
      }
#pragma unroll
      for (int c = 0; c < CPL; ++c) x[c] = cfma(m, q[c], x[c]);
      if (mycol) x[s] = m;
    }
  }
  if (live) {
#pragma unroll
    for (int c = 0; c < CPL; ++c)
      if (cg + c < nbk) M[(size_t)grow * b + g.k0 + cg + c] = x[c];
    if (cg == 0) {
      if (mypiv >= 0) {
        rowpiv[grow] = g.k0 + mypiv;
        g.pivslot[(size_t)f * b + g.k0 + mypiv] = grow;
      } else if (g.k0 == 0) {
        rowpiv[grow] = -1;
      }
    }
  }
  if (rank == 0 && tid == 0 && singular) g.flag[f % g.F] = 1;
  if (!ok && lane == 0) atomicExch(g.err, 1);
  if (!ok) tc::cluster_settle();
  tc::cluster_sync();  // no CTA leaves while another may still send to it
}

// B[f][j][m] = M[P_j][m] for the panel [k0, k0 + nbk), zero beyond nbk
template <typename T>
__global__ void gjp_gather_kernel(int b, int k0, int nbk, int nh, const C_t<T>* __restrict__ Mall,
                                  const int* __restrict__ pivslot_all, C_t<T>* __restrict__ Ball) {
  const int nt = gridDim.x / nh, half = blockIdx.x / nt;
  const int f = half * gridDim.z + blockIdx.z, j = blockIdx.y;
  const int m = (blockIdx.x - half * nt) * blockDim.x + threadIdx.x;
  if (m >= b) return;
  C_t<T> v = czero<C_t<T>>();
  if (j < nbk) v = Mall[((size_t)f * b + pivslot_all[(size_t)f * b + k0 + j]) * b + m];
  Ball[((size_t)f * GP_NB + j) * b + m] = v;
}

// (Summing onto the matrix entries instead rounds them sixteen times a panel: the
// unrefined residual of a 384-row FP64 adjoint solve was 6.3e-14 instead of 3.0e-14,
// of a 768-row FP32 one 8.6e-5 instead of 2.3e-5.  The sums go to the entries by
// reductions in L2, without registers, latency or FP64 operations for the old values.
// FP32, 960 rows, eight problems, 16 columns: 43.0 ms a factorisation; 55.9 with them
// requested ahead, 73 with them read at the end.  FP64, 192 rows, 64 problems: 64.2, and
// 65.8 with either.)
// The rank-16 update on TR x TR tiles (16 x 16 threads) of the columns outside
// [k0, k0 + nbk) and [n0, n1).  FP64 is bound by its pipe, so small tiles fill
// the SMs; FP32 by shared memory, so a thread holds 4 x 4 outputs.
__device__ __forceinline__ void red_add(float2* p, float2 v) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};\n" ::"l"(p), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void red_add(double2* p, double2 v) {
  asm volatile("red.global.add.f64 [%0], %1;\n" ::"l"(&p->x), "d"(v.x) : "memory");
  asm volatile("red.global.add.f64 [%0], %1;\n" ::"l"(&p->y), "d"(v.y) : "memory");
}
template <typename T> struct UpdCfg { static constexpr int TR = sizeof(T) == 8 ? 32 : 64; };
template <typename T>
__global__ void __launch_bounds__(256)
gjp_update_kernel(int b, int k0, int nbk, int n0, int n1, int nh, C_t<T>* __restrict__ Mall,
                  const C_t<T>* __restrict__ Ball, const int* __restrict__ rowpiv_all) {
  using C = C_t<T>;
  constexpr int NB = GP_NB, TR = UpdCfg<T>::TR, PT = TR / 16;
  __shared__ C As[TR][NB + 1];
  __shared__ C Bs[NB][TR];
  const int nt = gridDim.x / nh, half = blockIdx.x / nt;
  const int f = half * gridDim.z + blockIdx.z;
  C* M = Mall + (size_t)f * b * b;
  const C* B = Ball + (size_t)f * NB * b;
  const int* rowpiv = rowpiv_all + (size_t)f * b;
  const int r0 = blockIdx.y * TR, c0 = (blockIdx.x - half * nt) * TR;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  auto col_live = [&](int c) {
    return c < b && !(c >= k0 && c < k0 + nbk) && !(c >= n0 && c < n1);
  };
  C acc[PT][PT];
#pragma unroll
  for (int a = 0; a < PT; ++a)
#pragma unroll
    for (int d = 0; d < PT; ++d) acc[a][d] = czero<C>();
  for (int e = tid; e < TR * NB; e += 256) {
    const int rr = e / NB, m = e - rr * NB, r = r0 + rr;
    As[rr][m] = (r < b && m < nbk) ? M[(size_t)r * b + k0 + m] : czero<C>();
  }
  for (int e = tid; e < NB * TR; e += 256) {
    const int m = e / TR, cc = e - m * TR, c = c0 + cc;
    Bs[m][cc] = c < b ? B[(size_t)m * b + c] : czero<C>();
  }
  __syncthreads();
#pragma unroll 4
  for (int m = 0; m < NB; ++m) {
    C av[PT], bv[PT];
#pragma unroll
    for (int a = 0; a < PT; ++a) av[a] = As[ty + 16 * a][m];
#pragma unroll
    for (int d = 0; d < PT; ++d) bv[d] = Bs[m][tx + 16 * d];
#pragma unroll
    for (int a = 0; a < PT; ++a)
#pragma unroll
      for (int d = 0; d < PT; ++d) acc[a][d] = cfma(av[a], bv[d], acc[a][d]);
  }
  // (an entry has one writer a launch: the order of the sums is fixed)
#pragma unroll
  for (int a = 0; a < PT; ++a) {
    const int r = r0 + ty + 16 * a, rp = r < b ? rowpiv[r] : -1;
    if (r >= b) continue;
    const bool keep = !(rp >= k0 && rp < k0 + nbk);
#pragma unroll
    for (int d = 0; d < PT; ++d) {
      const int c = c0 + tx + 16 * d;
      if (!col_live(c)) continue;
      C* p = &M[(size_t)r * b + c];
      if (keep) red_add(p, acc[a][d]);
      else *p = acc[a][d];
    }
  }
}

// G_i[j][p_m] = M[p_j][m];  X_i = G_i C_i with C_i = -L_{i,i+1} (half 0) or
// G_i A_i with A_i = -L_{i,i-1} (half 1).
template <typename T>
__global__ void gjp_finalize_kernel(OpView op, int ldg, int nh, int col0, int col1, int RB,
                                    const C_t<T>* __restrict__ Mall,
                                    const int* __restrict__ pivslot_all, C_t<T>* __restrict__ Gall,
                                    C_t<T>* __restrict__ Xall) {
  using C = C_t<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int b = op.b, q = op.q;
  C* Gs = reinterpret_cast<C*>(smem_raw);                 // [RB][b]
  int* ps = reinterpret_cast<int*>(Gs + (size_t)RB * b);  // [b]
  const int nt = gridDim.x / nh, half = blockIdx.x / nt;
  const int f = blockIdx.y, pf = half * gridDim.y + f, i = half ? col1 : col0;
  const int r0 = (blockIdx.x - half * nt) * RB;
  const C* M = Mall + (size_t)pf * b * b;
  for (int c = threadIdx.x; c < b; c += blockDim.x) ps[c] = pivslot_all[(size_t)pf * b + c];
  __syncthreads();
  for (int e = threadIdx.x; e < RB * b; e += blockDim.x) {
    const int rr = e / b, c = e - rr * b, r = r0 + rr;
    if (r < b) Gs[rr * b + ps[c]] = M[(size_t)ps[r] * b + c];
  }
  __syncthreads();
  C* G = Gall + ((size_t)f * op.nx + i) * b * ldg;
  for (int e = threadIdx.x; e < RB * b; e += blockDim.x) {
    const int rr = e / b, c = e - rr * b, r = r0 + rr;
    if (r < b) G[(size_t)r * ldg + c] = Gs[rr * b + c];
  }
  if (Xall == nullptr) return;
  C* X = Xall + (size_t)pf * b * b;
  const int dx = half ? -1 : 1;
  for (int e = threadIdx.x; e < RB * b; e += blockDim.x) {
    const int rr = e / b, c = e - rr * b, r = r0 + rr;
    if (r >= b) continue;
    const int iyc = c / q, cc = c - iyc * q;
    C s = czero<C>();
    for (int dy = -1; dy <= 1; ++dy) {
      const int iym = nbr_y(iyc, -dy, op.ny, op.periodic);
      if (iym < 0) continue;
      for (int cm = 0; cm < q; ++cm) {
        const int m = iym * q + cm;
        const T a = coefv<T>(op, ((size_t)i * b + m) * op.S + slotx(dx, dy) * q + cc);
        if (a != (T)0) s = crfma(a, Gs[rr * b + m], s);
      }
    }
    X[(size_t)r * b + c] = cneg(s);
  }
}

template <typename T>
rr_status launch_schur(const OpView& ov, const double2* shifts, int F, int nh, int col0, int col1,
                  int dx0, int add, const C_t<T>* Xprev, C_t<T>* M, cudaStream_t st) {
  constexpr int CB = SchurCfg<T>::CB;
  const size_t smem = Xprev ? schur_smem<T>(ov.q) : 0;
  RR_TRY(smem_opt_in<schur_kernel<T>>(schur_smem<T>(4)));
  dim3 gs((ov.ny + SCHUR_Y - 1) / SCHUR_Y * nh, (ov.b + CB - 1) / CB, F);
  schur_kernel<T><<<gs, CB, smem, st>>>(ov, shifts, nh, col0, col1, dx0, add, Xprev, M);
  return RR_OK;
}

// M = S_i for step t of the factorisation (twist_steps)
template <typename T>
rr_status schur_step(rr_factors* fa, const TwistStep& t, cudaStream_t st) {
  const OpDev& d = fa->op->d;
  const OpView ov = view(d);
  using C = C_t<T>;
  C* M = reinterpret_cast<C*>(fa->M);
  const C* X = reinterpret_cast<const C*>(fa->X);
  prof_begin(PROF_SCHUR, st);
  RR_TRY(launch_schur<T>(ov, fa->shifts, fa->F, t.nh, t.col0, t.col1, -1, 0,
                         t.first ? nullptr : X, M, st));
  prof_end(PROF_SCHUR, st);
  if (t.middle) {
    prof_begin(PROF_SCHUR, st);
    RR_TRY(launch_schur<T>(ov, fa->shifts, fa->F, 1, t.col0, t.col1, 1, 1,
                           X + (size_t)fa->F * d.b * d.b, M, st));
    prof_end(PROF_SCHUR, st);
  }
  RR_CUDA(cudaGetLastError());
  return RR_OK;
}

template <typename T>
rr_status launch_panel(rr_factors* fa, int nh, int k0, int nbk, int kp0, cudaStream_t st) {
  const OpDev& d = fa->op->d;
  PanelArgs a;
  a.b = d.b;
  a.k0 = k0;
  a.nbk = nbk;
  a.kp0 = kp0;
  a.F = fa->F;
  a.CL = std::min(GP_CLMAX, (d.b + 7) / 8);  // at least eight rows per CTA
  a.rpc = (d.b + a.CL - 1) / a.CL;
  a.rowpiv = fa->rowpiv;
  a.pivslot = fa->pivslot;
  a.flag = fa->flag;
  a.err = fa->err;
  a.tries = wait_tries();
  const size_t smem = panel_smem<T>(a.rpc, a.CL);
  RR_TRY(smem_opt_in<gjp_panel_kernel<T>>(panel_smem<T>(GP_MAXW * 8, GP_CLMAX)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.CL * fa->F * nh), 1, 1);
  cfg.blockDim = dim3((unsigned)((a.rpc * GP_LPR + 31) / 32 * 32), 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = a.CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  prof_begin(PROF_PANEL, st);
  RR_CUDA(cudaLaunchKernelEx(&cfg, gjp_panel_kernel<T>, a, reinterpret_cast<C_t<T>*>(fa->M)));
  prof_end(PROF_PANEL, st);
  return RR_OK;
}

template <typename T>
rr_status factor_impl(rr_factors* fa) {
  using C = C_t<T>;
  constexpr int NB = GP_NB;
  const OpDev& d = fa->op->d;
  const OpView ov = view(d);
  const int b = d.b, F = fa->F;
  cudaStream_t st = fa->stream, st2 = fa->stream2;
  C* M = reinterpret_cast<C*>(fa->M);
  C* G = reinterpret_cast<C*>(fa->G);
  C* X = reinterpret_cast<C*>(fa->X);
  C* Bbuf = reinterpret_cast<C*>(fa->Bbuf);
  constexpr int RB = 4;
  const size_t fsmem = (size_t)RB * b * sizeof(C) + b * sizeof(int);  // (b <= 1024)
  RR_TRY(smem_opt_in<gjp_finalize_kernel<T>>(RB * 1024 * sizeof(C) + 1024 * sizeof(int)));
  constexpr int TR = UpdCfg<T>::TR;
  const int nt = (b + TR - 1) / TR, P = (b + NB - 1) / NB;
  rr_status s;
  for (int step = 0; step < twist_steps(fa); ++step) {
    const TwistStep t = twist_step(fa, step);
    const int nh = t.nh;
    if ((s = schur_step<T>(fa, t, st)) != RR_OK) return s;
    // The panels run in order on the second (high-priority) stream, the updates
    // in order on the main one.  Panel p applies panel p - 1's transformation to
    // its own columns, so it waits only for the update of panel p - 2 and runs
    // beside that of p - 1 (disjoint columns; rowpiv entries written meanwhile
    // go from "none" to a column outside p - 1, which the update reads as "not
    // its pivot row" either way).
    RR_CUDA(cudaEventRecord(fa->ev_next, st));
    RR_CUDA(cudaStreamWaitEvent(st2, fa->ev_next, 0));
    for (int p = 0; p < P; ++p) {
      const int k0 = p * NB, nbk = std::min(NB, b - k0);
      if (p >= 2) RR_CUDA(cudaStreamWaitEvent(st2, fa->ev_ring[4 + ((p - 2) & 3)], 0));
      if ((s = launch_panel<T>(fa, nh, k0, nbk, p > 0 ? k0 - NB : -1, st2)) != RR_OK) return s;
      RR_CUDA(cudaEventRecord(fa->ev_ring[p & 3], st2));
      RR_CUDA(cudaStreamWaitEvent(st, fa->ev_ring[p & 3], 0));
      if (P == 1) break;
      prof_begin(PROF_ROWBLOCK, st);
      gjp_gather_kernel<T><<<dim3((b + 127) / 128 * nh, NB, F), 128, 0, st>>>(b, k0, nbk, nh, M, fa->pivslot,
                                                                            Bbuf);
      prof_end(PROF_ROWBLOCK, st);
      const int n0 = p + 1 < P ? k0 + NB : 0, n1 = p + 1 < P ? std::min(b, n0 + NB) : 0;
      prof_begin(PROF_UPDATE, st);
      gjp_update_kernel<T><<<dim3(nt * nh, nt, F), 256, 0, st>>>(b, k0, nbk, n0, n1, nh, M, Bbuf,
                                                                 fa->rowpiv);
      prof_end(PROF_UPDATE, st);
      RR_CUDA(cudaEventRecord(fa->ev_ring[4 + (p & 3)], st));
      RR_CUDA(cudaGetLastError());
    }
    prof_begin(PROF_FINALIZE, st);
    gjp_finalize_kernel<T><<<dim3((b + RB - 1) / RB * nh, F), 256, fsmem, st>>>(
        ov, fa->ldg, nh, t.col0, t.col1, RB, M, fa->pivslot, G, t.middle ? nullptr : X);
    prof_end(PROF_FINALIZE, st);
    RR_CUDA(cudaGetLastError());
  }
  return RR_OK;
}

}  // namespace

// Steps of the factorisation: the pairs of columns from the ends inwards, then
// the middle one (factor_cols > 0 stops after that many: autotuner timing only)
int twist_steps(const rr_factors* fa) {
  const int n = twist_mid(fa->op->d.nx) + 1;
  return fa->factor_cols > 0 ? std::min(fa->factor_cols, n - 1) : n;
}

TwistStep twist_step(const rr_factors* fa, int t) {
  const int nx = fa->op->d.nx, m = twist_mid(nx);
  TwistStep s;
  s.first = t == 0;
  s.middle = t == m;
  s.nh = !s.middle && t < nx - 1 - m ? 2 : 1;
  s.col0 = t;
  s.col1 = nx - 1 - t;
  return s;
}

rr_status launch_schur_f32(rr_factors* fa, const TwistStep& t, cudaStream_t st) {
  return schur_step<float>(fa, t, st);
}

rr_status launch_factor(rr_factors* fa) {
  const OpDev& d = fa->op->d;
  const bool wide = fa->prec != RR_FP64 && factor_wide_ok(fa) && fa->tune_update != 1;
  if (fa->Fw < 1) {
    set_error("no memory for the factorisation's work buffers");
    return RR_ERR_NOMEM;
  }
  for (int f0 = 0; f0 < fa->F; f0 += fa->Fw) {
    rr_factors part = *fa;  // the problems of this pass (the work buffers are shared)
    part.F = std::min(fa->Fw, fa->F - f0);
    part.G = static_cast<char*>(fa->G) + (size_t)f0 * d.nx * d.b * fa->ldg * fa->csz;
    part.shifts = fa->shifts + f0;
    part.flag = fa->flag + f0;
    RR_TRY(fa->prec == RR_FP64 ? factor_impl<double>(&part)
           : wide              ? launch_factor_wide(&part)
                               : factor_impl<float>(&part));
  }
  return RR_OK;
}
