// Wide block factorisation of the Schur blocks for FP32 factors: the explicit
// inverse G_i = S_i^{-1} of Sec. III.A's one-factorisation-per-shift scheme
// (S_0 = D_0, X_i = G_i C_i, S_{i+1} = D_{i+1} - A_{i+1} X_i), formed by
// Gauss-Jordan elimination with partial pivoting in two levels so that the
// bulk of the work is a rank-128 complex update on the tensor cores.
//
// Pivoting is implicit: rows are never moved.  Column j is eliminated with
// the pivot row p_j (the largest |.|^2, to 18 bits, among rows not yet pivoted;
// ties: see gjw_slab_kernel) by the elementary transformation E_j (row p_j scaled by 1/m_pj,
// m_pj times it subtracted from every other row; column j then holds E_j's
// column p_j, the in-place inverse).  After all b columns the work matrix is
// M = Q^T S^{-1} Q^T with (Q x)_j = x_{p_j}, so S^{-1}[j, p_m] = M[p_j, m].
//
// Levels, for every slab of W = 128 columns [c0, c1):
//   inner: one cluster of CTAs per problem holds the slab on chip and runs
//     its panels K of 16 columns (gjw_slab_kernel): the 16 eliminations,
//     recording the pivot rows P, then the transformations of K applied to
//     the rest of the slab, M[r, m] += M[r, K] * M_old[P, m] for rows r not
//     in P and M[P, m] = M[P, K] * M_old[P, m] (the pivot rows take T^{-1} B
//     itself: adding (T^{-1} - I) B to B would cancel when T^{-1} is small),
//     in FP32 on the CUDA cores;
//   outer:
//     gather : B = M[P_slab, outside the slab] (the pivot rows, saved before
//              they change);
//     update : the composed transformation of the slab's 128 eliminations
//              applied at once, M[r, outside] += M[r, slab] * B (r not in
//              P_slab), M[P_slab, outside] = M[P_slab, slab] * B, as a complex
//              GEMM on tcgen05 with the operands split into TF32 or BF16
//              pieces (FP32-level products, FP32 accumulation in TMEM;
//              gjw_gemm_kernel).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "rr_internal.cuh"
#include "tc.cuh"

namespace {

constexpr int GW_W = 128;   // slab width (rank of the outer update)
constexpr int GW_NB = 16;   // panel width (rank of the slab update)
constexpr int GW_MAX = 768;  // largest block of the wide path

// -------------------------------------------------------------------- slab
// Factors one slab: eliminates the columns [c0, c1) (at most 128) of every row
// of M, the slab resident on chip for all of its steps.  A cluster of CL CTAs
// owns one problem; CTA rank r holds the rows r, r + CL, r + 2 CL, ... of the
// slab in shared memory (cyclic, so the pivot rows of a panel, which cluster
// around the diagonal, are spread over the CTAs that send them).  Per panel K
// of 16 columns:
//   steps  : the panel warps hold the panel in registers, LPR lanes per row.
//            Step j: the CTA's best eligible row of column j
//            (largest |.|^2 to 18 bits, lowest warp and lane among equals) by
//            warp reductions and a barrier of the panel warps, which send it,
//            128 bytes, to every CTA of the cluster (st.async into the
//            sender's candidate slot, completing on the receiver's mbarrier,
//            so data and signal travel together; a CTA without an eligible
//            row sends a zero pivot); every warp then reduces the CL
//            candidates itself (lowest CTA among equals) and eliminates:
//            x += m (pivot row), x_j = m with m = -x_j / pivot, and x = 0,
//            m = 1 / pivot in the pivot row;
//   B      : the CTAs that hold the panel's 16 pivot rows send them (the
//            slab's columns, before this panel's step) to every CTA, the other
//            warps' work as soon as a pivot is known;
//   update : M[r, m] += M[r, K] B[:, m] for the slab's other columns m,
//            M[r, m] = M[r, K] B[:, m] for the pivot rows (T^{-1} B itself), in
//            exact FP32 on the CUDA cores.  The panel warps take the next
//            panel's 16 columns as they load them; the rest is the other
//            warps' work while the panel warps run the next panel's steps.
// A problem that fits one CTA (SOLO) needs no exchange.
// Candidate slots are double-buffered by step parity: a CTA sends for step
// j + 2 only after it has received every CTA's candidate of step j + 1, each
// sent after a barrier that follows its panel warps' last reads of step j.  B
// is double-buffered by panel parity: a CTA sends for panel p + 2 only after
// every CTA took part in panel p + 2, which each begins after its update of
// panel p is complete.
//
// Bound: the chain of 128 dependent steps (reduce, send, receive, reduce,
// eliminate).  768 rows in clusters of eight CTAs: 108 us a slab of 128 columns,
// of which 58 in the local part of the steps, 22 in the exchange and the rest
// where the update competes for issue slots; one kernel per 16-column panel and
// one for its update of the slab took 8 x 39 us.  Sixteen warps keep the panel
// code out of local memory (96 registers and fewer spilled in the steps: 112
// to 150 us).
constexpr int SL_THREADS = 512, SL_WARPS = SL_THREADS / 32;
constexpr int SL_LD = GW_W + 2;  // row pitch: 16-byte reads down a column hit all banks
constexpr int SL_PWMAX = 12;     // most panel warps of a CTA (the others update)
constexpr int SL_WSLOTS = 16;    // slots of the panel warps' best rows
constexpr int SL_UR = 8;         // rows of an update tile
constexpr int SL_CLMAX = 8;      // largest cluster
constexpr int SL_CAND = GW_NB * 8;  // bytes of a candidate: one row of the panel
constexpr size_t SL_SMEM_CAP = 226 * 1024;  // dynamic shared memory of a CTA

struct SlabArgs {
  int b, c0, c1, rpc, CL;
  float2* M;                     // [2F][b][b]
  int* rowpiv;                   // [2F][b]
  int* pivslot;                  // [2F][b]
  int* flag;                     // [F] singular flags
  int* err;                      // wait timeout
  int F;
  uint32_t tries;
};

__host__ __device__ constexpr int slab_rows8(int rpc) { return (rpc + SL_UR - 1) / SL_UR * SL_UR; }
__host__ __device__ constexpr size_t slab_smem_bytes(int rpc, int CL) {
  return (size_t)slab_rows8(rpc) * (SL_LD * 8 + 8)                       // S, pivot steps
         + (size_t)(CL > 1 ? 2 : 1) * GW_NB * GW_W * 8                  // B
         + (size_t)2 * ((CL > 1 ? SL_CLMAX : 0) + SL_WSLOTS) * SL_CAND;  // candidates, staging
}

// 1 / v to FP32 accuracy without a call: the hardware approximation (1 ulp) and
// a Newton step where it cannot leave the normal range
__device__ __forceinline__ float recip(float v) {
  float r;
  asm("rcp.approx.f32 %0, %1;\n" : "=f"(r) : "f"(v));
  const float n = fmaf(r, fmaf(-v, r, 1.f), r);
  return v > 1e-37f && v < 1e37f ? n : r;
}
// 16-byte piece i of a candidate in slot c sits at piece i ^ (c % 8): the
// lanes of a warp that read one column of all slots spread over the banks
__device__ __forceinline__ int cand_piece(int i, int c) { return (i ^ (c & 7)) * 16; }
// key of a pivot candidate: orders like |x|^2 cut to 18 bits (the bits of a
// non-negative float order like the float), then the largest id < 32
__device__ __forceinline__ unsigned pivot_key(float a, unsigned id) {
  return (__float_as_uint(a) & ~31u) | id;
}

// The transformation of the panel at group kg (16 columns each) applied to
// the CTA's rows at the slab's other groups, except the group kg + 1 when
// skip_next, in tiles of 8 rows x 32 NS columns (slot t of a lane: column
// lane % 16 of the (2 (slot0 + t) + lane / 16)-th remaining group) taken by the warps
// w0, w0 + nw, ...; rowp[r] >= 0 marks the panel's pivot rows.
template <int NS>
__device__ __forceinline__ void slab_update_tiles(float2* S, const float2* Bs, const int* rowp,
                                                  int nrows, int ngrp, int kg, int nskip, int w0,
                                                  int nw, int lane, int slot0 = 0) {
  constexpr int NB = GW_NB;
  int col[NS];
  bool on[NS];
#pragma unroll
  for (int t = 0; t < NS; ++t) {
    const int gi = 2 * (t + slot0) + (lane >> 4), gr = gi < kg ? gi : gi + nskip;
    on[t] = gr < ngrp;
    col[t] = (on[t] ? gr : kg) * NB + (lane & 15);
  }
  for (int rg = w0 * SL_UR; rg < nrows; rg += nw * SL_UR) {
    float2 acc[SL_UR][NS];
#pragma unroll
    for (int i = 0; i < SL_UR; ++i) {
      const bool keep = rg + i < nrows && rowp[rg + i] < 0;
#pragma unroll
      for (int t = 0; t < NS; ++t)
        acc[i][t] = keep ? S[(rg + i) * SL_LD + col[t]] : make_float2(0.f, 0.f);
    }
#pragma unroll 1
    for (int j = 0; j < NB; j += 2) {
      float2 b0[NS], b1[NS];
#pragma unroll
      for (int t = 0; t < NS; ++t) {
        b0[t] = Bs[j * GW_W + col[t]];
        b1[t] = Bs[(j + 1) * GW_W + col[t]];
      }
#pragma unroll
      for (int i = 0; i < SL_UR; ++i) {
        const float4 a = *reinterpret_cast<const float4*>(&S[(rg + i) * SL_LD + kg * NB + j]);
#pragma unroll
        for (int t = 0; t < NS; ++t) acc[i][t] = cfma(make_float2(a.x, a.y), b0[t], acc[i][t]);
#pragma unroll
        for (int t = 0; t < NS; ++t) acc[i][t] = cfma(make_float2(a.z, a.w), b1[t], acc[i][t]);
      }
    }
#pragma unroll
    for (int i = 0; i < SL_UR; ++i) {
      if (rg + i >= nrows) break;
#pragma unroll
      for (int t = 0; t < NS; ++t)
        if (on[t]) S[(rg + i) * SL_LD + col[t]] = acc[i][t];
    }
  }
}

__device__ __forceinline__ void slab_update(float2* S, const float2* Bs, const int* rowp, int nrows,
                                            int ngrp, int kg, bool skip_next, int w0, int nw,
                                            int lane) {
  const int nskip = skip_next ? 2 : 1, left = ngrp - nskip;
  if (left <= 0) return;
  switch ((left + 1) >> 1) {
    case 1: slab_update_tiles<1>(S, Bs, rowp, nrows, ngrp, kg, nskip, w0, nw, lane); break;
    case 2: slab_update_tiles<2>(S, Bs, rowp, nrows, ngrp, kg, nskip, w0, nw, lane); break;
    case 3: slab_update_tiles<3>(S, Bs, rowp, nrows, ngrp, kg, nskip, w0, nw, lane); break;
    default:  // (four column slots at once exceed the registers of 24 warps)
      slab_update_tiles<2>(S, Bs, rowp, nrows, ngrp, kg, nskip, w0, nw, lane);
      slab_update_tiles<2>(S, Bs, rowp, nrows, ngrp, kg, nskip, w0, nw, lane, 2);
  }
}

template <bool SOLO, int LPR>
__global__ void __launch_bounds__(SL_THREADS, 1) gjw_slab_kernel(SlabArgs g) {
  constexpr int NB = GW_NB;
  constexpr int CPL = NB / LPR;  // panel columns per lane
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t mbar[2], mbarB;
  __shared__ unsigned wkey[2][32];  // the panel warps' keys of a step (0 beyond)
  // local row of the panel's pivots (-1: not known yet, -2: another CTA's)
  __shared__ int own_sm[2][NB];
  volatile int(*own)[NB] = own_sm;
  const int CL = SOLO ? 1 : g.CL;
  const int rpc8 = slab_rows8(g.rpc);
  const int pw = (g.rpc * LPR + 31) >> 5;  // panel warps
  float2* S = reinterpret_cast<float2*>(smem_raw);            // [rpc8][SL_LD]
  float2* Bs = S + (size_t)rpc8 * SL_LD;                      // [SOLO ? 1 : 2][NB][GW_W]
  unsigned char* cand = reinterpret_cast<unsigned char*>(Bs + (SOLO ? 1 : 2) * NB * GW_W);
  // candidate slots [2][SL_CLMAX] (slot 7 - rank) and the panel warps' best
  // rows [2][SL_WSLOTS] (slot 15 - warp)
  unsigned char* wst = cand + (SOLO ? 0 : 2 * SL_CLMAX * SL_CAND);
  int* rowp = reinterpret_cast<int*>(wst + 2 * SL_WSLOTS * SL_CAND);  // [2][rpc8]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = g.b, c0 = g.c0, ncol = g.c1 - g.c0;
  const uint32_t rank = SOLO ? 0u : tc::cluster_rank();
  const int f = blockIdx.x / CL;
  const int nrows = max(0, (b - (int)rank + CL - 1) / CL);
  float2* M = g.M + (size_t)f * b * b;
  int* rowpiv = g.rowpiv + (size_t)f * b;
  const int npan = (ncol + NB - 1) / NB;

  if (!SOLO && tid == 0) {
    tc::mbar_init(&mbar[0], 1);
    tc::mbar_init(&mbar[1], 1);
    tc::mbar_init(&mbarB, 1);
  }
  if (tid < 2 * NB) own[tid / NB][tid % NB] = -1;
  if (tid < 64) wkey[tid >> 5][tid & 31] = 0u;
  if (!SOLO)  // the slots of absent CTAs stay zero
    for (int e = tid; e < 2 * SL_CLMAX * SL_CAND / 4; e += SL_THREADS)
      reinterpret_cast<int*>(cand)[e] = 0;
  // the slab's rows (zero beyond its columns and rows)
  for (int e = tid; e < rpc8 * (GW_W / 2); e += SL_THREADS) {
    const int r = e / (GW_W / 2), u = e - r * (GW_W / 2);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < nrows && 2 * u < ncol)
      v = reinterpret_cast<const float4*>(M + (size_t)(r * CL + rank) * b + c0)[u];
    *reinterpret_cast<float4*>(&S[r * SL_LD + 2 * u]) = v;
  }
  // a panel lane: row prow, columns [cg, cg + CPL) of the panel
  const bool is_panel = warp < pw;
  const int prow = tid / LPR, cg = (tid % LPR) * CPL;
  const bool live = is_panel && prow < nrows;
  const int grow = prow * CL + (int)rank;
  bool elig = live && (c0 == 0 || rowpiv[grow] < 0);
  int mypiv = -1;        // column this row pivoted for in this slab
  int myj = -1;          // its step if it pivoted in the panel at hand
  bool singular = false;
  if (SOLO) __syncthreads();
  else tc::cluster_sync();  // barriers initialised before any CTA sends; S complete

  // sending the CTA's candidate: panel warp w takes the 16-byte piece lane % 8
  // for CTA 4 w + lane / 8 (and, with one panel warp, 4 + lane / 8)
  const int myslot = SL_CLMAX - 1 - (int)rank;
  const uint32_t cand_a = tc::smem_u32(cand) + myslot * SL_CAND + cand_piece(lane & 7, myslot);
  const uint32_t mbar_a = tc::smem_u32(&mbar[0]);
  const int rk1 = 4 * warp + (lane >> 3), rk2 = pw == 1 ? rk1 + 4 : CL;
  uint32_t ra1 = 0, ra2 = 0, rm1 = 0, rm2 = 0;
  if (!SOLO) {
    ra1 = tc::cluster_map(cand_a, min(rk1, CL - 1));
    ra2 = tc::cluster_map(cand_a, min(rk2, CL - 1));
    rm1 = tc::cluster_map(mbar_a, min(rk1, CL - 1));
    rm2 = tc::cluster_map(mbar_a, min(rk2, CL - 1));
  }
  const uint32_t cbytes = (uint32_t)(CL * SL_CAND);
  constexpr uint32_t CB = SL_CLMAX * SL_CAND, WB = SL_WSLOTS * SL_CAND;  // one buffer of each
  const unsigned row_id = 31u - (unsigned)(lane / LPR);
  unsigned char* my_wst = wst + (is_panel ? SL_WSLOTS - 1 - warp : 0) * SL_CAND + cg * 8;
  bool ok = true;
  for (int p = 0; p < npan; ++p) {
    const int kl = p * NB, nbk = min(NB, ncol - kl);
    int* rowp_p = rowp + (p & 1) * rpc8;
    float2* Bp = Bs + (SOLO ? 0 : (p & 1) * NB * GW_W);
    const float2* Bq = Bs + (SOLO ? 0 : ((p + 1) & 1) * NB * GW_W);  // the previous panel's
    if (is_panel) {
      if (tid < NB) own[(p + 1) & 1][tid] = -1;
      if (!SOLO && tid == 0 && npan > 1) tc::mbar_expect_tx(&mbarB, (uint32_t)nbk * (GW_W * 8));
      // the panel's columns, with the previous panel's transformation
      float2 x[CPL];
#pragma unroll
      for (int c = 0; c < CPL; c += 2) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (live && myj < 0) v = *reinterpret_cast<const float4*>(&S[prow * SL_LD + kl + cg + c]);
        x[c] = make_float2(v.x, v.y);
        x[c + 1] = make_float2(v.z, v.w);
      }
      if (p > 0 && live) {
        const float2* Ar = &S[prow * SL_LD + kl - NB];
#pragma unroll 2
        for (int j = 0; j < NB; j += 2) {
          const float4 a = *reinterpret_cast<const float4*>(Ar + j);
          const float2 a0 = make_float2(a.x, a.y), a1 = make_float2(a.z, a.w);
          const float2* B0 = Bq + j * GW_W + kl + cg;
#pragma unroll
          for (int c = 0; c < CPL; c += 2) {
            const float4 v0 = *reinterpret_cast<const float4*>(B0 + c);
            const float4 v1 = *reinterpret_cast<const float4*>(B0 + GW_W + c);
            x[c] = cfma(a0, make_float2(v0.x, v0.y), x[c]);
            x[c + 1] = cfma(a0, make_float2(v0.z, v0.w), x[c + 1]);
            x[c] = cfma(a1, make_float2(v1.x, v1.y), x[c]);
            x[c + 1] = cfma(a1, make_float2(v1.z, v1.w), x[c + 1]);
          }
        }
      }
      myj = -1;
      // column jb CPL + s is register s of lane jb of every row; b % 8 == 0,
      // so a panel has a multiple of CPL steps and the parities of a step are
      // those of s
#pragma unroll 1
      for (int jb = 0; jb * CPL < nbk; ++jb) {
        const int src_lane = (lane & ~(LPR - 1)) | jb;
        const bool mycol = cg == jb * CPL;
#pragma unroll
        for (int s = 0; s < CPL; ++s) {
          const int j = jb * CPL + s, buf = s & 1;
          const float2 xs = make_float2(__shfl_sync(0xffffffffu, x[s].x, src_lane),
                                        __shfl_sync(0xffffffffu, x[s].y, src_lane));
          const float av = elig ? xs.x * xs.x + xs.y * xs.y : 0.f;
          const unsigned kmax = __reduce_max_sync(0xffffffffu, pivot_key(av, row_id));
          const bool wrow = ((kmax ^ row_id) & 31u) == 0u;  // the warp's best row
          {
            // (a warp without an eligible row: zero in the pivot's place)
            const bool none = kmax < 32u && mycol;
            if (wrow && cg == 0) wkey[buf][warp] = kmax;
#pragma unroll
            for (int c = 0; c < CPL; c += 2) {
              float4 v = make_float4(x[c].x, x[c].y, x[c + 1].x, x[c + 1].y);
              if (c == s) v.x = none ? 0.f : v.x, v.y = none ? 0.f : v.y;
              if (c + 1 == s) v.z = none ? 0.f : v.z, v.w = none ? 0.f : v.w;
              if (wrow) *reinterpret_cast<float4*>(my_wst + buf * WB + c * 8) = v;
            }
          }
          // the CTA's candidate: the best of its panel warps
          asm volatile("bar.sync 1, %0;\n" ::"r"(pw * 32) : "memory");
          const unsigned wk = pivot_key(__uint_as_float(wkey[buf][lane]), (15u - lane) & 31u);
          const unsigned cw = __reduce_max_sync(0xffffffffu, wk) & 15u;  // 15 - warp
          const unsigned char* src = wst + buf * WB + cw * SL_CAND;
          float2 pinv;
          bool mine = true;  // this CTA holds the pivot row
          unsigned sw = 0;   // piece swizzle of the row at src
          if (!SOLO) {
            if (warp < 2) {  // (at most eight CTAs: two warps send)
              const float4 v = *reinterpret_cast<const float4*>(src + (lane & 7) * 16);
              if (rk1 < CL) tc::st_async16(ra1 + buf * CB, v, rm1 + buf * 8);
              if (rk2 < CL) tc::st_async16(ra2 + buf * CB, v, rm2 + buf * 8);
              if (tid == 0) tc::mbar_expect_tx(&mbar[buf], cbytes);
            }
            if (ok) ok = tc::cluster_wait(&mbar[buf], (s >> 1) & 1, g.tries);
            // every warp reduces the candidates the same way
            const unsigned char* cb = cand + buf * CB;
            const int sl = lane & 7;
            float2 cp = *reinterpret_cast<const float2*>(cb + sl * SL_CAND + cand_piece(j >> 1, sl) +
                                                         (s & 1) * 8);
            float cv = cp.x * cp.x + cp.y * cp.y;
            const unsigned cmax = __reduce_max_sync(0xffffffffu, pivot_key(cv, sl));
            if (cv == 0.f) {
              cp = make_float2(1e-18f, 0.f);
              cv = 1e-36f;
            }
            const float rv = recip(cv);
            sw = cmax & 7u;
            src = cb + sw * SL_CAND;
            mine = sw == (unsigned)myslot;
            pinv.x = __shfl_sync(0xffffffffu, cp.x * rv, sw);
            pinv.y = __shfl_sync(0xffffffffu, -cp.y * rv, sw);
            // a pivot of zero, or not a number
            singular |= cmax - 32u >= 0x7f800020u - 32u;
          } else {
            float2 pv = *reinterpret_cast<const float2*>(src + j * 8);
            float pd = pv.x * pv.x + pv.y * pv.y;
            singular |= !(pd > 0.f);
            if (pd == 0.f) {
              pv = make_float2(1e-18f, 0.f);
              pd = 1e-36f;
            }
            const float rv = recip(pd);
            pinv = make_float2(pv.x * rv, -pv.y * rv);
          }
          float2 q[CPL];
#pragma unroll
          for (int c = 0; c < CPL; c += 2) {
            const float4 v = *reinterpret_cast<const float4*>(src + cand_piece((cg + c) / 2, sw));
            q[c] = make_float2(v.x, v.y);
            q[c + 1] = make_float2(v.z, v.w);
          }
          float2 m = make_float2(xs.y * pinv.y - xs.x * pinv.x, -xs.x * pinv.y - xs.y * pinv.x);
          if (mine && cw + warp == 15u) {  // (the whole warp)
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
              x[c].x = wrow ? 0.f : x[c].x;
              x[c].y = wrow ? 0.f : x[c].y;
            }
            m.x = wrow ? pinv.x : m.x;
            m.y = wrow ? pinv.y : m.y;
            elig = elig && !wrow;
            myj = wrow ? j : myj;
            if (wrow && cg == 0) own[p & 1][j] = prow;
          }
          if (!SOLO && !mine && tid == 0) own[p & 1][j] = -2;
#pragma unroll
          for (int cc = 1; cc <= CPL; ++cc) {
            const int c = (s + cc) % CPL;
            x[c].x = fmaf(m.x, q[c].x, fmaf(-m.y, q[c].y, x[c].x));
            x[c].y = fmaf(m.x, q[c].y, fmaf(m.y, q[c].x, x[c].y));
          }
          if (mycol) x[s] = m;
        }
      }
      if (live) {
#pragma unroll
        for (int c = 0; c < CPL; c += 2)
          *reinterpret_cast<float4*>(&S[prow * SL_LD + kl + cg + c]) =
              make_float4(x[c].x, x[c].y, x[c + 1].x, x[c + 1].y);
        if (myj >= 0) mypiv = c0 + kl + myj;
        if (cg == 0) rowp_p[prow] = myj;
      }
    } else if (npan > 1) {
      // beside the steps: the previous panel's transformation of the rest,
      const int uw = warp - pw, nuw = SL_WARPS - pw;
      if (p > 0)
        slab_update(S, Bq, rowp + ((p + 1) & 1) * rpc8, nrows, npan, p - 1, true, uw, nuw, lane);
      // then, every row being complete, the pivot rows as they become known
      asm volatile("bar.sync 2, %0;\n" ::"r"(nuw * 32) : "memory");
      const uint32_t mb = tc::smem_u32(&mbarB);
      for (int j = uw; j < NB; j += nuw) {
        // (a row beyond a ragged panel's columns waits for the last pivot: with one
        // buffer the panel warps read B, the panel before's, until their first step)
        int lr = -1;
        for (uint32_t t = 0; lr == -1 && t < g.tries; ++t) {
          lr = own[p & 1][min(j, nbk - 1)];
          if (lr == -1) __nanosleep(400);
        }
        if (lr == -1) ok = false;
        if (lr < 0 || j >= nbk) {
          // (rows beyond a ragged panel's columns multiply zeros; keep them finite)
          if (j >= nbk)
            for (int c = lane; c < GW_W; c += 32) Bp[j * GW_W + c] = make_float2(0.f, 0.f);
          continue;
        }
        const float4 v0 = *reinterpret_cast<const float4*>(&S[lr * SL_LD + 2 * lane]);
        const float4 v1 = *reinterpret_cast<const float4*>(&S[lr * SL_LD + 64 + 2 * lane]);
        if (SOLO) {
          *reinterpret_cast<float4*>(&Bp[j * GW_W + 2 * lane]) = v0;
          *reinterpret_cast<float4*>(&Bp[j * GW_W + 64 + 2 * lane]) = v1;
        } else {
          const uint32_t ba = tc::smem_u32(Bp + j * GW_W + 2 * lane);
          for (int d = 0; d < CL; ++d) {
            const uint32_t rm = tc::cluster_map(mb, d), ra = tc::cluster_map(ba, d);
            tc::st_async16(ra, v0, rm);
            tc::st_async16(ra + 512, v1, rm);
          }
        }
      }
    }
    __syncthreads();  // panel columns, rowp, the previous update, the sends' reads
    if (!SOLO && npan > 1 && ok) ok = tc::cluster_wait(&mbarB, p & 1, g.tries);
    if (npan > 1 && p + 1 == npan) {
      slab_update(S, Bp, rowp_p, nrows, npan, p, false, warp, SL_WARPS, lane);
      __syncthreads();
    }
  }
  for (int e = tid; e < nrows * (GW_W / 2); e += SL_THREADS) {
    const int r = e / (GW_W / 2), u = e - r * (GW_W / 2);
    if (2 * u < ncol)
      reinterpret_cast<float4*>(M + (size_t)(r * CL + rank) * b + c0)[u] =
          *reinterpret_cast<const float4*>(&S[r * SL_LD + 2 * u]);
  }
  if (live && cg == 0) {
    if (mypiv >= 0) {
      rowpiv[grow] = mypiv;
      g.pivslot[(size_t)f * b + mypiv] = grow;
    } else if (c0 == 0) {
      rowpiv[grow] = -1;
    }
  }
  if (rank == 0 && tid == 0 && singular) g.flag[f % g.F] = 1;
  if (!ok && lane == 0) atomicExch(g.err, 1);
  if (!ok) tc::cluster_settle();
  if (!SOLO) tc::cluster_sync();  // no CTA leaves while another may still send to it
}

// lanes per row: four where that leaves warps for the update
int slab_lpr(int rpc) { return rpc <= 8 * SL_PWMAX ? 4 : 2; }

// Cluster size of the slab kernel: the one with the least modelled time, waves
// of clusters x time of a full slab.  Measured at two problems: 72 us with 24
// rows per CTA, 91 with 48, 108 with 96 in clusters of eight (82 and 104 with
// 48 and 96 rows in clusters of four), 116 with 192 rows in one CTA, where the
// update beside the steps weighs most.
int slab_cluster(int b, int F, int device) {
  int best = SL_CLMAX;
  double bt = 1e30;
  for (int cl = 1; cl <= SL_CLMAX; ++cl) {
    const int rpc = (b + cl - 1) / cl;
    if (rpc > (cl == 1 ? 16 : 8) * SL_PWMAX || slab_smem_bytes(rpc, cl) > SL_SMEM_CAP) continue;
    const int slots = cluster_slots(device, cl);
    const int waves = (F + slots - 1) / slots;
    const double t = waves * (cl > 1 ? 60.0 + 0.5 * rpc : 45.0 + 0.37 * rpc);
    if (t < bt) {
      bt = t;
      best = cl;
    }
  }
  return best;
}

rr_status launch_slab(rr_factors* fa, int nh, int c0, int c1, cudaStream_t st) {
  const OpDev& d = fa->op->d;
  SlabArgs a;
  a.b = d.b;
  a.c0 = c0;
  a.c1 = c1;
  a.F = fa->F;
  const int P = fa->F * nh;  // problems of this launch
  a.CL = slab_cluster(d.b, P, d.device);
  a.rpc = (d.b + a.CL - 1) / a.CL;
  a.M = reinterpret_cast<float2*>(fa->M);
  a.rowpiv = fa->rowpiv;
  a.pivslot = fa->pivslot;
  a.flag = fa->flag;
  a.err = fa->err;
  a.tries = wait_tries();
  const size_t smem = slab_smem_bytes(a.rpc, a.CL);
  const int lpr = slab_lpr(a.rpc);
  RR_TRY((smem_opt_in<gjw_slab_kernel<true, 2>>(SL_SMEM_CAP)));
  RR_TRY((smem_opt_in<gjw_slab_kernel<true, 4>>(SL_SMEM_CAP)));
  RR_TRY((smem_opt_in<gjw_slab_kernel<false, 4>>(SL_SMEM_CAP)));
  prof_begin(PROF_PANEL, st);
  if (a.CL == 1) {
    if (lpr == 4) gjw_slab_kernel<true, 4><<<P, SL_THREADS, smem, st>>>(a);
    else gjw_slab_kernel<true, 2><<<P, SL_THREADS, smem, st>>>(a);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.CL * P), 1, 1);
    cfg.blockDim = dim3(SL_THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = a.CL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    RR_CUDA(cudaLaunchKernelEx(&cfg, gjw_slab_kernel<false, 4>, a));
  }
  prof_end(PROF_PANEL, st);
  RR_CUDA(cudaGetLastError());
  return RR_OK;
}

// Outer-update right operand: Bout[f][c][m] = M[P_{c0+c}][m] for m outside
// [c0, c1) and c < c1 - c0; zero elsewhere (rows up to GW_W).
__global__ void gjw_gather_kernel(int b, int c0, int c1, const float2* __restrict__ Mall,
                                  const int* __restrict__ pivslot_all, float2* __restrict__ Bout) {
  const int half = blockIdx.x / GW_W;
  const int f = half * gridDim.y + blockIdx.y;
  const int c = blockIdx.x - half * GW_W;  // 0 .. GW_W - 1
  const float2* M = Mall + (size_t)f * b * b;
  float2* dst = Bout + ((size_t)f * GW_W + c) * b;
  const bool row_ok = c < c1 - c0;
  const int p = row_ok ? pivslot_all[(size_t)f * b + c0 + c] : 0;
  for (int m = threadIdx.x; m < b; m += blockDim.x) {
    float2 v = make_float2(0.f, 0.f);
    if (row_ok && (m < c0 || m >= c1)) v = M[(size_t)p * b + m];
    dst[m] = v;
  }
}

// --------------------------------------------------------------- tensor GEMM
// C[f][rows][cols] (+)= A[f] B[f] for complex FP32 data:
//   A = M[f][:, ka .. ka + Kc)          (b x Kc, from M by TMA)
//   B = Wbuf[f][0..Kc)[cols]            (Kc x b rows by TMA: the slab's pivot rows)
// rows pivoted in [ka, ka + Kc) are overwritten with the product, the other
// rows accumulate it, and the columns [ka, ka + Kc) are left alone.
// Items (problem, 128-row tile, 64-column tile) over the column tiles of up
// to two ranges; persistent CTAs take items round-robin.  Per item the
// contraction runs in chunks of 16 complex columns of A (32 reals of K):
//   control warp : TMA of the raw A chunk (128 x 32 floats) and B chunk (16 x
//                  64 complex) into a 4-stage ring, and the MMAs of each
//                  converted chunk into the item's TMEM accumulator (two, by
//                  item parity);
//   8 converter warps: split the raw chunk into operand pieces (K-major
//                  core-matrix tiles; B expanded to the real 128 x 32 matrix
//                  with rows (Re, -Im), (Im, Re) so one real GEMM gives the
//                  complex product), double-buffered;
//   8 epilogue warps: prefetch the item's rows of C, read the accumulator
//                  (TMEM lane = row) and add it in place,
// so the epilogue of item t overlaps the chunks of item t + 1.  Every wait is
// bounded (tries polls); a timeout sets *err, every role winds down, and the
// control thread drains its copies and MMAs before TMEM is freed.
using tc::SPLIT_BF16X3;
using tc::SPLIT_BF16X6;
using tc::SPLIT_TF32X3;
template <int SPLIT> struct SplitCfg : tc::SplitCfg<SPLIT> {
  static constexpr int KSTEPS = tc::ksteps32<SPLIT>();
};

// piece products (A piece, B piece) in the order they are accumulated: the
// first three are hi.hi, hi.lo, lo.hi (x3 splits); BF16x6 adds the three
// products of the next order, hi.lo2, lo.lo, lo2.hi
__device__ __forceinline__ int prod_a(int pr) { return pr == 2 || pr == 4 ? 1 : pr == 5 ? 2 : 0; }
__device__ __forceinline__ int prod_b(int pr) { return pr == 1 || pr == 4 ? 1 : pr == 3 ? 2 : 0; }

constexpr int GG_RT = 128, GG_CT = 64, GG_KC = 16;  // rows, complex cols, complex K per chunk
constexpr int GG_STAGES = 4;
constexpr uint32_t GG_RAW_A = GG_RT * 2 * GG_KC * 4;  // 16 KB
constexpr uint32_t GG_RAW_B = GG_KC * GG_CT * 8;      // 8 KB
constexpr uint32_t GG_RAW_STAGE = GG_RAW_A + GG_RAW_B;
constexpr int GG_EPI = 256, GG_CONV = 256;
constexpr int GG_THREADS = GG_EPI + GG_CONV + 32;
constexpr uint32_t GG_LBO = 128;

template <int SPLIT>
__host__ __device__ constexpr uint32_t gg_piece_bytes() {
  return (uint32_t)GG_RT * 2 * GG_KC * SplitCfg<SPLIT>::ESZ;  // 128 rows x 32 reals
}
template <int SPLIT>
__host__ __device__ constexpr uint32_t gg_sbo() {
  return tc::sbo32<SPLIT>();  // 32 reals of K per row
}
template <int SPLIT>
__host__ __device__ constexpr uint32_t gg_opbuf_bytes() {
  return 2 * SplitCfg<SPLIT>::PIECES * gg_piece_bytes<SPLIT>();  // A pieces + B pieces
}
template <int SPLIT>
__host__ __device__ constexpr size_t gg_smem_bytes() {
  return 2 * (size_t)gg_opbuf_bytes<SPLIT>() + (size_t)GG_STAGES * GG_RAW_STAGE + 1024;
}

struct GemmArgs {
  int b, F, ka, Kc;            // K range [ka, ka + Kc) of M's columns, Kc % 16 == 0
  int x0, x1, y0, y1;          // column tiles [x0, x1) and [y0, y1) (64 complex each)
  float2* M;
  const int* rowpiv;           // [F][b]
  int* err;
  uint32_t tries;
};

__device__ __forceinline__ bool gg_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                        uint32_t tries) {
  for (uint32_t t = 0; t < tries; ++t) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}

__device__ __forceinline__ void gg_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tc::smem_u32(bar)) : "memory");
}

template <int SPLIT>
__global__ void __launch_bounds__(GG_THREADS, 1)
gjw_gemm_kernel(const __grid_constant__ CUtensorMap tmapA, const __grid_constant__ CUtensorMap tmapB,
                GemmArgs g) {
  using Cfg = SplitCfg<SPLIT>;
  constexpr int PIECES = Cfg::PIECES;
  constexpr uint32_t PB = gg_piece_bytes<SPLIT>();
  constexpr uint32_t OPB = gg_opbuf_bytes<SPLIT>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t full_bar[GG_STAGES], opready[2], opfree[2], accfull[2], accempty[2], drain;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* ops = base;                    // 2 operand buffers
  unsigned char* raw = base + 2 * OPB;          // GG_STAGES raw stages
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool is_epi = tid < GG_EPI;
  const bool is_conv = tid >= GG_EPI && tid < GG_EPI + GG_CONV;
  const bool is_ctrl = tid == GG_EPI + GG_CONV;
  const int b = g.b;
  const int nrt = (b + GG_RT - 1) / GG_RT;
  const int n1 = g.x1 - g.x0, nct = n1 + (g.y1 - g.y0);
  const int nitems = g.F * nrt * nct;
  const int nk = g.Kc / GG_KC;
  const int my_items = nitems > (int)blockIdx.x
                           ? (nitems - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x
                           : 0;
  auto item = [&](int t, int& f, int& rt, int& ctile) {
    const int it = (int)blockIdx.x + t * (int)gridDim.x;
    const int ct = it % nct;
    rt = (it / nct) % nrt;
    f = it / (nct * nrt);
    ctile = ct < n1 ? g.x0 + ct : g.y0 + (ct - n1);
  };

  if (warp == 0) tc::tmem_alloc(&tmem_base, 256);
  if (tid == 0) {
    for (int s = 0; s < GG_STAGES; ++s) tc::mbar_init(&full_bar[s], 1);
    for (int q = 0; q < 2; ++q) {
      tc::mbar_init(&opready[q], GG_CONV);
      tc::mbar_init(&opfree[q], 1);
      tc::mbar_init(&accfull[q], 1);
      tc::mbar_init(&accempty[q], GG_EPI);
    }
    tc::mbar_init(&drain, 1);
    abort_sh = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base;

  if (is_ctrl) {
    // ---------------------------------------------------- control thread
    const uint32_t idesc = SPLIT == SPLIT_TF32X3 ? tc::idesc_tf32(GG_RT, 2 * GG_CT)
                                                 : tc::idesc_bf16(GG_RT, 2 * GG_CT);
    int p_t = 0, p_kc = 0, issued = 0;
    int pf = 0, prt = 0, pct = 0;
    if (my_items > 0) item(0, pf, prt, pct);
    auto issue_next = [&]() {
      if (p_t >= my_items) return;
      const int s = issued % GG_STAGES;
      unsigned char* st = raw + s * GG_RAW_STAGE;
      tc::mbar_expect_tx(&full_bar[s], GG_RAW_STAGE);
      tc::tma_load_3d(st, &tmapA, 2 * (g.ka + p_kc * GG_KC), prt * GG_RT, pf, &full_bar[s]);
      tc::tma_load_3d(st + GG_RAW_A, &tmapB, 2 * pct * GG_CT, p_kc * GG_KC, pf, &full_bar[s]);
      ++issued;
      if (++p_kc == nk) {
        p_kc = 0;
        if (++p_t < my_items) item(p_t, pf, prt, pct);
      }
    };
    for (int q = 0; q < GG_STAGES; ++q) issue_next();
    int gch = 0;
    bool ok = true;
    for (int t = 0; t < my_items && ok; ++t) {
      const int a = t & 1;
      if (t >= 2) ok = gg_wait(&accempty[a], (uint32_t)((t - 2) >> 1) & 1u, abort_flag, g.tries);
      for (int kc = 0; kc < nk && ok; ++kc, ++gch) {
        const int q = gch & 1;
        ok = gg_wait(&opready[q], (uint32_t)(gch >> 1) & 1u, abort_flag, g.tries);
        if (!ok) break;
        issue_next();  // raw stage of chunk gch has been converted: refill it
        tc::fence_after_sync();
        const uint32_t acc = tmem + (uint32_t)a * (2 * GG_CT);
        const uint32_t ob = tc::smem_u32(ops + q * OPB);
#pragma unroll
        for (int ks = 0; ks < Cfg::KSTEPS; ++ks) {
#pragma unroll
          for (int pr = 0; pr < Cfg::NPROD; ++pr) {
            const int pa = prod_a(pr), pb = prod_b(pr);
            const uint64_t da = tc::smem_desc(ob + pa * PB + ks * 2 * GG_LBO, GG_LBO, gg_sbo<SPLIT>());
            const uint64_t db = tc::smem_desc(ob + (PIECES + pb) * PB + ks * 2 * GG_LBO, GG_LBO,
                                              gg_sbo<SPLIT>());
            const uint32_t accum = (kc > 0 || ks > 0 || pr > 0) ? 1u : 0u;
            if (SPLIT == SPLIT_TF32X3) tc::mma_tf32(acc, da, db, idesc, accum);
            else tc::mma_bf16(acc, da, db, idesc, accum);
          }
        }
        tc::mma_commit(&opfree[q]);
        if (kc == nk - 1) tc::mma_commit(&accfull[a]);
      }
    }
    if (!ok) {
      *abort_flag = 1;
      // copies still in flight: the last GG_STAGES issued chunks
      for (int c = max(0, issued - GG_STAGES); c < issued; ++c)
        tc::mbar_wait(&full_bar[c % GG_STAGES], (uint32_t)(c / GG_STAGES) & 1u, 1u << 22);
    }
    // every MMA this thread issued completes before TMEM is freed
    tc::mma_commit(&drain);
    tc::mbar_wait(&drain, 0, 1u << 22);
  } else if (is_conv) {
    // -------------------------------------------------------- converters
    const int ct_id = tid - GG_EPI;
    int gch = 0;
    bool ok = true;
    for (int t = 0; t < my_items && ok; ++t) {
      int f, rt, ctile;
      item(t, f, rt, ctile);
      for (int kc = 0; kc < nk; ++kc, ++gch) {
        const int s = gch % GG_STAGES, q = gch & 1;
        ok = gg_wait(&full_bar[s], (uint32_t)(gch / GG_STAGES) & 1u, abort_flag, g.tries);
        if (ok && gch >= 2) ok = gg_wait(&opfree[q], (uint32_t)((gch - 2) >> 1) & 1u, abort_flag, g.tries);
        if (!ok) break;
        const float* RA = reinterpret_cast<const float*>(raw + s * GG_RAW_STAGE);
        const float2* RB = reinterpret_cast<const float2*>(raw + s * GG_RAW_STAGE + GG_RAW_A);
        unsigned char* ob = ops + q * OPB;
        unsigned char* pa[3] = {ob, ob + PB, ob + 2 * PB};
        unsigned char* pbp[3] = {ob + PIECES * PB, ob + (PIECES + 1) * PB, ob + (PIECES + 2) * PB};
        // A: 128 rows x 8 units of 4 reals; rotated order for distinct banks
        for (int it = ct_id; it < GG_RT * 8; it += GG_CONV) {
          const int row = (it & 7) + 8 * (it >> 6);
          const int p = (((it >> 3) & 7) + row) & 7;
          const float4 v = *reinterpret_cast<const float4*>(RA + row * 32 + 4 * p);
          tc::store_split<SPLIT>(v, pa, tc::kmajor_off32<SPLIT>(row, 4 * p));
        }
        // B: 64 complex columns j x 8 pairs of K rows -> real rows 2j, 2j+1
        for (int it = ct_id; it < GG_CT * 8; it += GG_CONV) {
          const int j = it % GG_CT, pp = it / GG_CT;
          const float2 t0 = RB[(2 * pp) * GG_CT + j], t1 = RB[(2 * pp + 1) * GG_CT + j];
          tc::store_split<SPLIT>(make_float4(t0.x, -t0.y, t1.x, -t1.y), pbp, tc::kmajor_off32<SPLIT>(2 * j, 4 * pp));
          tc::store_split<SPLIT>(make_float4(t0.y, t0.x, t1.y, t1.x), pbp, tc::kmajor_off32<SPLIT>(2 * j + 1, 4 * pp));
        }
        tc::fence_async_smem();
        gg_arrive(&opready[q]);
      }
    }
    if (!ok) *abort_flag = 1;
  } else if (is_epi) {
    // ---------------------------------------------------------- epilogue
    // warp w reads TMEM lanes 32 (w % 4) .. + 31 (its quadrant) in two
    // 16-lane blocks, complex columns 32 (w / 4) .. + 31 of the tile, with
    // the 16x256b fragment: thread t holds rows base + t/4 and base + t/4 + 8
    // and complex columns 4 r + t % 4 (r = 0..7), so every global access of
    // a warp covers 8 rows x 32 contiguous bytes
    const int lq = warp & 3, half = warp >> 2;
    bool ok = true;
    for (int t = 0; t < my_items && ok; ++t) {
      int f, rt, ctile;
      item(t, f, rt, ctile);
      const int a = t & 1;
      const int cb = ctile * GG_CT + half * 32 + (lane & 3);  // + 4 r
      float2* Mf = g.M + (size_t)f * b * b;
      const int* rpf = g.rowpiv + (size_t)f * b;
      int row[4];
      bool add[4];
      float2 cm[4][8];
#pragma unroll
      for (int u = 0; u < 4; ++u) {  // u = 2 * sub-block + (second row)
        row[u] = rt * GG_RT + lq * 32 + 16 * (u >> 1) + (lane >> 2) + 8 * (u & 1);
        // a pivot row of the contraction's columns takes the product itself
        // (E[p, P] B = T^{-1} B); every other row adds it
        const int rp = row[u] < b ? rpf[row[u]] : -1;
        add[u] = !(rp >= g.ka && rp < g.ka + g.Kc);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int c = cb + 4 * r;
          cm[u][r] = (row[u] < b && add[u] && c < b) ? Mf[(size_t)row[u] * b + c]
                                                      : make_float2(0.f, 0.f);
        }
      }
      ok = gg_wait(&accfull[a], (uint32_t)(t >> 1) & 1u, abort_flag, g.tries);
      if (!ok) break;
      tc::fence_after_sync();
#pragma unroll
      for (int sb = 0; sb < 2; ++sb) {
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          float v[16];
          tc::tmem_ld_16x256b_x4(tmem + ((uint32_t)(lq * 32 + 16 * sb) << 16) +
                                     (uint32_t)a * (2 * GG_CT) + (uint32_t)(half * 64 + hh * 32),
                                 v);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            cm[2 * sb][4 * hh + r].x += v[4 * r];
            cm[2 * sb][4 * hh + r].y += v[4 * r + 1];
            cm[2 * sb + 1][4 * hh + r].x += v[4 * r + 2];
            cm[2 * sb + 1][4 * hh + r].y += v[4 * r + 3];
          }
        }
      }
      tc::fence_before_sync();
      gg_arrive(&accempty[a]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (row[u] >= b) continue;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          // the contraction's own columns (the slab) keep their values
          const int c = cb + 4 * r;
          if (c < b && !(c >= g.ka && c < g.ka + g.Kc)) Mf[(size_t)row[u] * b + c] = cm[u][r];
        }
      }
    }
    if (!ok) *abort_flag = 1;
  }
  tc::fence_before_sync();
  __syncthreads();
  if (tid == 0 && *abort_flag) atomicExch(g.err, 1);
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

// ---------------------------------------------------------------- finalize
// G_i[j][p_m] = M[p_j][m] (S^{-1} from the implicitly pivoted work matrix),
// X_i = G_i C_i with C_i = -L_{i,i+1} in half 0 and G_i A_i with A_i = -L_{i,i-1}
// in half 1 (at most 3q entries per column).  A CTA
// gathers RB rows into shared memory (scattering the columns), writes them
// as rows of G_i and forms the same rows of X_i; each thread owns fixed
// columns of X_i, so the (up to 3q) coupling coefficients of a column are
// loaded once and reused for all RB rows.
constexpr int FIN_THREADS = 256, FIN_CPT = 4;  // columns per thread (b <= 1024)

__global__ void __launch_bounds__(FIN_THREADS)
gjw_finalize_kernel(OpView op, int nh, int col0, int col1, int RB,
                    const float2* __restrict__ Mall, const int* __restrict__ pivslot_all,
                    float2* __restrict__ Gall, float2* __restrict__ Xall) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int b = op.b, q = op.q;
  float2* Gs = reinterpret_cast<float2*>(smem_raw);        // [RB][b]
  int* ps = reinterpret_cast<int*>(Gs + (size_t)RB * b);   // [b]
  const int nt = gridDim.x / nh, half = blockIdx.x / nt;
  const int f = blockIdx.y, pf = half * gridDim.y + f, i = half ? col1 : col0;
  const int r0 = (blockIdx.x - half * nt) * RB;
  const int nr = min(RB, b - r0);
  const float2* M = Mall + (size_t)pf * b * b;
  for (int c = threadIdx.x; c < b; c += FIN_THREADS) ps[c] = pivslot_all[(size_t)pf * b + c];
  __syncthreads();
  for (int e = threadIdx.x; e < nr * b; e += FIN_THREADS) {
    const int rr = e / b, c = e - rr * b;
    Gs[rr * b + ps[c]] = M[(size_t)ps[r0 + rr] * b + c];
  }
  __syncthreads();
  float2* G = Gall + ((size_t)f * op.nx + i) * b * b;  // (b % 8 == 0: ldg is b)
  for (int e = threadIdx.x; e < nr * b; e += FIN_THREADS) {
    const int rr = e / b, c = e - rr * b;
    G[(size_t)(r0 + rr) * b + c] = Gs[rr * b + c];
  }
  if (Xall == nullptr) return;
  float2* X = Xall + (size_t)pf * b * b;
#pragma unroll
  for (int k = 0; k < FIN_CPT; ++k) {
    const int c = threadIdx.x + k * FIN_THREADS;
    if (c >= b) break;
    // the coupling of column c: entries L[(i, m), (i +- 1, c)] (half 0: + 1) for
    // the rows m of the y neighbours of c's point
    const int iyc = c / q, cc = c - iyc * q;
    int mm[12];  // 3 y neighbours x q <= 4 variables
    float aa[12];
#pragma unroll
    for (int t = 0; t < 12; ++t) {
      mm[t] = 0;
      aa[t] = 0.f;
      if (t < 3 * q) {
        const int dy = t / q - 1, cm = t - (t / q) * q;
        const int iym = nbr_y(iyc, -dy, op.ny, op.periodic);
        if (iym >= 0) {
          mm[t] = iym * q + cm;
          aa[t] = op.coef32[((size_t)i * b + mm[t]) * op.S + ((half ? 0 : 6) + (dy + 1)) * q + cc];
        }
      }
    }
    for (int rr = 0; rr < nr; ++rr) {
      float2 s = make_float2(0.f, 0.f);
#pragma unroll
      for (int t = 0; t < 12; ++t)
        if (aa[t] != 0.f) s = crfma(aa[t], Gs[rr * b + mm[t]], s);
      X[(size_t)(r0 + rr) * b + c] = make_float2(-s.x, -s.y);
    }
  }
}

template <int SPLIT>
rr_status launch_gemm(rr_factors* fa, int nh, const CUtensorMap* ta, const CUtensorMap* tb, int ka, int Kc,
                      int x0, int x1, int y0, int y1, cudaStream_t st) {
  const OpDev& d = fa->op->d;
  GemmArgs a;
  a.b = d.b;
  a.F = fa->F * nh;
  a.ka = ka;
  a.Kc = Kc;
  a.x0 = x0; a.x1 = x1; a.y0 = y0; a.y1 = y1;
  a.M = reinterpret_cast<float2*>(fa->M);
  a.rowpiv = fa->rowpiv;
  a.err = fa->err;
  a.tries = wait_tries();
  const int nrt = (d.b + GG_RT - 1) / GG_RT;
  const long items = (long)a.F * nrt * ((x1 - x0) + (y1 - y0));
  if (items <= 0) return RR_OK;
  // small launches (up to 8 items per SM): one wave of persistent CTAs;
  // large ones: about four items per CTA, so CTAs retire during the launch
  // and the second stream's panels find SMs as they free up
  const long nsm = num_sms(d.device);
  const int grid = (int)(items <= 8 * nsm ? std::min<long>(items, nsm) : (items + 3) / 4);
  RR_TRY(smem_opt_in<gjw_gemm_kernel<SPLIT>>(gg_smem_bytes<SPLIT>()));
  prof_begin(PROF_UPDATE, st);
  gjw_gemm_kernel<SPLIT><<<grid, GG_THREADS, gg_smem_bytes<SPLIT>(), st>>>(*ta, *tb, a);
  prof_end(PROF_UPDATE, st);
  RR_CUDA(cudaGetLastError());
  return RR_OK;
}

template <int SPLIT>
rr_status factor_wide_impl(rr_factors* fa) {
  const OpDev& d = fa->op->d;
  const OpView ov = view(d);
  const int b = d.b, F = fa->F;
  cudaStream_t st = fa->stream;
  float2* M = reinterpret_cast<float2*>(fa->M);
  float2* G = reinterpret_cast<float2*>(fa->G);
  float2* X = reinterpret_cast<float2*>(fa->X);
  const CUtensorMap* tA = reinterpret_cast<const CUtensorMap*>(fa->wmap[0]);
  const CUtensorMap* tBout = reinterpret_cast<const CUtensorMap*>(fa->wmap[1]);
  const int RB = 8;
  const size_t fsmem = (size_t)RB * b * sizeof(float2) + b * sizeof(int);
  RR_TRY(smem_opt_in<gjw_finalize_kernel>((size_t)RB * GW_MAX * sizeof(float2) +
                                          GW_MAX * sizeof(int)));
  const int nct_all = (b + GG_CT - 1) / GG_CT;
  for (int step = 0; step < twist_steps(fa); ++step) {
    const TwistStep t = twist_step(fa, step);
    const int nh = t.nh;
    rr_status s = launch_schur_f32(fa, t, st);
    if (s != RR_OK) return s;
    // Look-ahead: once the next slab's columns have received this slab's
    // rank-128 update, the next slab's inner factorisation runs on the second
    // (high-priority) stream while the rank-128 update of the remaining
    // columns proceeds on the main stream; the two touch disjoint columns of
    // M (rowpiv entries of the next slab's pivot rows change meanwhile, but
    // only from "not pivoted" to a column outside this slab, which the main
    // stream's update reads as "not a pivot of this slab" either way).  The
    // next slab's pivot rows are gathered on the main stream after both.
    cudaStream_t st2 = fa->stream2;
    if ((s = launch_slab(fa, nh, 0, std::min(b, GW_W), st)) != RR_OK) return s;
    for (int c0 = 0; c0 < b; c0 += GW_W) {
      const int c1 = std::min(b, c0 + GW_W);
      if (c1 >= b && c0 == 0) break;  // one slab: no outer update
      prof_begin(PROF_ROWBLOCK, st);
      gjw_gather_kernel<<<dim3(GW_W * nh, F), 256, 0, st>>>(b, c0, c1, M, fa->pivslot,
                                                      reinterpret_cast<float2*>(fa->Wbuf));
      prof_end(PROF_ROWBLOCK, st);
      const int s0 = c0 / GG_CT, s1 = (c1 + GG_CT - 1) / GG_CT;
      if (c1 < b) {
        const int n1 = std::min(b, c1 + GW_W);
        const int u1 = (n1 + GG_CT - 1) / GG_CT;  // tiles [s1, u1): the next slab
        if ((s = launch_gemm<SPLIT>(fa, nh, tA, tBout, c0, GW_W, s1, u1, 0, 0, st)) != RR_OK) return s;
        if (st2 != nullptr) {
          RR_CUDA(cudaEventRecord(fa->ev_next, st));
          RR_CUDA(cudaStreamWaitEvent(st2, fa->ev_next, 0));
          if ((s = launch_slab(fa, nh, c1, n1, st2)) != RR_OK) return s;
          RR_CUDA(cudaEventRecord(fa->ev_panel, st2));
          if ((s = launch_gemm<SPLIT>(fa, nh, tA, tBout, c0, GW_W, 0, s0, u1, nct_all, st)) != RR_OK)
            return s;
          RR_CUDA(cudaStreamWaitEvent(st, fa->ev_panel, 0));
        } else {
          if ((s = launch_gemm<SPLIT>(fa, nh, tA, tBout, c0, GW_W, 0, s0, u1, nct_all, st)) != RR_OK)
            return s;
          if ((s = launch_slab(fa, nh, c1, n1, st)) != RR_OK) return s;
        }
      } else {
        if ((s = launch_gemm<SPLIT>(fa, nh, tA, tBout, c0, GW_W, 0, s0, 0, 0, st)) != RR_OK) return s;
      }
    }
    prof_begin(PROF_FINALIZE, st);
    gjw_finalize_kernel<<<dim3((b + RB - 1) / RB * nh, F), FIN_THREADS, fsmem, st>>>(
        ov, nh, t.col0, t.col1, RB, M, fa->pivslot, G, t.middle ? nullptr : X);
    prof_end(PROF_FINALIZE, st);
    RR_CUDA(cudaGetLastError());
  }
  return RR_OK;
}

}  // namespace

// Clusters of cl CTAs (at most eight, one CTA per SM) resident at once: what the
// GPCs hold, 152, 76, 46, 36, 28, 23, 15 and 15 on the GB300 measured.
int cluster_slots(int device, int cl) {
  static int cached[64][SL_CLMAX + 1];
  static std::mutex mu;
  if (cl < 1 || cl > SL_CLMAX) return 1;
  const int dev = device >= 0 && device < 64 ? device : 0;
  std::lock_guard<std::mutex> lock(mu);
  int& n = cached[dev][cl];
  if (n == 0) {
    constexpr int smem = 200 * 1024;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cl * 64), 1, 1);
    cfg.blockDim = dim3(SL_THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (smem_opt_in<gjw_slab_kernel<false, 4>>(SL_SMEM_CAP) != RR_OK ||
        cudaOccupancyMaxActiveClusters(&n, gjw_slab_kernel<false, 4>, &cfg) != cudaSuccess ||
        n <= 0) {
      cudaGetLastError();
      n = std::max(1, num_sms(device) / 19 * (19 / cl));  // (a GPC of 19 SMs)
    }
  }
  return n;
}

// The wide path needs FP32 factors, a block of a multiple of 8 rows, at most
// 768 and at least 64, and the TMA maps of M and of the
// gathered pivot rows.
bool factor_wide_ok(const rr_factors* fa) {
  const int b = fa->op->d.b;
  return fa->wide_ok && b >= 64 && b <= GW_MAX && (b % 8) == 0 &&
         (fa->prec == RR_FP32 || fa->prec == RR_FP32_BF16X3 || fa->prec == RR_FP32_BF16X6);
}

rr_status launch_factor_wide(rr_factors* fa) {
  switch (fa->prec) {
    case RR_FP32_BF16X3: return factor_wide_impl<SPLIT_BF16X3>(fa);
    case RR_FP32_BF16X6: return factor_wide_impl<SPLIT_BF16X6>(fa);
    default: return factor_wide_impl<SPLIT_TF32X3>(fa);
  }
}
