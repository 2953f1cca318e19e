// Whole block sweeps in two launches: the sweeps of a solve from both ends to the
// middle column and back out (see sweep.cu for the recurrences), each run by one
// thread-block cluster per problem, half and group of right-hand-side columns,
// in FP32 or FP64 on the CUDA cores.  The halves meet between the launches: the
// inward one leaves each half's last result in an edge buffer, from which both
// halves of the outward one form the middle column's right-hand side (and both
// multiply it: cheaper than an exchange between clusters).
//
// CTA `rank` of a cluster owns the grid points [rank npt, (rank + 1) npt) of
// every streamwise column (npt q rows).  Step s of a solve multiplies one G_i
// (or G_i^H) into the staged block t_s, which every CTA holds whole:
//   product : warp w takes the chunks w, w + W, ... of the contraction; its
//             slices of G (the CTA's rows, 64 bytes of each, or for G^H 64 bytes
//             worth of G's rows at the CTA's columns) arrive by cp.async in a
//             ring of the warp's own, two chunks ahead and across steps (G does
//             not depend on the sweep), so no barrier orders them; a lane holds
//             RPL x CPL outputs;
//   sum     : the warps' partial blocks are added in order, the step's result o
//             is stored, and its first and last point go to the neighbouring
//             CTAs (the couplings reach one point in y);
//   couple  : t_{s+1} = in + (stencil coupling) o at the CTA's rows, sent to
//             every CTA of the cluster (st.async completing on the receiver's
//             mbarrier).
// t is double-buffered by step parity: a CTA sends t_{s+2} only after it has
// all of t_{s+1}, of which each CTA sends its part after its product s.  Waits
// are bounded; a CTA that gives up records it in *err and leaves the step loop.
//
// Bound: at small blocks the chain of a step (products of a few hundred cycles,
// two exchanges), at large ones FP32 (FP64) arithmetic.
#pragma once

#include <algorithm>

#include "rr_internal.cuh"
#include "tc.cuh"

namespace sweepcl {

constexpr int MAXW = 16;         // warps of a CTA
constexpr int CLMAX = 8;         // largest cluster
constexpr int PITCH = 80;        // bytes of a staged row of G: 64 and a bank shift
constexpr size_t SMEM_CAP = 220 * 1024;

template <typename T>
struct Args {
  OpView op;
  const C_t<T>* G;     // [F][nx][b][ldg]
  size_t gstride;      // one problem of G
  int ldg;
  const C_t<T>* in;    // [F][N][k]
  C_t<T>* x;           // [F][N][k]
  C_t<T>* h;           // [F][N][k] scratch (adjoint)
  C_t<T>* edge;        // [2][F][b][k] last inward result of each half
  int F, out;          // problems; inward (0) or outward (1) launch
  int k, ng, npt, CL;
  const int* amap;
  int* err;
  uint32_t tries;
  int stall;           // diagnostic: the first CTA sends nothing
};

template <typename T, int KC, bool TRANS>
__host__ __device__ constexpr size_t stage_bytes(int rmax) {
  return TRANS ? ((size_t)KC * rmax * sizeof(C_t<T>) + 15) & ~(size_t)15 : (size_t)rmax * PITCH;
}
template <typename T, bool TRANS>
size_t smem_bytes(int b, int rmax, int q, int kc, int W) {
  constexpr int KC = 64 / sizeof(C_t<T>);
  const int bp = (b + KC - 1) / KC * KC;
  return ((size_t)2 * bp * kc + (size_t)W * rmax * kc + (size_t)(rmax + 2 * q) * kc) *
             sizeof(C_t<T>) +
         (size_t)2 * W * stage_bytes<T, KC, TRANS>(rmax);
}

__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, int bytes, bool ok) {
  // bytes: 16 or 8; zero-filled when !ok
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(dst), "l"(src),
                 "r"(ok ? 8 : 0)
                 : "memory");
}

// Warps of a CTA: large lane tiles need more than the 128 registers that sixteen
// warps leave them
template <typename T, int CPL, int RPL>
constexpr int max_warps() { return sizeof(T) == 4 && CPL * RPL >= 20 ? 8 : MAXW; }

// LR = 32 / LC lanes over rows x LC over columns; a lane holds RPL rows (LR
// apart) x CPL adjacent columns.  PITCHED: G's rows are a.ldg apart, else b.  (The forward
// kernels are pitched always: up to a third faster at 384 and 768 rows than with b; the
// adjoint ones were 2 to 5 % slower at 192 rows.)
template <typename T, bool TRANS, int LC, int CPL, int RPL, bool PITCHED>
__global__ void __launch_bounds__(max_warps<T, CPL, RPL>() * 32, 1) sweep_cl_kernel(Args<T> a) {
  using C = C_t<T>;
  constexpr int CS = sizeof(C);
  constexpr int KC = 64 / CS;            // contraction columns of a chunk
  constexpr int LR = 32 / LC, NC = LC * CPL;
  constexpr int VEC = 16 / CS;           // columns of a 16-byte unit
  constexpr int UPR = NC / VEC;          // units of a row
  constexpr int EP = 2;                  // units of a thread, at most
  static_assert(NC % VEC == 0, "whole units");
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint64_t mT[2], mH[2];
  const OpView& op = a.op;
  const int b = op.b, q = op.q, nx = op.nx, ny = op.ny, CL = a.CL, npt = a.npt;
  const int W = blockDim.x >> 5, nthr = blockDim.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)tc::cluster_rank();
  const int cl = blockIdx.x / CL, half = cl & 1, f = active_problem(a.amap, (cl >> 1) / a.ng);
  const int j0 = ((cl >> 1) % a.ng) * NC;
  const int rmax = npt * q, bp = (b + KC - 1) / KC * KC, nch = bp / KC;
  const int pts = max(0, min(npt, ny - rank * npt)), rows = pts * q, row0 = rank * rmax;
  const size_t SB = stage_bytes<T, KC, TRANS>(rmax);
  C* tb = reinterpret_cast<C*>(smem);                         // [2][bp][NC]
  C* red = tb + (size_t)2 * bp * NC;                          // [W][rmax][NC]
  C* ob = red + (size_t)W * rmax * NC;                        // [rmax + 2 q][NC]
  unsigned char* ring = reinterpret_cast<unsigned char*>(ob + (size_t)(rmax + 2 * q) * NC) +
                        (size_t)warp * 2 * SB;
  const C* Gf = a.G + (size_t)f * a.gstride;
  const int ldg = PITCHED ? a.ldg : b;
  const size_t bb = (size_t)b * ldg, NK = (size_t)op.n * a.k;
  const C* in = a.in + (size_t)f * NK;
  C* x = a.x + (size_t)f * NK;
  C* h = TRANS ? a.h + (size_t)f * NK : nullptr;
  const int k = a.k;
  // columns of the half: step s of the inward launch is column s (nx - 1 - s), of
  // the outward one column mid - s (mid + s), the middle first
  const bool outw = a.out != 0;
  const int mid = twist_mid(nx);
  const int nstep = (half ? nx - 1 - mid : mid) + (outw ? 1 : 0);
  const int dcol = (half != 0) == outw ? 1 : -1;      // column of step s + 1 minus that of s
  const int col0 = outw ? mid : half ? nx - 1 : 0;
  auto step_col = [&](int s) { return col0 + s * dcol; };

  if (tid < 2) {
    tc::mbar_init(&mT[tid], 1);
    tc::mbar_init(&mH[tid], 1);
  }
  for (int e = tid; e < 2 * bp * NC; e += nthr) tb[e] = czero<C>();
  for (int e = tid; e < (rmax + 2 * q) * NC; e += nthr) ob[e] = czero<C>();
  tc::cluster_sync();  // barriers and zeroed buffers before any CTA sends

  // ---- this warp's stream of G chunks: two in flight, step after step
  // bytes of a copy: 16 where every segment starts and ends on 16 bytes
  const int gb = (b % VEC == 0 && (!TRANS || rmax % VEC == 0)) ? 16 : CS;
  int is = 0, ic = warp;  // next chunk to request
  const int per = (TRANS ? rmax * CS : 64) / gb;   // copies of a segment
  const int walk_s = 32 / per, walk_u = 32 - walk_s * per;
  const int first_s = lane / per, first_u = lane - first_s * per;
  auto issue = [&](int st) {
    if (is < nstep && ic < nch) {
      const C* Gi = Gf + (size_t)step_col(is) * bb;
      const uint32_t dst = tc::smem_u32(ring + (size_t)st * SB);
      const int m0 = ic * KC;
      const int nseg = TRANS ? KC : rows;
      for (int sg = first_s, u = first_u; sg < nseg;) {
        if (TRANS) {  // G row m0 + sg at the CTA's columns
          const int c = row0 + u * (gb / CS);
          const bool ok = m0 + sg < b && c < row0 + rows;
          cp_async(dst + (uint32_t)(sg * rmax * CS + u * gb),
                   ok ? Gi + (size_t)(m0 + sg) * ldg + c : Gi, gb, ok);
        } else {      // the CTA's row sg at columns m0 ..
          const int c = m0 + u * (gb / CS);
          const bool ok = c < b;
          cp_async(dst + (uint32_t)(sg * PITCH + u * gb),
                   ok ? Gi + (size_t)(row0 + sg) * ldg + c : Gi, gb, ok);
        }
        sg += walk_s;
        u += walk_u;
        if (u >= per) {
          u -= per;
          ++sg;
        }
      }
      ic += W;
      if (ic >= nch) {
        ic = warp;
        ++is;
      }
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  issue(0);
  issue(1);
  int st = 0;

  // ---- coupling of unit e for the block of step s (own rows)
  const int units = rows * UPR;
  struct Unit {
    T cf[3][4];  // y offset -1, 0, 1; variable
    C in[VEC];
  };
  Unit un[EP];
  const T* coef = sizeof(T) == 8 ? reinterpret_cast<const T*>(op.coef)
                                 : reinterpret_cast<const T*>(op.coef32);
  // coefficients and input of t_s: requested early, used after the halos
  auto load_unit = [&](Unit& w, int e, int s) {
    const int r = e / UPR, j = j0 + (e - r * UPR) * VEC, m = row0 + r;
    const int i = step_col(s), iy = m / q, c = m - iy * q;
    // the column before, i - dcol, couples in.  !TRANS: L[(i, m), (i - dcol, ...)],
    // slots dx = -dcol of the row; TRANS: L[(i - dcol, r), (i, m)], rows r of the
    // points whose stencil reaches m
    const T* cb = coef + (size_t)(!TRANS ? i : s > 0 ? i - dcol : i) * b * op.S;
    const int slot = (!TRANS ? 1 - dcol : 1 + dcol) * 3;
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
      int off = 0, stride = 1;
      bool ok = s > 0;
      if (!TRANS) {
        off = m * op.S + (slot + d + 1) * q;
      } else {
        const int jy = nbr_y(iy, -d, ny, op.periodic);
        ok = ok && jy >= 0;
        off = jy * q * op.S + (slot + d + 1) * q + c;
        stride = op.S;
      }
#pragma unroll
      for (int cp = 0; cp < 4; ++cp) {
        T v = (T)0;
        if (ok && cp < q) v = cb[off + cp * stride];
        w.cf[d + 1][cp] = !TRANS && outw ? -v : v;
      }
    }
    // right-hand side: in (inward, middle), nothing (outward), the stored h
    // (adjoint outward)
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      C z = czero<C>();
      const size_t g = ((size_t)i * b + m) * k + j + v;
      if (j + v < k) {
        if (!outw || s == 0) z = in[g];
        else if (TRANS) z = h[g];
      }
      w.in[v] = z;
    }
  };
  // the middle column's: both neighbours' last inward results
  auto load_middle = [&](Unit& w, int e) {
    const int r = e / UPR, j = j0 + (e - r * UPR) * VEC, m = row0 + r;
    const int iy = m / q, c = m - iy * q;
    for (int side = 0; side < 2; ++side) {
      const int dx = side ? 1 : -1;
      const C* E = a.edge + ((size_t)side * a.F + f) * (size_t)b * k;
      for (int d = -1; d <= 1; ++d) {
        const int jy = nbr_y(iy, TRANS ? -d : d, ny, op.periodic);
        if (jy < 0) continue;
        for (int cp = 0; cp < q; ++cp) {
          const T v = TRANS ? coef[((size_t)(mid + dx) * b + jy * q + cp) * op.S +
                                   ((1 - dx) * 3 + d + 1) * q + c]
                            : coef[((size_t)mid * b + m) * op.S + ((1 + dx) * 3 + d + 1) * q + cp];
#pragma unroll
          for (int u = 0; u < VEC; ++u)
            if (j + u < k) w.in[u] = crfma(v, E[(size_t)(jy * q + cp) * k + j + u], w.in[u]);
        }
      }
    }
  };
  const uint32_t tb_a = tc::smem_u32(tb), mT_a = tc::smem_u32(&mT[0]);
  const bool mute = a.stall && blockIdx.x == 0;
  // t_s of unit e: couple and send
  auto couple_unit = [&](const Unit& w, int e, int s) {
    const int r = e / UPR, cu = e - r * UPR, j = j0 + cu * VEC, m = row0 + r;
    const int lp = r / q, i = step_col(s);
    C t[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) t[v] = w.in[v];
    if (s > 0) {
#pragma unroll
      for (int d = -1; d <= 1; ++d) {
        const C* o = ob + (size_t)((lp + 1 + (TRANS ? -d : d)) * q) * NC + cu * VEC;
#pragma unroll
        for (int cp = 0; cp < 4; ++cp) {
          if (cp >= q) break;
#pragma unroll
          for (int v = 0; v < VEC; ++v) t[v] = crfma(w.cf[d + 1][cp], o[cp * NC + v], t[v]);
        }
      }
    }
    if (TRANS && !outw) {  // h_i for the outward sweep (own rows only)
#pragma unroll
      for (int v = 0; v < VEC; ++v)
        if (j + v < k) h[((size_t)i * b + m) * k + j + v] = t[v];
    }
    if (mute) return;
    const uint32_t off = (uint32_t)(((s & 1) * bp + m) * NC + cu * VEC) * CS;
    const float4 val = *reinterpret_cast<const float4*>(t);
    for (int dst = 0; dst < CL; ++dst)
      tc::st_async16(tc::cluster_map(tb_a + off, dst), val,
                     tc::cluster_map(mT_a + (s & 1) * 8, dst));
  };
  const uint32_t t_bytes = (uint32_t)b * NC * CS;
  const bool has_prev = op.periodic || rank > 0;
  const bool has_next = op.periodic || rank + 1 < CL;
  const int prev = rank > 0 ? rank - 1 : CL - 1, next = rank + 1 < CL ? rank + 1 : 0;
  const int prev_pts = min(npt, ny - prev * npt);
  const uint32_t h_bytes = (uint32_t)((has_prev ? 1 : 0) + (has_next ? 1 : 0)) * q * NC * CS;
  const uint32_t ob_a = tc::smem_u32(ob), mH_a = tc::smem_u32(&mH[0]);

  if (tid == 0) tc::mbar_expect_tx(&mT[0], t_bytes);
  for (int e = tid; e < units; e += nthr) {
    load_unit(un[0], e, 0);
    if (outw) load_middle(un[0], e);
    couple_unit(un[0], e, 0);
  }
  const int lr = lane / LC, lc = (lane % LC) * CPL;
  bool ok = true;
  for (int s = 0; s < nstep; ++s) {
    const int i = step_col(s);
    const bool last = s + 1 == nstep;
    if (tid == 0 && !last) {
      tc::mbar_expect_tx(&mT[(s + 1) & 1], t_bytes);
      if (h_bytes) tc::mbar_expect_tx(&mH[s & 1], h_bytes);
    }
    ok = tc::cluster_wait(&mT[s & 1], (uint32_t)(s >> 1) & 1u, a.tries);
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
    // ---- product
    C acc[RPL][CPL];
#pragma unroll
    for (int u = 0; u < RPL; ++u)
#pragma unroll
      for (int v = 0; v < CPL; ++v) acc[u][v] = czero<C>();
    const C* t = tb + (size_t)(s & 1) * bp * NC + lc;
    for (int c = warp; c < nch; c += W) {
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      __syncwarp();
      const unsigned char* tile = ring + (size_t)st * SB;
      const C* tc0 = t + (size_t)c * KC * NC;
#pragma unroll 2
      for (int m = 0; m < KC; m += VEC) {
        C gv[RPL][VEC];
#pragma unroll
        for (int u = 0; u < RPL; ++u) {
          const int r = min(lr + LR * u, rmax - 1);
          if (!TRANS) {
            *reinterpret_cast<float4*>(gv[u]) =
                *reinterpret_cast<const float4*>(tile + r * PITCH + m * CS);
          } else {
#pragma unroll
            for (int v = 0; v < VEC; ++v)
              gv[u][v] = cconj(reinterpret_cast<const C*>(tile)[(m + v) * rmax + r]);
          }
        }
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          C tv[CPL];
#pragma unroll
          for (int n = 0; n < CPL; n += VEC)
            *reinterpret_cast<float4*>(&tv[n]) =
                *reinterpret_cast<const float4*>(tc0 + (size_t)(m + v) * NC + n);
#pragma unroll
          for (int u = 0; u < RPL; ++u)
#pragma unroll
            for (int n = 0; n < CPL; ++n) acc[u][n] = cfma(gv[u][v], tv[n], acc[u][n]);
        }
      }
      __syncwarp();
      issue(st);  // the slot is free: two chunks ahead
      st ^= 1;
    }
    // requests for the next block, in flight during the sum and the halos
    C xo[EP][VEC];
#pragma unroll
    for (int p = 0; p < EP; ++p) {
      const int e = tid + p * nthr;
      if (e >= units) break;
      if (!last) load_unit(un[p], e, s + 1);
      if (!TRANS && outw && s > 0) {
        const int r = e / UPR, j = j0 + (e - r * UPR) * VEC;
#pragma unroll
        for (int v = 0; v < VEC; ++v)
          xo[p][v] = j + v < k ? x[((size_t)i * b + row0 + r) * k + j + v] : czero<C>();
      }
    }
#pragma unroll
    for (int u = 0; u < RPL; ++u) {
      const int r = lr + LR * u;
      if (r < rows) {
        C* dst = red + ((size_t)warp * rmax + r) * NC + lc;
#pragma unroll
        for (int n = 0; n < CPL; n += VEC)
          *reinterpret_cast<float4*>(dst + n) = *reinterpret_cast<const float4*>(&acc[u][n]);
      }
    }
    __syncthreads();
    // ---- sum, store, halos
#pragma unroll
    for (int p = 0; p < EP; ++p) {
      const int e = tid + p * nthr;
      if (e >= units) break;
      const int r = e / UPR, cu = e - r * UPR, j = j0 + cu * VEC;
      C o[VEC];
#pragma unroll
      for (int v = 0; v < VEC; ++v) o[v] = czero<C>();
      for (int w = 0; w < W; ++w) {
        C pv[VEC];
        *reinterpret_cast<float4*>(pv) =
            *reinterpret_cast<const float4*>(red + ((size_t)w * rmax + r) * NC + cu * VEC);
#pragma unroll
        for (int v = 0; v < VEC; ++v) o[v] = cadd(o[v], pv[v]);
      }
      if (!TRANS && outw && s > 0) {
#pragma unroll
        for (int v = 0; v < VEC; ++v) o[v] = csub(xo[p][v], o[v]);
      }
      // (the middle column's result is half 0's to store)
      if (outw ? s > 0 || half == 0 : !TRANS) {
#pragma unroll
        for (int v = 0; v < VEC; ++v)
          if (j + v < k) x[((size_t)i * b + row0 + r) * k + j + v] = o[v];
      }
      if (!outw && last) {
        C* E = a.edge + ((size_t)half * a.F + f) * (size_t)b * k;
#pragma unroll
        for (int v = 0; v < VEC; ++v)
          if (j + v < k) E[(size_t)(row0 + r) * k + j + v] = o[v];
      }
      const float4 val = *reinterpret_cast<const float4*>(o);
      *reinterpret_cast<float4*>(ob + (size_t)(q + r) * NC + cu * VEC) = val;
      if (!last) {
        const uint32_t mh = mH_a + (s & 1) * 8;
        if (has_prev && r < q)  // first point: the last halo of the CTA before
          tc::st_async16(tc::cluster_map(ob_a + (uint32_t)((((prev_pts + 1) * q + r) * NC + cu * VEC) * CS),
                                         prev),
                         val, tc::cluster_map(mh, prev));
        if (has_next && r >= rows - q)  // last point: the first halo of the next CTA
          tc::st_async16(tc::cluster_map(ob_a + (uint32_t)(((r - (rows - q)) * NC + cu * VEC) * CS), next),
                         val, tc::cluster_map(mh, next));
      }
    }
    if (last) break;
    if (h_bytes) ok = tc::cluster_wait(&mH[s & 1], (uint32_t)(s >> 1) & 1u, a.tries);
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
    // ---- couple
#pragma unroll
    for (int p = 0; p < EP; ++p) {
      const int e = tid + p * nthr;
      if (e < units) couple_unit(un[p], e, s + 1);
    }
  }
  if (!ok && tid == 0) atomicExch(a.err, 1);
  if (!ok) tc::cluster_settle();
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  tc::cluster_sync();  // no CTA leaves while another may still send to it
}

// ------------------------------------------------------------------- plan
struct Plan {
  int kc, CL, npt, W, rpl;
  double us;       // modelled time of the solve
  double form_us;  // the same by form_step_us
};

// Microseconds of a column step: the chain of a step plus a part that grows
// with the block and the lane tile.  Measured (two problems, FP32, CPL = 2):
// blocks of 192 rows 2.9 us with clusters of eight (RPL 2), 3.6 of four (RPL 3),
// 6.0 of two (RPL 6); 384 rows 5.8 and 10.7; 768 rows 18 to 22; CPL = 4 takes
// 3.6 / 4.9 / 8.3 at 192 rows and 7.9 at 384 (RPL 3).  FP64, a lane tile of
// one row and column: 10.3 us at 192 rows (arithmetic).
inline double step_us(bool dp, int b, int rpl, int cpl) {
  if (dp) return 3.0 + 0.037 * b * rpl * cpl;
  const double two[10] = {0, 5, 6.8, 11, 15, 24, 24, 32, 40, 46};
  const double four[10] = {0, 6, 11, 17, 24, 36, 36, 60, 60, 70};
  return 1.6 + 1e-3 * b * (cpl == 2 ? two[rpl] : four[rpl]);
}

// The FP32 step beside the tensor-core form's (sweep.cu), for the choice between the
// two: fitted to unrefined solves of 96 columns of 48 to 768 rows, 1 to 64 right-hand
// sides and 1 to 128 problems in both forms.  Odd blocks take 8-byte copies.
inline double form_step_us(int b, int rpl, int cpl) {
  const double two[10] = {0, 9.7, 10.2, 13.4, 17.4, 25.6, 27.6, 42.7, 52.6, 70.2};
  const double four[10] = {0, 8.8, 15.6, 18.6, 29.4, 35.9, 37.0, 43.6, 44, 70};
  return 0.94 + 1e-3 * b * (cpl == 2 ? two[rpl] : four[rpl]) * (b % 2 ? 1.33 : 1.0);
}

// Column groups and cluster size with the least modelled time: waves of
// clusters x steps.  us < 0 when the block does not fit.
template <typename T>
Plan make_plan(const OpDev& d, int Fa, int k, int trans) {
  constexpr bool DP = sizeof(T) == 8;
  constexpr int KC = 64 / sizeof(C_t<T>);
  const int kcs[3] = {DP ? 1 : 4, DP ? 2 : 8, 4};
  Plan best{0, 0, 0, 0, 0, -1.0, -1.0};
  const int lr = DP ? 32 : 16, rplmax = DP ? 5 : 9;
  for (int ki = 0; ki < (DP ? 3 : 2); ++ki) {
    const int kc = kcs[ki], ng = (k + kc - 1) / kc, cpl = DP ? kc : kc / 2;
    for (int cl0 = CLMAX; cl0 >= 1; --cl0) {
      const int npt = (d.ny + cl0 - 1) / cl0, CL = (d.ny + npt - 1) / npt;
      if (CL != cl0) continue;
      const int rmax = npt * d.q, rpl = (rmax + lr - 1) / lr;
      if (rpl > rplmax) continue;
      const int nch = (d.b + KC - 1) / KC;
      const int upr = kc * (int)sizeof(C_t<T>) / 16, units = rmax * upr;
      int W = 0;
      const int wmax = !DP && cpl * (rpl == 5 ? 6 : rpl) >= 20 ? 8 : MAXW;
      for (int w = std::min(wmax, nch); w >= 1; --w) {
        const int rounds = (nch + w - 1) / w, wb = (nch + rounds - 1) / rounds;
        const size_t sm = trans ? smem_bytes<T, true>(d.b, rmax, d.q, kc, wb)
                                : smem_bytes<T, false>(d.b, rmax, d.q, kc, wb);
        if (sm <= SMEM_CAP && units <= 2 * 32 * wb) {
          W = wb;
          break;
        }
      }
      if (W == 0) continue;
      const int slots = cluster_slots(d.device, CL);
      const int waves = (int)((2L * Fa * ng + slots - 1) / slots);
      const double us = waves * (d.nx + 1.0) * step_us(DP, d.b, rpl, cpl);
      if (best.us < 0 || us < best.us)
        best = Plan{kc, CL, npt, W, rpl, us,
                    DP ? us : waves * (d.nx + 1.0) * form_step_us(d.b, rpl, cpl)};
    }
  }
  return best;
}

template <typename T, bool TRANS, int LC, int CPL, int RPL, bool PITCHED = !TRANS>
rr_status launch(const Args<T>& a, int clusters, size_t smem, int W, cudaStream_t st) {
  if constexpr (sizeof(T) == 4 && !PITCHED)
    if (a.ldg != a.op.b) return launch<T, TRANS, LC, CPL, RPL, true>(a, clusters, smem, W, st);
  RR_TRY((smem_opt_in<sweep_cl_kernel<T, TRANS, LC, CPL, RPL, PITCHED>>(SMEM_CAP)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.CL * clusters), 1, 1);
  cfg.blockDim = dim3((unsigned)(32 * W), 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = a.CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  RR_CUDA(cudaLaunchKernelEx(&cfg, sweep_cl_kernel<T, TRANS, LC, CPL, RPL, PITCHED>, a));
  return RR_OK;
}

template <typename T, bool TRANS, int LC, int CPL>
rr_status launch_rpl(const Args<T>& a, int rpl, int clusters, size_t smem, int W, cudaStream_t st) {
  switch (rpl) {
    case 1: return launch<T, TRANS, LC, CPL, 1>(a, clusters, smem, W, st);
    case 2: return launch<T, TRANS, LC, CPL, 2>(a, clusters, smem, W, st);
    case 3: return launch<T, TRANS, LC, CPL, 3>(a, clusters, smem, W, st);
    case 4: return launch<T, TRANS, LC, CPL, 4>(a, clusters, smem, W, st);
    default: break;
  }
  if constexpr (sizeof(T) == 4) {
    if (rpl <= 6) return launch<T, TRANS, LC, CPL, 6>(a, clusters, smem, W, st);
    if (rpl <= 8) return launch<T, TRANS, LC, CPL, 8>(a, clusters, smem, W, st);
    return launch<T, TRANS, LC, CPL, 9>(a, clusters, smem, W, st);
  } else {
    return launch<T, TRANS, LC, CPL, 5>(a, clusters, smem, W, st);
  }
}

template <typename T, bool TRANS>
rr_status launch_plan(rr_factors* fa, const Plan& p, int k, const void* in, void* x, void* h) {
  const OpDev& d = fa->op->d;
  Args<T> a;
  a.op = view(d);
  a.G = reinterpret_cast<const C_t<T>*>(fa->G);
  a.ldg = fa->ldg;
  a.gstride = (size_t)d.nx * d.b * fa->ldg;
  a.in = reinterpret_cast<const C_t<T>*>(in);
  a.x = reinterpret_cast<C_t<T>*>(x);
  a.h = reinterpret_cast<C_t<T>*>(h);
  a.edge = reinterpret_cast<C_t<T>*>(fa->Tbuf);
  a.F = fa->F;
  a.k = k;
  a.ng = (k + p.kc - 1) / p.kc;
  a.npt = p.npt;
  a.CL = p.CL;
  a.amap = fa->amap;
  a.err = fa->err;
  a.tries = wait_tries();
  const int clusters = 2 * active_count(fa) * a.ng;
  const size_t smem = smem_bytes<T, TRANS>(d.b, p.npt * d.q, d.q, p.kc, p.W);
  cudaStream_t st = fa->stream;
  for (a.out = 0; a.out < 2; ++a.out) {
    a.stall = take_stall();
    prof_begin(PROF_SWEEP, st);
    rr_status s;
    if constexpr (sizeof(T) == 8) {
      if (p.kc == 1) s = launch_rpl<T, TRANS, 1, 1>(a, p.rpl, clusters, smem, p.W, st);
      else if (p.kc == 2) s = launch_rpl<T, TRANS, 1, 2>(a, p.rpl, clusters, smem, p.W, st);
      else s = launch_rpl<T, TRANS, 1, 4>(a, p.rpl, clusters, smem, p.W, st);
    } else {
      if (p.kc == 4) s = launch_rpl<T, TRANS, 2, 2>(a, p.rpl, clusters, smem, p.W, st);
      else s = launch_rpl<T, TRANS, 2, 4>(a, p.rpl, clusters, smem, p.W, st);
    }
    prof_end(PROF_SWEEP, st);
    if (s != RR_OK) return s;
  }
  return RR_OK;
}

}  // namespace sweepcl
