// Block forward/back sweeps with the stored factors: the linear solves of
// Algorithm 1 (Sec. II.B, second, fourth and sixth steps), all reusing the
// one factorisation of s I - L (Sec. III.A).
//
// With G_i = S_i^{-1}, C_i = -L_{i,i+1} (at most 3q entries per row) and the
// factorisation run from both ends to the middle column m (factor.cu), a solve goes
// inwards in both halves, through the middle, and outwards (written for the left
// half, i < m; the right one is the mirror image):
// Normal solve (s I - L) y = f:
//   inward   z_0 = G_0 f_0,      z_i = G_i (f_i + L_{i,i-1} z_{i-1})
//   middle   y_m = G_m (f_m + L_{m,m-1} z_{m-1} + L_{m,m+1} z_{m+1})
//   outward  y_i = z_i - G_i (C_i y_{i+1})
// Adjoint solve (s I - L)^H w = g:
//   inward   h_0 = g_0,          h_{i+1} = g_{i+1} - C_i^H (G_i^H h_i)
//   middle   h_m from both sides, w_m = G_m^H h_m
//   outward  w_i = G_i^H (h_i + L_{i+1,i}^T w_{i+1})
// The chain is nx + 1 products instead of the 2 nx - 1 of a sweep from one end.
// Only G_i is stored.  Two forms: two launches per solve with a cluster of CTAs
// per problem and half (sweep_cl.cuh), or, for large blocks and batches, two
// launches per pair of streamwise columns for all problems of the batch: the dense
// (b x b) x (b x k) product on the tensor cores, its contraction split over CTAs
// (sweep_tc2_kernel), or for RR_FP32_SIMT on the CUDA cores (sweep_cc_kernel), and
// the sum of the partial blocks with the sparse coupling that forms the next
// column's right-hand side (sweep_couple_kernel).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include <cuda.h>

#include "rr_internal.cuh"
#include "tc.cuh"

namespace {

// A step of the tensor-core sweeps: for half 0 and, when nh == 2, half 1 (the
// mirror image), a column of the inward sweep, the middle one, or one of the
// outward sweep.  Half h has its `own` columns h == 0: 0 .. mid - 1,
// h == 1: nx - 1 .. mid + 1.
enum { SW_IN = 0, SW_MID = 1, SW_OUT = 2 };
struct SweepStep {
  int phase, t, nh;  // t: columns from the end (SW_IN) or from the middle (SW_OUT)
};
__host__ __device__ __forceinline__ int half_cols(int half, int nx) {
  return half ? nx - 1 - twist_mid(nx) : twist_mid(nx);
}
__host__ __device__ __forceinline__ int step_col(const SweepStep& s, int half, int nx) {
  if (s.phase == SW_IN) return half ? nx - 1 - s.t : s.t;
  return half ? twist_mid(nx) + s.t : twist_mid(nx) - s.t;
}

// Result of a step and right-hand side of the next.  Per problem, half and tile of
// CPL_Y grid points: o = the sum of the KS partial products in a fixed order
// (outward: z_i minus it), of the tile's rows and of one point on either
// side (recomputed, not exchanged), kept in shared memory; then, with i the
// column before of the half,
//   t = in + L_{i',i} o (inward), -L_{i',i} o (outward),
//   t = in + L_{i,i'}^T o (adjoint inward, stored as h too),
//   t = h + L_{i,i'}^T o (adjoint outward)
// for the next column i'.  z goes to zh in the inward sweep, so the outward one's
// results (x) never overwrite a value a neighbouring tile still needs.
// One grid dimension: the others hold 65,535 problems, not two halves of them, and with
// the halves in a third one an adjoint step of 384 rows took 4 % longer.
// (part is not __restrict__: the product writes it while this kernel already runs,
// until grid_wait, so no load of it may go through the read-only path or move up.)
// Bound: L2 latency (the partials were just written), so the coefficients and
// inputs of the coupling are requested before the partials are summed, and a
// thread has one element (two columns) of each phase at k <= 32.
// V is a unit of a row: two columns (float4) where k is even, else one (float2).
// (Odd k on the cluster form instead, 768 rows, 31 columns, 16 problems, 16 columns of
// the grid: 10.2 ms forward and 5.8 adjoint; here 1.9 both.)
constexpr int CPL_Y = 4, CPL_MAXTHR = 512;
inline int couple_threads(int q, int units) {
  return std::min(CPL_MAXTHR, ((CPL_Y + 2) * q * units + 31) & ~31);
}
__device__ __forceinline__ float4 vadd(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float2 vadd(float2 a, float2 b) {
  return make_float2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ float4 vsub(float4 a, float4 b) {
  return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float2 vsub(float2 a, float2 b) {
  return make_float2(a.x - b.x, a.y - b.y);
}
__device__ __forceinline__ float4 vfma(float a, float4 u, float4 t) {
  return make_float4(fmaf(a, u.x, t.x), fmaf(a, u.y, t.y), fmaf(a, u.z, t.z), fmaf(a, u.w, t.w));
}
__device__ __forceinline__ float2 vfma(float a, float2 u, float2 t) {
  return make_float2(fmaf(a, u.x, t.x), fmaf(a, u.y, t.y));
}

template <bool TRANS, typename V>
__global__ void __launch_bounds__(CPL_MAXTHR)
sweep_couple_kernel(OpView op, SweepStep s, int F, int Fa, int k, int KS,
                    const float2* part, const float2* __restrict__ in, float2* x, float2* zh,
                    float2* __restrict__ tbuf, const int* __restrict__ amap) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int VW = sizeof(V) / sizeof(float2);  // columns of a unit
  V* o = reinterpret_cast<V*>(smem_raw);           // [(CPL_Y + 2) q][P]
  const int b = op.b, q = op.q, ny = op.ny, nx = op.nx, P = k / VW;
  const int nty = (ny + CPL_Y - 1) / CPL_Y, p = blockIdx.x / nty;
  const int half = p >= Fa, f = active_problem(amap, half ? p - Fa : p);
  const int y0 = (blockIdx.x - p * nty) * CPL_Y, npt = min(CPL_Y, ny - y0);
  const size_t NK = (size_t)op.n * k, total = (size_t)s.nh * F * b * k;
  const int i = step_col(s, half, nx);
  const bool inw = s.phase == SW_IN, outw = s.phase == SW_OUT;
  const int dcol = (half != 0) == inw ? -1 : 1;  // to the next column
  // (the middle's right-hand side needs both halves: sweep_middle_kernel)
  const bool last = s.phase != SW_MID && s.t + (inw ? 1 : 0) == half_cols(half, nx);
  const int i1 = last ? i : i + dcol;
  // L[(i1, .), (i, .)]: slots dx = -dcol of the rows of i1; transposed, dx = dcol of
  // those of i
  const float* cb = op.coef32 + (size_t)(!TRANS ? i1 : i) * b * op.S;
  const int slot = (!TRANS ? 1 - dcol : 1 + dcol) * 3;
  // (h of the end columns is the input itself: no step stores it)
  const V* src = reinterpret_cast<const V*>(
      (inw || i1 == 0 || i1 == nx - 1 ? in : zh) + (size_t)f * NK + (size_t)i1 * b * k);
  struct Term {
    float cf[3][4];
    V t;
  };
  auto load_term = [&](Term& w, int e) {
    const int lrow = e / P, jp = e - lrow * P;
    const int lp = lrow / q, c = lrow - lp * q, iy = y0 + lp, m = iy * q + c;
    w.t = TRANS || inw ? src[m * P + jp] : V{};
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
      int off, stride = 1;
      bool ok = true;
      if (!TRANS) {
        off = m * op.S + (slot + d + 1) * q;
      } else {
        const int jy = nbr_y(iy, -d, ny, op.periodic);
        ok = jy >= 0;
        off = jy * q * op.S + (slot + d + 1) * q + c;
        stride = op.S;
      }
#pragma unroll
      for (int cp = 0; cp < 4; ++cp) {
        const float v = ok && cp < q ? cb[off + cp * stride] : 0.f;
        w.cf[d + 1][cp] = !TRANS && !inw ? -v : v;
      }
    }
  };
  Term w;
  const int nown = npt * q * P;
  if (!last && (int)threadIdx.x < nown) load_term(w, threadIdx.x);
  // (the middle's partials are the first half's)
  const size_t pidx = s.phase == SW_MID ? f : (size_t)half * F + f;
  tc::grid_wait();  // (above: what kernels before the product's wrote, and constants)
  tc::grid_trigger();
  const V* pf = reinterpret_cast<const V*>(part + pidx * b * k);
  V* xi = reinterpret_cast<V*>(x + (size_t)f * NK + (size_t)i * b * k);
  V* zi = reinterpret_cast<V*>(zh + (size_t)f * NK + (size_t)i * b * k);
  for (int e = threadIdx.x; e < (npt + 2) * q * P; e += blockDim.x) {
    const int lrow = e / P, jp = e - lrow * P;
    const int lp = lrow / q, c = lrow - lp * q;
    int y = y0 - 1 + lp;
    const bool own = lp >= 1 && lp <= npt;
    if (op.periodic) y = (y + ny) % ny;
    V v = V{};
    if (y >= 0 && y < ny) {
      const int e0 = (y * q + c) * P + jp;
      V z = v;
      if (!TRANS && outw) z = zi[e0];
#pragma unroll 4
      for (int t = 0; t < KS; ++t) v = vadd(v, pf[(size_t)t * (total / VW) + e0]);
      if (!TRANS && outw) v = vsub(z, v);
      if (own) {
        if (!TRANS && inw) zi[e0] = v;
        // x; the adjoint's last inward result waits there for the middle
        if (outw || (s.phase == SW_MID && half == 0) || (TRANS && inw && last)) xi[e0] = v;
      }
    }
    o[e] = v;
  }
  if (last) return;
  __syncthreads();
  V* h = reinterpret_cast<V*>(zh + (size_t)f * NK + (size_t)i1 * b * k);
  V* tf = reinterpret_cast<V*>(tbuf + ((size_t)half * F + f) * b * k);
  for (int e = threadIdx.x; e < nown; e += blockDim.x) {
    if (e != (int)threadIdx.x) load_term(w, e);
    const int lrow = e / P, jp = e - lrow * P;
    const int lp = lrow / q, m = (y0 + lp) * q + lrow - lp * q;
    V t = w.t;
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
      const V* ov = o + ((lp + 1 + (TRANS ? -d : d)) * q) * P + jp;
#pragma unroll
      for (int cp = 0; cp < 4; ++cp) {
        if (cp >= q) break;
        t = vfma(w.cf[d + 1][cp], ov[cp * P], t);
      }
    }
    if (TRANS && inw) h[m * P + jp] = t;
    tf[m * P + jp] = t;
  }
}

// Right-hand side of the middle column: in + the couplings of both halves' last
// inward results (z in zh, adjoint p in x), one thread per row and unit of columns;
// a few microseconds of L2 latency, once per solve.
template <bool TRANS, typename V>
__global__ void sweep_middle_kernel(OpView op, int k, const float2* __restrict__ in,
                                    const float2* __restrict__ src, float2* __restrict__ tbuf,
                                    const int* __restrict__ amap) {
  const int b = op.b, q = op.q, mid = twist_mid(op.nx);
  const int P = k / (int)(sizeof(V) / sizeof(float2));
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= b * P) return;
  const int f = active_problem(amap, blockIdx.y);
  const int m = e / P, jp = e - m * P, iy = m / q, c = m - iy * q;
  const size_t NK = (size_t)op.n * k;
  V t = reinterpret_cast<const V*>(in + f * NK + (size_t)mid * b * k)[e];
  for (int dx = -1; dx <= 1; dx += 2) {
    const V* o = reinterpret_cast<const V*>(src + f * NK + (size_t)(mid + dx) * b * k);
    const float* cb = op.coef32 + (size_t)(TRANS ? mid + dx : mid) * b * op.S;
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
      const int jy = nbr_y(iy, TRANS ? -d : d, op.ny, op.periodic);
      if (jy < 0) continue;
#pragma unroll
      for (int cp = 0; cp < 4; ++cp) {
        if (cp >= q) break;
        const int r = jy * q + cp;
        const float a = TRANS ? cb[r * op.S + ((1 - dx) * 3 + d + 1) * q + c]
                              : cb[m * op.S + ((1 + dx) * 3 + d + 1) * q + cp];
        t = vfma(a, o[r * P + jp], t);
      }
    }
  }
  reinterpret_cast<V*>(tbuf + (size_t)f * b * k)[e] = t;
}

// ---------------------------------------------------------------------------
// Tensor-core sweep step fed by TMA, with the contraction split over KS CTAs.
//
// The complex product acc = op(G) t (128 rows of G per item, all k columns) is
// one real GEMM: the interleaved rows of op(G) are the K-major A operand and the
// right-hand side is expanded to the real matrix B~ with rows (Re t, -Im t, ...)
// and (Im t, Re t, ...), so D = A B~^T holds (Re, Im) pairs.  FP32 accuracy
// comes from splitting every operand (TF32 part and remainder, or BF16
// pieces).  Chunks of 16 complex columns: the raw 128 x 16 complex tiles of G_i
// (or of G_i^H) arrive by 3-D TMA (one tensor map over all factors, coordinate 2
// = problem * nx + column), and the matching 16 right-hand-side rows by a 1-D
// bulk copy, into a ring of tc2_stages guarded by mbarriers.  The pieces of A go
// straight to TMEM (a thread has one row of the tile and half of its columns),
// those of B~ to shared memory, into one of tc2_bufs operand buffers.  Roles:
// two groups of eight warps, each splitting every other chunk (splitting one is
// a chain of latencies, about 1000 cycles, with 420 cycles of MMAs); one thread
// that issues the MMAs of a chunk when its group has arrived on conv_bar; one
// that refills a stage when its group has read it (free_bar).  The launches of a
// solve follow each other by programmatic dependence: set-up and the first tiles
// of G do not wait for the coupling before.
// Bound: splitting and MMAs, which share shared memory (with neither, the same
// loop takes the time of the tiles from memory).  Measured, 12 blocks of 768 x 768
// by 32 columns: 17 us a launch, 23 with both operands staged in shared memory and
// one barrier a chunk, 8 for G's bytes; the step with its coupling and gaps 20 us
// instead of 27 before the dependent launches.  32 blocks: 34 instead of 59.
// CTA (row tile, part) handles the chunks [part*cpp, (part+1)*cpp) and writes a
// partial 128 x k block; sweep_couple_kernel adds the KS partials in a fixed
// order.  All waits are bounded (flag *err).
constexpr int TC_RT = 128;                                // rows of an item
constexpr uint32_t TC_LBO = 128;
constexpr uint32_t TC_WAIT_TRIES = 1u << 22;
constexpr int TC2_KC = 16;                                // complex columns per chunk
constexpr int TC2_MAXSTAGES = 8;
constexpr int TC2_MAXBUFS = 4;
__host__ __device__ constexpr int tc2_stages(int kp) { return kp > 32 ? 6 : TC2_MAXSTAGES; }
constexpr uint32_t TC2_TILE_BYTES = TC_RT * TC2_KC * 8;   // 16 KB raw tile

__host__ __device__ constexpr uint32_t tc2_stage_bytes(int kp) {
  return (TC2_TILE_BYTES + (uint32_t)TC2_KC * kp * 8 + 1023u) & ~1023u;
}
// one operand piece of a chunk (32 reals of K): A, TMEM columns of 128 rows; B~,
// shared memory of 2 kp rows
template <int SPLIT>
__host__ __device__ constexpr uint32_t tc2_a_cols() { return 8u * tc::SplitCfg<SPLIT>::ESZ; }
template <int SPLIT>
__host__ __device__ constexpr uint32_t tc2_b_piece(int kp) {
  return (uint32_t)(2 * kp / 8) * tc::sbo32<SPLIT>();
}
template <int SPLIT>
__host__ __device__ constexpr uint32_t tc2_buf_bytes(int kp) {
  return tc::SplitCfg<SPLIT>::PIECES * tc2_b_piece<SPLIT>(kp);
}
// TMEM: accumulator sets, then the buffers of A pieces.  A set sums the piece
// products by order (x3: hi.hi | hi.lo + lo.hi; x6: three orders), N = 2 kp
// columns each; consecutive K steps go to different sets, because the tensor
// core's accumulation rounds towards zero (one set instead of two at 32 columns:
// 35 % more error in a solve).  The small orders need no such care.
template <int SPLIT>
__host__ __device__ constexpr int tc2_orders() { return SPLIT == tc::SPLIT_BF16X6 ? 3 : 2; }
template <int SPLIT>
__host__ __device__ constexpr int tc2_sets(int kp) {
  const int fit = 256 / (tc2_orders<SPLIT>() * 2 * kp);
  return fit < 1 ? 1 : fit < tc::ksteps32<SPLIT>() ? fit : tc::ksteps32<SPLIT>();
}
// Where one set fits (64 columns), a second accumulator of hi.hi alone takes every other
// K step of the TF32 split (384 rows, 24 problems: unrefined residual 1.0e-5 instead
// of 8.7e-6 without it, 4.7e-5 and 3.8e-5 adjoint; 0 to 3 % of a solve).  BF16x3's
// errors are its products'.
template <int SPLIT>
__host__ __device__ constexpr int tc2_extra(int kp) {
  return SPLIT == tc::SPLIT_TF32X3 && tc2_sets<SPLIT>(kp) == 1 ? 1 : 0;
}
template <int SPLIT>
__host__ __device__ constexpr uint32_t tc2_acc_cols(int kp) {
  return (uint32_t)((tc2_sets<SPLIT>(kp) * tc2_orders<SPLIT>() + tc2_extra<SPLIT>(kp)) * 2 * kp +
                    31) &
         ~31u;
}
// operand buffers: two for each group of warps where shared memory has the room
__host__ __device__ constexpr int tc2_bufs(int kp) { return kp > 32 ? 2 : TC2_MAXBUFS; }
template <int SPLIT>
__host__ __device__ constexpr uint32_t tc2_tmem_cols(int kp) {
  return tc2_acc_cols<SPLIT>(kp) +
         tc2_bufs(kp) * tc::SplitCfg<SPLIT>::PIECES * tc2_a_cols<SPLIT>();
}
static_assert(tc2_tmem_cols<tc::SPLIT_TF32X3>(32) <= 512 &&
                  tc2_tmem_cols<tc::SPLIT_TF32X3>(64) <= 512 &&
                  tc2_tmem_cols<tc::SPLIT_TF32X3>(16) <= 512 &&
                  tc2_tmem_cols<tc::SPLIT_BF16X3>(64) <= 512 &&
                  tc2_tmem_cols<tc::SPLIT_BF16X6>(32) <= 512,
              "tensor memory of a CTA");
template <int SPLIT>
__host__ __device__ constexpr size_t tc2_smem_bytes(int kp) {
  return tc2_bufs(kp) * (size_t)tc2_buf_bytes<SPLIT>(kp) +
         (size_t)tc2_stages(kp) * tc2_stage_bytes(kp);
}

__device__ __forceinline__ bool tc_poll(uint64_t* bar, uint32_t parity, uint32_t tries) {
  return tc::mbar_wait(bar, parity, tries);
}

constexpr int TC2_CONV = 512;                 // converter threads (warps 0-15)
constexpr int TC2_GROUP = TC2_CONV / 2;       // threads of a group
constexpr int TC2_THREADS = TC2_CONV + 64;    // + warp 16, issues the MMAs, and 17, the copies

// (WIDE: more than 32 columns)
template <bool TRANS, int SPLIT, bool WIDE>
__global__ void __launch_bounds__(TC2_THREADS, 1)
sweep_tc2_kernel(const __grid_constant__ CUtensorMap tmap, int b, int k, int kp, SweepStep step,
                 int nx, int nrt, int KS, int cpp, const float2* rhs, size_t rstride,
                 size_t hstride, float2* __restrict__ part, int F, int Fa, const int* __restrict__ amap, int* err,
                 uint32_t tries, int stall) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t full_bar[TC2_MAXSTAGES], free_bar[TC2_MAXSTAGES];  // raw stage in, read
  __shared__ uint64_t conv_bar[TC2_MAXBUFS], mma_bar[TC2_MAXBUFS];     // buffer split, used
  __shared__ uint64_t item_bar, acc_bar;                               // accumulator done, read
  __shared__ uint32_t tmem_base;
  __shared__ int sfail;
  constexpr int PIECES = tc::SplitCfg<SPLIT>::PIECES;
  constexpr bool X6 = SPLIT == tc::SPLIT_BF16X6;
  const int N = 2 * kp;
  constexpr uint32_t AC = tc2_a_cols<SPLIT>();
  const uint32_t bt_bytes = tc2_b_piece<SPLIT>(kp);
  const uint32_t buf_bytes = tc2_buf_bytes<SPLIT>(kp);  // pieces of B~ of one chunk
  unsigned char* ops = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int stages = tc2_stages(kp), NB = tc2_bufs(kp), nbs = NB == 4 ? 2 : 1;
  unsigned char* raw = ops + NB * buf_bytes;  // stages, 1 KB aligned
  const uint32_t stage_bytes = tc2_stage_bytes(kp);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool ctrl = (tid == TC2_CONV);       // the one thread that feeds the tensor core
  const bool prod = (tid == TC2_CONV + 32);  // the one that feeds TMA
  const int nch = (b + TC2_KC - 1) / TC2_KC;
  const int nitems = nrt * KS * Fa * step.nh;  // over the active problems of both halves
  const int my_items = nitems > (int)blockIdx.x
                           ? (nitems - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x
                           : 0;
  // x3 splits, per K step two MMAs: A_hi x [B_hi | B_lo] into [hi.hi | cross] and
  // A_lo x B_hi into cross.  BF16 x6 (up to 32 columns), three: p0 x [q0 | q1 | q2],
  // p1 x [q0 | q1], p2 x q0.
  constexpr int ORDERS = tc2_orders<SPLIT>();
  const int SETS = WIDE ? 1 : tc2_sets<SPLIT>(kp);
  constexpr int EXTRA = WIDE ? tc2_extra<SPLIT>(64) : 0;
  const uint32_t set_cols = (uint32_t)(ORDERS * N);
  const uint32_t ncols = tc2_tmem_cols<SPLIT>(kp) <= 256 ? 256u : 512u;
  // work item t of this CTA -> (half, problem, row tile, contraction part)
  auto item = [&](int t, int& half, int& f, int& rt, int& ks) {
    const int it = (int)blockIdx.x + t * (int)gridDim.x;
    rt = it % nrt;
    ks = (it / nrt) % KS;
    const int p = it / (nrt * KS);
    half = p >= Fa;
    f = active_problem(amap, half ? p - Fa : p);
  };
  auto item_len = [&](int ks) { return min(nch, ks * cpp + cpp) - ks * cpp; };

  if (warp == 0) tc::tmem_alloc(&tmem_base, ncols);
  if (tid == 0) {
    for (int s = 0; s < stages; ++s) {
      tc::mbar_init(&full_bar[s], 1);
      tc::mbar_init(&free_bar[s], TC2_GROUP / 32);
    }
    for (int q = 0; q < NB; ++q) {
      tc::mbar_init(&conv_bar[q], TC2_GROUP / 32);
      tc::mbar_init(&mma_bar[q], 1);
    }
    tc::mbar_init(&item_bar, 1);
    tc::mbar_init(&acc_bar, TC2_CONV / 32);
    sfail = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base;
  const uint32_t abuf = tmem + tc2_acc_cols<SPLIT>(kp);

  // the stream of chunks of all this CTA's items.  With
  // stall set (a diagnostic of the bounded waits) the first CTA issues
  // nothing at all, so its first wait runs out with no copy or MMA in flight.
  const bool stalled = stall && blockIdx.x == 0;
  int p_item = 0, p_lc = 0, issued = 0, p_h = 0, p_f = 0, p_rt = 0, p_ks = 0, p_len = 0, p_s = 0;
  int committed = 0;  // chunks whose MMAs this thread has committed
  if (prod && my_items > 0) {
    item(0, p_h, p_f, p_rt, p_ks);
    p_len = item_len(p_ks);
  }
  struct Rhs {
    unsigned char* dst;
    const float2* src;
    uint32_t bytes;
    uint64_t* bar;
  };
  // the tile of the next chunk; its right-hand side is left to the caller
  auto issue_tile = [&]() {
    Rhs w{nullptr, nullptr, 0, nullptr};
    if (stalled || p_item >= my_items) return w;
    const int m0 = (p_ks * cpp + p_lc) * TC2_KC;
    const int s = p_s;
    if (++p_s == stages) p_s = 0;
    // an odd block and an odd k put every other right-hand side off 16 bytes: the
    // copy starts an element early and ends on 16 bytes (inside the workspace)
    const size_t e0 = p_h * hstride + p_f * rstride + (size_t)m0 * k;
    const int off = (int)(e0 & 1);
    const uint32_t rhs_bytes = (uint32_t)((min(TC2_KC, b - m0) * k + off) * 8 + 15) & ~15u;
    unsigned char* st = raw + s * stage_bytes;
    const int zblk = p_f * nx + step_col(step, p_h, nx);
    tc::mbar_expect_tx(&full_bar[s], TC2_TILE_BYTES + rhs_bytes);
    if (!TRANS) tc::tma_load_3d(st, &tmap, 2 * m0, p_rt * TC_RT, zblk, &full_bar[s]);
    else tc::tma_load_3d(st, &tmap, 2 * p_rt * TC_RT, m0, zblk, &full_bar[s]);
    w = Rhs{st + TC2_TILE_BYTES, rhs + e0 - off, rhs_bytes, &full_bar[s]};
    ++issued;
    if (++p_lc == p_len) {
      p_lc = 0;
      if (++p_item < my_items) {
        item(p_item, p_h, p_f, p_rt, p_ks);
        p_len = item_len(p_ks);
      }
    }
    return w;
  };
  auto issue_next = [&]() {
    const Rhs w = issue_tile();
    if (w.bytes) tc::bulk_load(w.dst, w.src, w.bytes, w.bar);
  };
  if (prod) {
    Rhs first[TC2_MAXSTAGES];
#pragma unroll
    for (int q = 0; q < TC2_MAXSTAGES; ++q)
      first[q] = q < stages ? issue_tile() : Rhs{nullptr, nullptr, 0, nullptr};
    tc::grid_wait();
    tc::grid_trigger();
#pragma unroll
    for (int q = 0; q < TC2_MAXSTAGES; ++q)
      if (first[q].bytes) tc::bulk_load(first[q].dst, first[q].src, first[q].bytes, first[q].bar);
  }
  // operand addresses of both buffers; a K step (32 bytes) advances 8 TMEM
  // columns of A and 256 bytes of B~
  constexpr uint32_t SBO = tc::sbo32<SPLIT>();
  auto idesc = [](int n) {
    return SPLIT == tc::SPLIT_TF32X3 ? tc::idesc_tf32(TC_RT, n) : tc::idesc_bf16(TC_RT, n);
  };
  const uint32_t id1 = idesc(N), id2 = idesc(2 * N), id3 = idesc(3 * N);
  auto mma = [](uint32_t d, uint32_t a, uint64_t bb, uint32_t id, uint32_t acc) {
    if (SPLIT == tc::SPLIT_TF32X3) tc::mma_tf32_ta(d, a, bb, id, acc);
    else tc::mma_bf16_ta(d, a, bb, id, acc);
  };
  int g = 0;  // chunk of this CTA, over all its items
  bool failed = false;
  if (tid >= TC2_CONV + 32) {
    // ---- refills
    if (prod) {
      int s = 0;
      uint32_t sp = 0;
      while (!stalled && p_item < my_items) {
        if (!tc_poll(&free_bar[s], sp, tries)) {
          failed = true;
          break;
        }
        issue_next();
        if (++s == stages) {
          s = 0;
          sp ^= 1u;
        }
      }
    }
  } else if (tid >= TC2_CONV) {
    // ---- MMAs of the split chunks
    for (int t = 0; ctrl && t < my_items && !failed; ++t) {
      int half, f, rt, ks;
      item(t, half, f, rt, ks);
      const int nl = item_len(ks);
      if (t > 0 && !tc_poll(&acc_bar, (uint32_t)(t - 1) & 1u, tries)) {
        failed = true;
        break;
      }
      for (int lc = 0; lc < nl; ++lc, ++g) {
        const int q = g & (NB - 1);
        if (!tc_poll(&conv_bar[q], (uint32_t)(g >> nbs) & 1u, tries)) {
          failed = true;
          break;
        }
        tc::fence_after_sync();
        const uint64_t dB = tc::smem_desc(tc::smem_u32(ops + q * buf_bytes), TC_LBO, SBO);
        const uint32_t aq = abuf + (uint32_t)(q * PIECES) * AC;
        if constexpr (EXTRA) {
          const uint64_t lo = bt_bytes >> 4;  // to B_lo
#pragma unroll
          for (int kk = 0; kk < tc::ksteps32<SPLIT>(); ++kk) {
            const uint64_t bk = dB + (uint64_t)(kk * 2 * TC_LBO >> 4);
            const uint32_t ak = aq + (uint32_t)kk * 8;
            const uint32_t acc = (lc > 0 || kk > 1) ? 1u : 0u;
            if (kk & 1) {
              mma(tmem + 2 * N, ak, bk, id1, acc);
              mma(tmem + N, ak, bk + lo, id1, 1u);
            } else {
              mma(tmem, ak, bk, id2, acc);
            }
            mma(tmem + N, ak + AC, bk, id1, 1u);
          }
        } else {
#pragma unroll
          for (int kk = 0; kk < tc::ksteps32<SPLIT>(); ++kk) {
            const uint64_t bk = dB + (uint64_t)(kk * 2 * TC_LBO >> 4);
            const uint32_t ak = aq + (uint32_t)kk * 8;
            const uint32_t set = tmem + (uint32_t)(kk & (SETS - 1)) * set_cols;
            const uint32_t acc = (lc > 0 || kk >= SETS) ? 1u : 0u;
            mma(set, ak, bk, X6 ? id3 : id2, acc);
            if (X6) {
              mma(set + N, ak + AC, bk, id2, 1u);
              mma(set + 2 * N, ak + 2 * AC, bk, id1, 1u);
            } else {
              mma(set + N, ak + AC, bk, id1, 1u);
            }
          }
        }
        tc::mma_commit(&mma_bar[q]);
        if (lc == nl - 1) tc::mma_commit(&item_bar);
        ++committed;
      }
    }
  } else {
    // ---- converters: group gi splits the chunks g with g % 2 == gi
    const int gi = warp >> 3, gt = tid & (TC2_GROUP - 1);
    const int r = (warp & 3) * 32 + lane, kh = (warp >> 2) & 1;  // row and K half of A
    const int lkp = 31 - __clz(kp), j = gt & (kp - 1), p0 = gt >> lkp, pstep = TC2_GROUP >> lkp;
    const int first = (j >> 2) & 1;
    const uint32_t alane = abuf + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)kh * (AC / 2);
    int s = gi;
    uint32_t sp = 0;  // stage of the group's next chunk, and its parity
    for (int t = 0; t < my_items && !failed; ++t) {
      int half, f, rt, ks;
      item(t, half, f, rt, ks);
      const int nl = item_len(ks);
      const int off = (b & k & 1) ? (int)((half * hstride + f * rstride) & 1) : 0;  // (issue_tile)
      for (int lc = 0; lc < nl; ++lc, ++g) {
        if ((g & 1) != gi) continue;
        const int q = g & (NB - 1);
        bool ok = tc_poll(&full_bar[s], sp, tries);
        if (ok && g >= NB) ok = tc_poll(&mma_bar[q], (uint32_t)((g >> nbs) - 1) & 1u, tries);
        ok = __all_sync(0xffffffffu, ok);  // the stores to TMEM are a warp's
        if (!ok) {
          failed = true;
          break;
        }
        tc::fence_after_sync();
        const float* R = reinterpret_cast<const float*>(raw + s * stage_bytes);
        const float2* Rt =
            reinterpret_cast<const float2*>(raw + s * stage_bytes + TC2_TILE_BYTES) + off;
        // A: the lane's row, reals 16 kh ..; the 16-byte units of a swizzled row are
        // exchanged by its number mod 8
        float v[2][8];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (!TRANS) {
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
              const float4 g4 = *reinterpret_cast<const float4*>(
                  R + r * 32 + 4 * ((4 * kh + 2 * u + h2) ^ (r & 7)));
              v[u][4 * h2] = g4.x;
              v[u][4 * h2 + 1] = g4.y;
              v[u][4 * h2 + 2] = g4.z;
              v[u][4 * h2 + 3] = g4.w;
            }
          } else {
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              const float2 c =
                  *reinterpret_cast<const float2*>(R + (8 * kh + 4 * u + m) * 256 + 2 * r);
              v[u][2 * m] = c.x;
              v[u][2 * m + 1] = -c.y;
            }
          }
        }
        const int m0 = (ks * cpp + lc) * TC2_KC;
        // B~ rows 2j (x_r, -x_i) and 2j + 1 (x_i, x_r) of column j: both by one
        // thread, in the order that gives each 8-thread phase of the 16-byte
        // stores the eight row slots of a core matrix
        unsigned char* ob = ops + q * buf_bytes;
        unsigned char* bp[3] = {ob, ob + bt_bytes, ob + 2 * bt_bytes};
        for (int p = p0; p < 8; p += pstep) {
          const int ma = m0 + 2 * p, mb = ma + 1;
          const float2 t0 = (j < k && ma < b) ? Rt[(2 * p) * k + j] : make_float2(0.f, 0.f);
          const float2 t1 = (j < k && mb < b) ? Rt[(2 * p + 1) * k + j] : make_float2(0.f, 0.f);
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2) {
            const int odd = first ^ h2;
            const float4 w = odd ? make_float4(t0.y, t0.x, t1.y, t1.x)
                                 : make_float4(t0.x, -t0.y, t1.x, -t1.y);
            tc::store_split<SPLIT>(w, bp, tc::kmajor_off32<SPLIT>(2 * j + odd, 4 * p));
          }
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&free_bar[s]);
#pragma unroll
        for (int u = 0; u < 2; ++u)
          tc::tmem_store_split<SPLIT>(v[u], alane + (uint32_t)(q * PIECES) * AC + u * (AC / 4), AC);
        tc::fence_async_smem();
        tc::tmem_wait_st();
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&conv_bar[q]);
        s += 2;
        if (s >= stages) {
          s -= stages;
          sp ^= 1u;
        }
      }
      if (failed) break;
      // item done: wait for its last MMAs, then move the accumulator to its slot
      // (item_bar: a group does not follow the other one's buffers phase by phase)
      const bool ok = tc_poll(&item_bar, (uint32_t)t & 1u, tries);
      if (!__all_sync(0xffffffffu, ok)) {
        failed = true;
        break;
      }
      tc::fence_after_sync();
      tc::grid_wait();  // the partials are the coupling's before, until it is done
      // 16x256b fragments: warp w reads lanes 32 (w % 4) + 16 sb + [0, 16)
      // (sb = (w / 4) & 1) and float columns 32 hh + [0, 32) (hh = w / 8) of
      // each partial product; thread t holds rows t/4 and t/4 + 8 and complex
      // columns 4 r + t % 4, so four consecutive threads write 32 contiguous
      // bytes of a row (whole sectors)
      const int lq = warp & 3, sb = (warp >> 2) & 1;
      float2* pf = part + (((size_t)ks * step.nh + half) * F + f) * (size_t)b * k;
      for (int hh = warp >> 3; hh < (N + 31) / 32; hh += 2) {
        float v[16], w[16];
        const uint32_t ta =
            tmem + ((uint32_t)(lq * 32 + 16 * sb) << 16) + (uint32_t)(hh * 32);
        tc::tmem_ld_16x256b_x4(ta, v);
#pragma unroll
        for (int a = 1; a < SETS * ORDERS + EXTRA; ++a) {  // the partial sums
          tc::tmem_ld_16x256b_x4(ta + (uint32_t)(a * N), w);
#pragma unroll
          for (int tt = 0; tt < 16; ++tt) v[tt] += w[tt];
        }
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
          const int r = rt * TC_RT + lq * 32 + 16 * sb + (lane >> 2) + 8 * h2;
          if (r >= b) continue;
#pragma unroll
          for (int rr = 0; rr < 4; ++rr) {
            const int j = hh * 16 + 4 * rr + (lane & 3);
            if (j < k)
              pf[(size_t)r * k + j] = make_float2(v[4 * rr + 2 * h2], v[4 * rr + 2 * h2 + 1]);
          }
        }
      }
      tc::fence_before_sync();  // accumulator reads complete before the next item's MMAs
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acc_bar);
    }
  }
  if (failed) sfail = 1;
  tc::fence_before_sync();
  __syncthreads();
  if (sfail) {
    // the copies in flight land before the CTA's shared memory goes, the MMAs
    // committed complete before their tensor memory is freed (the uses before of
    // these stages and buffers were waited for)
    if (prod)
      for (int qq = max(0, issued - stages); qq < issued; ++qq)
        tc::mbar_wait(&full_bar[qq % stages], (uint32_t)(qq / stages) & 1u, TC_WAIT_TRIES);
    if (ctrl) {
      atomicExch(err, 1);
      if (committed > 0) {
        const int last = committed - 1;
        tc::mbar_wait(&mma_bar[last & (NB - 1)], (uint32_t)(last >> nbs) & 1u, TC_WAIT_TRIES);
      }
    }
    __syncthreads();
  }
  if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// ---------------------------------------------------------------------------
// The same product on the CUDA cores in FP32 (RR_FP32_SIMT), one contraction part:
// a CTA forms RT = 2048 / kp rows by kp columns of one problem and half, 4 x 2
// outputs a thread, over chunks of 32 columns of op(G) in three stages filled by
// cp.async (16 bytes where every row starts on 16 bytes).
// Bound: FP32 and shared memory; batches that fill the chip many times over, where
// a cluster per problem, half and column group reads G again for each group.  Rows of a
// chunk are swizzled, not padded: two CTAs an SM from kp = 16 on.
constexpr int CC_THREADS = 256, CC_KC = 32, CC_STAGES = 3, CC_RT = 2048;
template <bool TRANS>
__host__ __device__ constexpr int cc_pitch(int kp) { return TRANS ? CC_RT / kp : CC_KC; }
template <bool TRANS>
__host__ __device__ constexpr int cc_stage(int kp) {  // complex values
  return (TRANS ? CC_KC : CC_RT / kp) * cc_pitch<TRANS>(kp) + CC_KC * kp;
}

__device__ __forceinline__ void cc_copy(float2* smem, const float2* gmem, int bytes, bool ok) {
  const uint32_t s = tc::smem_u32(smem);
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem),
                 "r"(ok ? 16 : 0)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem),
                 "r"(ok ? 8 : 0)
                 : "memory");
}

template <bool TRANS>
__global__ void __launch_bounds__(CC_THREADS)
sweep_cc_kernel(const float2* __restrict__ G, int b, int ldg, int k, int kp, SweepStep step, int nx,
                int nrt, const float2* __restrict__ rhs, size_t rstride, size_t hstride,
                float2* __restrict__ part, int F, int Fa, const int* __restrict__ amap) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* base = reinterpret_cast<float2*>(smem_raw);
  const int RT = CC_RT / kp, pitch = cc_pitch<TRANS>(kp), stage_len = cc_stage<TRANS>(kp);
  const int p = blockIdx.x / nrt, r0 = (blockIdx.x - p * nrt) * RT;
  const int half = p >= Fa, f = active_problem(amap, half ? p - Fa : p);
  const float2* Gi = G + ((size_t)f * nx + step_col(step, half, nx)) * b * ldg;
  const float2* t = rhs + half * hstride + f * rstride;
  const int tid = threadIdx.x, TX = kp >> 1, TY = CC_THREADS / TX;
  const int tx = tid % TX, ty = tid / TX;
  const int gv = (b & 1) ? 1 : 2;  // columns of G a copy
  const int sw = (ty & 7) * 2;     // (rows of a chunk are swizzled; TY is a multiple of 8)
  auto load = [&](int st, int m0) {
    float2* Ms = base + st * stage_len;
    float2* Ts = Ms + stage_len - CC_KC * kp;
    const int nr = TRANS ? CC_KC : RT, per = (TRANS ? RT : CC_KC) / gv;
    for (int e = tid; e < nr * per; e += CC_THREADS) {
      const int a = e / per, u = (e - a * per) * gv;
      const int row = (TRANS ? m0 : r0) + a, col = (TRANS ? r0 : m0) + u;
      const bool ok = row < b && col < b;
      cc_copy(&Ms[a * pitch + (TRANS ? u : u ^ (a & 7) * 2)], ok ? Gi + (size_t)row * ldg + col : Gi, 8 * gv, ok);
    }
    for (int e = tid; e < CC_KC * kp; e += CC_THREADS) {
      const int mm = e / kp, j = e - mm * kp, m = m0 + mm;
      const bool ok = m < b && j < k;
      cc_copy(&Ts[e], ok ? t + (size_t)m * k + j : t, 8, ok);
    }
  };
  float2 acc[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
  const int nch = (b + CC_KC - 1) / CC_KC;
#pragma unroll
  for (int s = 0; s < CC_STAGES - 1; ++s) {
    if (s < nch) load(s, s * CC_KC);
    asm volatile("cp.async.commit_group;\n" ::);
  }
  for (int c = 0; c < nch; ++c) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(CC_STAGES - 2) : "memory");
    __syncthreads();
    if (c + CC_STAGES - 1 < nch) load((c + CC_STAGES - 1) % CC_STAGES, (c + CC_STAGES - 1) * CC_KC);
    asm volatile("cp.async.commit_group;\n" ::);
    const float2* Ms = base + (c % CC_STAGES) * stage_len;
    const float2* Ts = Ms + stage_len - CC_KC * kp;
#pragma unroll 2
    for (int mm = 0; mm < CC_KC; mm += 2) {
      float2 a[2][4], v[2][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (TRANS) {
          a[0][i] = cconj(Ms[mm * pitch + ty + TY * i]);
          a[1][i] = cconj(Ms[(mm + 1) * pitch + ty + TY * i]);
        } else {
          const float4 w = *reinterpret_cast<const float4*>(&Ms[(ty + TY * i) * pitch + (mm ^ sw)]);
          a[0][i] = make_float2(w.x, w.y);
          a[1][i] = make_float2(w.z, w.w);
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        v[h][0] = Ts[(mm + h) * kp + tx];
        v[h][1] = Ts[(mm + h) * kp + tx + TX];
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[i][0] = cfma(a[h][i], v[h][0], acc[i][0]);
          acc[i][1] = cfma(a[h][i], v[h][1], acc[i][1]);
        }
    }
  }
  float2* pf = part + ((size_t)half * F + f) * b * k;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + TY * i;
    if (r >= b) continue;
    if (tx < k) pf[(size_t)r * k + tx] = acc[i][0];
    if (tx + TX < k) pf[(size_t)r * k + tx + TX] = acc[i][1];
  }
}

// Launch that may start before its predecessor in the stream has finished; the
// kernel orders itself by grid_wait
cudaLaunchConfig_t dependent_launch(dim3 grid, int threads, size_t smem, cudaStream_t st,
                                    cudaLaunchAttribute* at, bool dependent) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cfg;
}

// One launch of the TMA-fed tensor-core sweep step in the factors' operand
// split (partial products into Pbuf).
template <bool TRANS, int SPLIT, bool WIDE>
rr_status launch_tc2(const CUtensorMap* tm, int grid_x, int b, int k, int kp,
                     const SweepStep& step, int nx, int nrt, int KS, int cpp, const float2* rhs,
                     size_t rstride, size_t hstride, bool first, rr_factors* fa, cudaStream_t st) {
  const size_t smem = tc2_smem_bytes<SPLIT>(kp) + 1024;
  RR_TRY((smem_opt_in<sweep_tc2_kernel<TRANS, SPLIT, WIDE>>(
      tc2_smem_bytes<SPLIT>(WIDE ? 64 : 32) + 1024)));
  // dependent launch, but for the first: its predecessor is not of this solve
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = dependent_launch(dim3(grid_x), TC2_THREADS, smem, st, at, !first);
  RR_CUDA(cudaLaunchKernelEx(&cfg, sweep_tc2_kernel<TRANS, SPLIT, WIDE>, *tm, b, k, kp, step, nx, nrt,
                             KS, cpp, rhs, rstride, hstride, reinterpret_cast<float2*>(fa->Pbuf),
                             fa->F, active_count(fa), (const int*)fa->amap, fa->err,
                             wait_tries(), take_stall()));
  return RR_OK;
}

}  // namespace

namespace {

template <bool TRANS>
rr_status launch_cc(int k, int kp, const SweepStep& step, const float2* rhs, size_t rstride,
                    size_t hstride, rr_factors* fa, cudaStream_t st) {
  const OpDev& d = fa->op->d;
  const int nrt = (d.b * kp + CC_RT - 1) / CC_RT, Fa = active_count(fa);
  const size_t smem = (size_t)CC_STAGES * cc_stage<TRANS>(kp) * sizeof(float2);
  RR_TRY(smem_opt_in<sweep_cc_kernel<TRANS>>(CC_STAGES * cc_stage<TRANS>(8) * sizeof(float2)));
  sweep_cc_kernel<TRANS><<<nrt * Fa * step.nh, CC_THREADS, smem, st>>>(
      reinterpret_cast<const float2*>(fa->G), d.b, fa->ldg, k, kp, step, d.nx, nrt, rhs, rstride,
      hstride, reinterpret_cast<float2*>(fa->Pbuf), fa->F, Fa, fa->amap);
  RR_CUDA(cudaGetLastError());
  return RR_OK;
}

}  // namespace

// The split tensor-core sweep (sweep_tc2_kernel) serves FP32 factors with a block
// of at least 48 (one tile of 128 rows still beats the cluster form in large batches:
// 126 rows, 32 right-hand sides, 128 problems 1.6 ms a solve instead of 2.2) and at most
// 64 columns.  The three orders of the BF16 x6 split need 6N accumulator columns, so
// beyond 32 its sweeps take the TF32 split (768 rows, 64 right-hand sides, 16
// problems: 2.7 ms a solve instead of 20 in the cluster form, no larger an error).
static bool sweep_tc2_ok(const rr_factors* fa, int k) {
  return tc_prec(fa->prec) && k <= 64 && fa->tma_ok;
}

namespace {

// Split count of a product: the smallest whose items fill the persistent CTAs to
// 85 % (each split adds a partial block to write and sum), else the best
// balance.  The partial buffer holds 4 F b 64 complex, so up to 256 / k splits
// of one half's problems fit; few active problems (refinement corrections) take more splits to keep
// the SMs busy.
int split_count(const rr_factors* fa, int k, int nh, int nrt, int nch, int nsm) {
  const int ks_max = std::min(16, std::max(1, 256 / (k * nh)));
  if (fa->tune_ks > 0) {  // tuned (as far as the partial buffer goes)
    const int ksc = std::min(fa->tune_ks, ks_max);
    const int cpp = (nch + ksc - 1) / ksc;
    return (nch + cpp - 1) / cpp;
  }
  int KS = 1;
  double best = 0.0;
  for (int ksc = 1; ksc <= ks_max && ksc <= nch; ++ksc) {
    const int cpp = (nch + ksc - 1) / ksc;
    const int ksr = (nch + cpp - 1) / cpp;
    if (ksr > ks_max) continue;
    const long items = (long)nrt * active_count(fa) * nh * ksr;
    const long waves = (items + nsm - 1) / nsm;
    const double eff = (double)items / (double)(waves * nsm);
    if (eff >= 0.85) return ksr;
    if (eff > best + 1e-9) {
      best = eff;
      KS = ksr;
    }
  }
  return KS;
}

template <bool TRANS, typename V>
rr_status solve_tc2(rr_factors* fa, int k, const float2* in, float2* x, float2* zh) {
  const OpDev& d = fa->op->d;
  const int b = d.b, nx = d.nx, F = fa->F, Fa = active_count(fa);
  const int units = k / (int)(sizeof(V) / sizeof(float2));  // of a row
  int kp = 8;
  while (kp < k) kp <<= 1;
  cudaStream_t st = fa->stream;
  float2* tb = reinterpret_cast<float2*>(fa->Tbuf);  // [2][F][b][k]
  const int nrt = (b + TC_RT - 1) / TC_RT, nch = (b + TC2_KC - 1) / TC2_KC;
  const int nsm = num_sms(d.device);
  const CUtensorMap* tm = reinterpret_cast<const CUtensorMap*>(fa->tmap[TRANS ? 1 : 0]);
  const size_t csmem = (size_t)(CPL_Y + 2) * d.q * k * sizeof(float2);
  const int n0 = half_cols(0, nx), n1 = half_cols(1, nx);  // n1 is n0 or n0 - 1
  for (int s = 0; s <= 2 * n0; ++s) {
    SweepStep step;
    step.phase = s < n0 ? SW_IN : s == n0 ? SW_MID : SW_OUT;
    step.t = s < n0 ? s : s - n0;
    step.nh = step.phase == SW_IN ? (step.t < n1 ? 2 : 1) : step.phase == SW_MID ? 1
              : step.t <= n1 ? 2 : 1;
    const float2* rhs = s == 0 ? in : tb;
    const size_t rstride = s == 0 ? (size_t)d.n * k : (size_t)b * k;
    const size_t hstride = s == 0 ? (size_t)(nx - 1) * b * k : (size_t)F * b * k;
    const bool cc = fa->prec == RR_FP32_SIMT;
    const int KS = cc ? 1 : split_count(fa, k, step.nh, nrt, nch, nsm), cpp = (nch + KS - 1) / KS;
    const int grid_x = std::min(nrt * Fa * step.nh * KS, nsm);
    if (step.phase == SW_MID) {
      prof_begin(PROF_SWEEP, st);
      sweep_middle_kernel<TRANS, V><<<dim3((b * units + 255) / 256, Fa), 256, 0, st>>>(
          view(d), k, in, TRANS ? x : zh, tb, fa->amap);
      prof_end(PROF_SWEEP, st);
    }
    prof_begin(PROF_SWEEP, st);
    auto product = [&](auto launch) {
      return launch(tm, grid_x, b, k, kp, step, nx, nrt, KS, cpp, rhs, rstride, hstride, s == 0, fa,
                    st);
    };
    rr_status ls;
    if (cc)
      ls = launch_cc<TRANS>(k, kp, step, rhs, rstride, hstride, fa, st);
    else if (fa->prec == RR_FP32_BF16X3)
      ls = kp > 32 ? product(launch_tc2<TRANS, tc::SPLIT_BF16X3, true>)
                   : product(launch_tc2<TRANS, tc::SPLIT_BF16X3, false>);
    else if (fa->prec == RR_FP32_BF16X6 && kp <= 32)
      ls = product(launch_tc2<TRANS, tc::SPLIT_BF16X6, false>);
    else
      ls = kp > 32 ? product(launch_tc2<TRANS, tc::SPLIT_TF32X3, true>)
                   : product(launch_tc2<TRANS, tc::SPLIT_TF32X3, false>);
    if (ls != RR_OK) return ls;
    // (the middle's result starts both halves' outward sweeps)
    const int ch = step.phase == SW_MID ? 2 : step.nh;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg =
        dependent_launch(dim3((d.ny + CPL_Y - 1) / CPL_Y * Fa * ch), couple_threads(d.q, units),
                         csmem, st, at, true);
    RR_CUDA(cudaLaunchKernelEx(&cfg, sweep_couple_kernel<TRANS, V>, view(d), step, F, Fa, k, KS,
                               reinterpret_cast<const float2*>(fa->Pbuf), in, x, zh, tb,
                               (const int*)fa->amap));
    prof_end(PROF_SWEEP, st);
    prof_count(1);
    RR_CUDA(cudaGetLastError());
  }
  return RR_OK;
}

}  // namespace

// Modelled microseconds of a solve in the tensor-core form, less what the cluster form
// also takes: per pair of columns the launches, and the busiest CTA's chunks and
// items.  Fitted together with form_step_us (sweep_cl.cuh) to 1467 shapes, forward and
// adjoint: the form taken is the slower one by more than 5 % in 2 % of them.  Measured,
// ms of a whole unrefined solve of 16 columns, tensor-core and cluster form: 48 rows, 16
// right-hand sides, 128 problems 0.48 and 0.37; 96 rows, 32, 128 problems 1.09 and
// 1.50; 192 rows, 8, 32 problems 0.61 and 0.34; 387 rows, 32, 64 problems 2.8 and
// 7.6; 768 rows, 32, 1 and 16 problems 0.40 and 1.6 instead of 1.13 and 7.1.
static double sweep_tc2_us(const rr_factors* fa, int k) {
  const OpDev& d = fa->op->d;
  const int nrt = (d.b + TC_RT - 1) / TC_RT, nch = (d.b + TC2_KC - 1) / TC2_KC;
  const int nsm = num_sms(d.device), KS = split_count(fa, k, 2, nrt, nch, nsm);
  const double items = std::ceil(2.0 * nrt * active_count(fa) * KS / nsm);  // of a CTA
  const int cpp = (nch + KS - 1) / KS;
  return (d.nx + 1.0) * (4.3 + items * (1.34 + 0.67 * cpp));
}

// The same for the product on the CUDA cores (RR_FP32_SIMT): the chunks' latency per
// wave of resident CTAs and their arithmetic.  Measured, ms of a whole unrefined
// forward solve of 16 columns, this and the cluster form: 192 rows, 8 right-hand sides,
// 64 problems 0.76 and 0.58; 384 rows, 64, 16 problems 2.3 and 2.8; 768 rows, 64, 64
// problems 23.6 and 55.
static double sweep_cc_us(const rr_factors* fa, int k) {
  const OpDev& d = fa->op->d;
  int kp = 8;
  while (kp < k) kp <<= 1;
  const int nch = (d.b + CC_KC - 1) / CC_KC, Fa = active_count(fa), nsm = num_sms(d.device);
  const double ctas = 2.0 * Fa * ((d.b * kp + CC_RT - 1) / CC_RT);
  const double waves = std::ceil(ctas / (nsm * (kp <= 8 ? 1.0 : kp == 16 ? 2.0 : 3.0)));
  return (d.nx + 1.0) * (4.5 + nch * (2.8 * waves + 0.96 * ctas / nsm));
}

// FP32 solves that take the column-pair form: where both forms serve a shape, the
// one with the smaller modelled time.
static bool sweep_steps_taken(const rr_factors* fa, int k, int adjoint) {
  const bool simt = fa->prec == RR_FP32_SIMT;
  if (!simt && !sweep_tc2_ok(fa, k)) return false;
  return (simt ? sweep_cc_us(fa, k) : sweep_tc2_us(fa, k)) < sweep_cl32_us(fa, k, adjoint);
}

bool sweep_tc2_taken(const rr_factors* fa, int k, int adjoint) {
  return tc_prec(fa->prec) && sweep_steps_taken(fa, k, adjoint);
}

// FP64 factors and FP32 shapes that the column-pair form does not take run the
// whole-sweep cluster kernels.
rr_status launch_solve_lo(rr_factors* fa, int k, int adjoint, const void* b, void* x, void* tmp) {
  if (fa->prec == RR_FP64) return launch_sweep_cl64(fa, k, adjoint, b, x, tmp);
  if (sweep_steps_taken(fa, k, adjoint)) {
    const float2* in = reinterpret_cast<const float2*>(b);
    float2 *xo = reinterpret_cast<float2*>(x), *zh = reinterpret_cast<float2*>(tmp);
    if (k % 2)
      return adjoint ? solve_tc2<true, float2>(fa, k, in, xo, zh)
                     : solve_tc2<false, float2>(fa, k, in, xo, zh);
    return adjoint ? solve_tc2<true, float4>(fa, k, in, xo, zh)
                   : solve_tc2<false, float4>(fa, k, in, xo, zh);
  }
  return launch_sweep_cl32(fa, k, adjoint, b, x, tmp);
}
