// psl_lin.cu -- neighbourhood score of batches with long walks (arXiv 2107.09801), split into a
// correlation on the tensor cores and one table lookup per five two-partner shifts.
//
// For neighbour j and shift k let sigma = s_j s_{j+k} and tau = s_j s_{j-k}.  A two-partner shift
// changes F by Tp4_k (sigma = tau = -1), Tm4_k (sigma = tau = +1) or nothing, a one-partner shift
// by Tp2_k or Tm2_k.  With
//   A_k = (Tp4_k + Tm4_k) / 2,  B_k = (Tm4_k - Tp4_k) / 4,  D_k = (Tm2_k - Tp2_k) / 2,
//   E_k = (Tp2_k + Tm2_k) / 2
// the two cases are A_k [sigma = tau] + B_k (sigma + tau) and E_k + D_k sigma, so
//   score(j) = sum_{k <= kin} A_k [s_{j+k} = s_{j-k}]                 (k_quad: subset-sum tables)
//            + s_j sum_{p != j} g_{|p-j|} s_p + sum_{kin < k <= kout} E_k   (k_lin)
// with g = B where both j + |p-j| and j - |p-j| lie inside the sequence and D elsewhere.  The middle
// sum is a correlation of the sequence with a fixed vector: a matrix product.  The tables need one
// lookup where the direct form needs two (W1, W0), and one-partner shifts need none.
//
// k_lin.  Window positions are tiled as j = jA + 64 b + a (rows b < 128, a < 64) and partners as
// p = jA + 64 (b + tau) + x, x < 64.  For one chunk tau,
//   Y[b, a] += sum_x S[b + tau, x] G[64 tau + x - a],   S[r, x] = s_{jA + 64 r + x} (0 outside),
// is a 128 x 64 x 64 product: tcgen05.mma kind::f16, M = 128, N = 192, four steps of K = 16.
//   * G in fixed point: B_k and D_k are rounded once to multiples of 2^-lin_sh (35 bits for the largest; a
//     coefficient 2^-11 of it keeps as many as FP32, smaller ones fewer, the least round to zero) and split
//     into three balanced base-4096 digits, each exact in f16; the digits are the three column
//     groups of N.  Sums of at most 8192 products of +-1 with |digit| <= 2048 stay within 2^24, so
//     the FP32 accumulators hold exact integers; every 128 chunks they are added into 64-bit
//     integers.  The result is the exact sum of the rounded coefficients, whatever the order.
//   * both operands are K-major without swizzle, and neither is stored as a matrix.  S is kept by
//     eight-element columns x/8 with consecutive rows 16 bytes apart, so chunk tau + 1 is the same
//     buffer 16 bytes further on: 8192 positions are expanded from bits once per 128 chunks.  G is a
//     Toeplitz matrix: eight copies of the digit vector, copy c shifted by c elements, interleaved in
//     16-byte units are its core matrices at a stride of one unit in both directions.
//   * which of B and D a partner takes changes along p = 2j (and p = 2j - (L-1)): decided per row and
//     chunk (p0 <= 2 j0 of row and chunk).  A chunk where rows differ is done twice, with an S tile
//     whose rows of the other kind are zero.  k_quad adds the (at most 126) terms per side by which
//     this rule differs from the exact boundary.
// Roles: warps 0-7 expand S and drain the accumulators (256 TMEM columns per pipe), warps 8-13 build G
// (a chunk each, a ring of stages per pipe), one thread of either of warps 14 and 15 issues a pipe's
// products.  Every wait on an mbarrier is bounded.  When one runs out, every role of the block leaves its
// item, the walk whose item the epilogue was at gets its error, and the block starts again at its next item
// with fresh barriers; if products may still be in flight, the walks of all its remaining items get theirs and
// it ends.  k_quad then fails those walks: no status changes while k_lin runs, so that all threads of a block
// agree on which items exist.
//
// What bounds it, at 304 walks of L = 131071 (N = 6912; two or three tiles per SM): k_lin 2.3 ms, the
// tensor pipe active 58% of it (386 cycles a chunk; the rest is the issuing threads' instruction latency, the
// chunks done twice and the readings of the accumulators); k_quad 2.9 ms, 77% of the issue slots, 71% of the ALU
// pipe and 57% of the shared-memory wavefronts (two ALU instructions and one lookup per five shifts).  The
// tables alone took 10.1 ms.  A whole step of 1024 such walks: 35.2 -> 17.9 ms.
#include <climits>
#include <cstdint>
#include <cstdio>

#include "psl_async.cuh"
#include "psl_device.cuh"
#include "psl_internal.h"

namespace psl {

namespace {

constexpr int kP = 64;                       // positions per row and per chunk
constexpr int kRows = 128;                   // rows of a tile (M)
constexpr int kTilePos = kP * kRows;         // window positions per tile
constexpr int kSegTau = 128;                 // chunks per segment, between two readings of the accumulators
                                             // (half of them in either one: 4096 terms, 8192 would be exact)
constexpr int kWinRows = kRows + kSegTau;    // rows of S one segment reads
constexpr int kWinPlane = kWinRows * 16;     // bytes between the columns of S
constexpr int kWinBytes = kP / 8 * kWinPlane;
constexpr int kDig = 3;                      // base-4096 digits
constexpr int kHCh = 2 * kP / 8 - 1;         // eight-element units of G per chunk
constexpr int kHDig = 128 + 16;              // bytes per digit of a unit: eight copies x 16, and 16 so that the
constexpr int kHUnit = kDig * kHDig;         // builders' words of eight units lie in distinct banks
constexpr int kHBytes = kHCh * kHUnit;
constexpr int kSPlane = kRows * 16;
constexpr int kSTileBytes = kP / 8 * kSPlane;  // S tile of a chunk whose rows differ in kind
// Two product pipelines, for the even and the odd chunks of a tile: an issuing thread waits about 65
// cycles per instruction, so that one alone (4 products, a wait, a commit: 900 cycles a chunk) would
// leave the tensor cores idle more than half the time (386 cycles a chunk).
constexpr int kPipes = 2;
constexpr int kStages = 7, kSTiles = 2;      // rings of G and of S tiles, per pipe
constexpr int kLinEpiWarps = 8, kPipeBuilders = 3, kLinBuilders = kPipes * kPipeBuilders;
constexpr int kLinThreads = 32 * (kLinEpiWarps + kLinBuilders + kPipes);
constexpr int kAccCols = 256;                // TMEM columns between the two accumulator buffers
constexpr size_t kLinSmem = 128 + 2 * (size_t)kWinBytes + kPipes * (kStages * (size_t)kHBytes + kSTiles * (size_t)kSTileBytes);
// A builder's wait on a stage for product q - kStages is sound when product q - 2 kStages is known to be
// complete: its own last product, at most 2 kPipeBuilders before q, waited for the one kStages before that.
static_assert(kStages >= 2 * kPipeBuilders, "a stage's barrier is at most one phase behind its builder");
static_assert(kSTiles == 2, "one for B's rows, one for D's");
static_assert(kWinRows <= 32 * kLinEpiWarps, "a thread expands a row");
static_assert(kTilePos == (int)kLinTilePos, "tile size shared with the host's item list");

// instruction descriptor: f16 x f16 -> f32, both operands K-major, M = 128, N = 192
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(kDig * kP / 8) << 17) | ((128u / 16u) << 24);

// shared-memory matrix descriptor, no swizzle: lbo = bytes between core matrices along K,
// sbo = bytes between core matrices along M or N
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)((lbo >> 4) & 0x3fffu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3fffu) << 32) | (1ull << 46);
}

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, bool acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(kIdesc), "r"((uint32_t)acc)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t (&r)[8], uint32_t addr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

constexpr int kWaitLimit = 1 << 20;  // polls, each of which may itself suspend for a while
// Bounded wait that also ends when another thread of the block gave up.
__device__ __forceinline__ bool wait_or_err(uint32_t mbar, uint32_t parity, volatile int *err) {
  for (int it = 0; it < kWaitLimit; it++) {
    if (mbar_try_wait(mbar, parity)) return true;
    if (*err) return false;
  }
  *err = 1;
  return false;
}
// The same for a whole warp with one lane polling, `ns` apart; every lane then observes the completed
// phase itself.
__device__ __forceinline__ bool warp_wait(uint32_t mbar, uint32_t parity, volatile int *err, uint32_t ns,
                                          int limit = kWaitLimit) {
  bool ok = true;
  if ((threadIdx.x & 31) == 0) {
    ok = false;
    for (int it = 0; it < limit && !*err; it++) {
      if ((ok = mbar_try_wait(mbar, parity))) break;
      __nanosleep(ns);
    }
    if (!ok) *err = 1;
  }
  ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
  return ok && mbar_wait_bounded(mbar, parity);
}

__device__ __forceinline__ int floor_div64(int v) { return v >> 6; }

// A tile of one walk's window: positions jA .. jA + cnt - 1 and the chunks tau_lo .. tau_hi of its
// partners this item does.   A window that wraps around the end of the sequence has a tile list
// on either side; the full neighbourhood (N = L) is taken from position 0 and never wraps.
struct LinTile {
  int L, jA, cnt, nb, rmin, rmax, qa, tau_lo, tau_hi, shares;
  int b_lo, b_hi, d_lo, d_hi;  // chunks with rows that take B: [b_lo, b_hi]; D: tau <= d_lo or tau >= d_hi
  bool ok, stall;              // stall: the test hook withholds the item's products
};

__device__ __forceinline__ LinTile lin_tile(const WalkDev &W, const HotItem &it) {
  LinTile g;
  g.ok = false;
  if (W.status != kRunning) return g;
  g.stall = (W.inject_stall & kStallProducts) != 0;
  const int L = (int)W.L, N = (int)W.N;
  const int f = ((int)W.start + 1) % L;
  int s0 = f, n0 = min(N, L - f), s1 = 0, n1 = N - n0;
  if (N == L) s0 = 0, n0 = L, n1 = 0;
  const int t0 = (n0 + kTilePos - 1) / kTilePos;
  int t = (int)it.i0;
  if (t >= t0) t -= t0, s0 = s1, n0 = n1;
  if (t * kTilePos >= n0) return g;
  g.L = L;
  g.jA = s0 + t * kTilePos;
  g.cnt = min(kTilePos, n0 - t * kTilePos);
  g.nb = (g.cnt + kP - 1) / kP;
  g.qa = floor_div64(g.jA);
  g.rmin = -floor_div64(g.jA + kP - 1);
  g.rmax = floor_div64(L - 1 - g.jA);
  const int lo = g.rmin - (g.nb - 1), n = g.rmax - lo + 1;
  const int per = (n + (int)it.pad - 1) / (int)it.pad;  // chunks per item when the partners are split
  g.shares = (n + per - 1) / per;  // shares with anything to do
  g.tau_lo = lo + (int)it.kc * per;
  g.tau_hi = min(g.rmax, g.tau_lo + per - 1);
  g.ok = g.tau_lo <= g.tau_hi;
  // Row b of chunk tau takes B for b in [tau - qa, tau + rmax] and has partners inside the sequence for
  // b in [max(0, rmin - tau), min(nb - 1, rmax - tau)]
  g.b_lo = max(-g.rmax, -((g.rmax - g.rmin) >> 1));
  g.b_hi = min(g.qa + g.nb - 1, (g.rmax + g.qa) >> 1);
  g.d_lo = min(0, g.nb - 1 - g.rmax) - 1;
  g.d_hi = g.qa + 1;
  return g;
}

// The kinds of rows in a chunk: bit 0 B, bit 1 D.  A chunk with both is two products, B's first, each
// with an S tile whose rows of the other kind are zero.
__device__ __forceinline__ int lin_kinds(const LinTile &g, int tau) {
  return (tau >= g.b_lo && tau <= g.b_hi ? 1 : 0) | (tau <= g.d_lo || tau >= g.d_hi ? 2 : 0);
}
// chunks of a pipe with both kinds in [tau_lo, tau)
__device__ __forceinline__ int lin_doubles(const LinTile &g, int tau, int pipe) {
  const int par = (g.tau_lo + pipe) & 1;
  // numbers of that parity in [lo, hi]
  auto count = [&](int lo, int hi) { return hi < lo ? 0 : ((hi - par) >> 1) - ((lo - par + 1) >> 1) + 1; };
  const int hi = tau - 1;
  return count(max(g.b_lo, g.tau_lo), min(min(g.b_hi, g.d_lo), hi)) +
         count(max(max(g.b_lo, g.d_hi), g.tau_lo), min(g.b_hi, hi));
}

// the low eight bits as f16 values, +1 for 0 and -1 for 1
__device__ __forceinline__ uint4 pm1_f16(uint32_t v) {
  auto pair = [](uint32_t x) { return (((x & 3u) * 0x40008000u) & 0x80008000u) ^ 0x3C003C00u; };
  return make_uint4(pair(v), pair(v >> 2), pair(v >> 4), pair(v >> 6));
}
// zeroes those of eight positions p .. p+7 that lie outside the sequence
__device__ __forceinline__ void clip8(uint4 &o, int L, int p) {
  auto keep = [&](int q) {
    return (p + q >= 0 && p + q < L ? 0x0000ffffu : 0u) | (p + q + 1 >= 0 && p + q + 1 < L ? 0xffff0000u : 0u);
  };
  o.x &= keep(0), o.y &= keep(2), o.z &= keep(4), o.w &= keep(6);
}
// bits of positions p .. p+63 (a row; those outside the sequence are clipped later)
__device__ __forceinline__ void load64(const uint32_t *__restrict__ bits, int L, int p, uint32_t &lo, uint32_t &hi) {
  lo = hi = 0u;
  if (p + 63 < 0 || p >= L) return;
  const int w = p >> 5, nw = (L + 31) >> 5;  // words -2 .. nw+1 exist
  const uint32_t a = __ldg(bits + w), b = __ldg(bits + w + 1), c = __ldg(bits + min(w + 2, nw + 1));
  lo = __funnelshift_r(a, b, p & 31);
  hi = __funnelshift_r(b, c, p & 31);
}

__device__ __forceinline__ void sts128(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// a - b (|a - b| < 2^35, both rounded to 24 bits) to within one unit as d[0] + 4096 d[1] + 2^24 d[2],
// each an integer of at most 2048 in magnitude.  a - b is hi + e exactly; hi - 2^24 d[2] is exact,
// adding e rounds to half a unit at most (below 2^23 + 2^10), and so does the last digit.
__device__ __forceinline__ void lin_digits(float a, float b, float (&d)[kDig]) {
  constexpr float kMagic = 12582912.f;  // 1.5 * 2^23: adding and subtracting it rounds to an integer
  const float hi = a - b, bb = hi - a, e = (a - (hi - bb)) - (b + bb);
  d[2] = __fadd_rn(__fmaf_rn(hi, 0x1p-24f, kMagic), -kMagic);
  const float r = __fmaf_rn(d[2], -0x1p24f, hi) + e;
  d[1] = __fadd_rn(__fmaf_rn(r, 0x1p-12f, kMagic), -kMagic);
  d[0] = __fadd_rn(__fadd_rn(__fmaf_rn(d[1], -0x1p12f, r), kMagic), -kMagic);
}
template <int ID, int N>
__device__ __forceinline__ void named_sync() {
  asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory");
}
// the same, returning whether v holds for any of the threads
__device__ __forceinline__ bool named_any(int id, int n, bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, %2, %3, p;\n selp.b32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}

// E_k in units of 2^-sh
__device__ __forceinline__ long long e_fixed(const float4 *__restrict__ T, int k, float s2) {
  const float2 v = __ldg(reinterpret_cast<const float2 *>(T + k) + 1);
  return __float2ll_rn(v.x * s2) + __float2ll_rn(v.y * s2);
}
// E summed over (kin, kout] of position j minus the same of position j - 1
__device__ __forceinline__ long long e_step(const float4 *__restrict__ T, int j, int L, float s2) {
  const int kp = min(j - 1, L - j), kc = min(j, L - 1 - j);
  const int op = max(j - 1, L - j), oc = max(j, L - 1 - j);
  long long d = 0;
  if (kc > kp) d -= e_fixed(T, kc, s2);
  if (kc < kp) d += e_fixed(T, kp, s2);
  if (oc > op) d += e_fixed(T, oc, s2);
  if (oc < op) d -= e_fixed(T, op, s2);
  return d;
}

// What the roles of a block share.
constexpr int kPipeBars = 2 * kStages + 2 * kSTiles + 2;  // full, empty, S full, S empty, accumulated, drained
constexpr int kLinBars = kPipes * kPipeBars + 3;
struct LinShared {
  uint64_t bar[kLinBars];
  long long seg[kLinEpiWarps], red[kLinEpiWarps];
  uint32_t tmem;
  uint32_t first, at;  // the block's first item, and the one the epilogue is at (past the last: their number)
  int err, pending;    // a wait ran out; products may still be in flight
  int limit;           // polls of the epilogue's wait for products
};
__shared__ LinShared s_lin;

__device__ __forceinline__ uint32_t lin_bars() { return (uint32_t)__cvta_generic_to_shared(s_lin.bar); }
__device__ __forceinline__ uint32_t pipe_b(int pipe, uint32_t at) { return lin_bars() + 8u * ((uint32_t)(pipe * kPipeBars) + at); }
__device__ __forceinline__ uint32_t full_b(int pipe, uint32_t s) { return pipe_b(pipe, s); }
__device__ __forceinline__ uint32_t empty_b(int pipe, uint32_t s) { return pipe_b(pipe, kStages + s); }
__device__ __forceinline__ uint32_t sfull_b(int pipe, uint32_t s) { return pipe_b(pipe, 2 * kStages + s); }
__device__ __forceinline__ uint32_t sempty_b(int pipe, uint32_t s) { return pipe_b(pipe, 2 * kStages + kSTiles + s); }
__device__ __forceinline__ uint32_t accf_b(int pipe) { return pipe_b(pipe, 2 * kStages + 2 * kSTiles); }
__device__ __forceinline__ uint32_t drain_b(int pipe) { return pipe_b(pipe, 2 * kStages + 2 * kSTiles + 1); }
__device__ __forceinline__ uint32_t win_b(uint32_t s) { return lin_bars() + 8u * (kPipes * kPipeBars + s); }
__device__ __forceinline__ uint32_t acce_b() { return lin_bars() + 8u * (kPipes * kPipeBars + 2); }

__device__ __forceinline__ void lin_init_bars() {
  for (int pipe = 0; pipe < kPipes; pipe++) {
    for (uint32_t s = 0; s < kStages; s++) {
      mbar_init(full_b(pipe, s), 32);
      mbar_init(empty_b(pipe, s), 1);
    }
    for (uint32_t s = 0; s < kSTiles; s++) {
      mbar_init(sfull_b(pipe, s), 32 * kLinEpiWarps);
      mbar_init(sempty_b(pipe, s), 1);
    }
    mbar_init(accf_b(pipe), 1);
    mbar_init(drain_b(pipe), 1);
    mbar_init(win_b((uint32_t)pipe), 32 * kLinEpiWarps);
  }
  mbar_init(acce_b(), 32 * kLinEpiWarps);
  fence_mbar_init();
  s_lin.err = s_lin.pending = 0;
}

// The block's items from s_lin.first on (every gridDim.x-th), until they are done or a wait runs out.
// A call of its own: inlined into the loop of k_lin, the epilogue spills (304 walks of L = 131071: 5.96 ms a
// step, 5.87 so).
__device__ __noinline__ void lin_items(WalkDev *hdr, const HotItem *items, uint32_t nitems) {
  extern __shared__ __align__(128) uint8_t lin_smem[];
  LinShared &s = s_lin;
  const uint32_t base = ((uint32_t)__cvta_generic_to_shared(lin_smem) + 127u) & ~127u;
  const uint32_t win_s = base, stile_s = win_s + 2 * kWinBytes, h_s = stile_s + kPipes * kSTiles * kSTileBytes;
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t tmem = s.tmem;
  volatile int *err = &s.err;
  if (warp < kLinEpiWarps) {
    // ---------------- expand S, drain the accumulators, write Y ----------------
    uint32_t sg = 0, sq[kPipes] = {0, 0};  // segments, and chunks with S tiles of either pipe, so far
    bool ok = true;
    for (uint32_t n = s.first; ok && n < nitems; n += gridDim.x) {
      const HotItem it = items[n];
      const WalkDev &W = hdr[it.slot];
      const LinTile g = lin_tile(W, it);
      if (!g.ok) continue;
      if (tid == 0) s.at = n, s.limit = g.stall ? 64 : kWaitLimit;
      const int L = g.L;
      const uint32_t *__restrict__ bits = W.bits;
      const float4 *__restrict__ T = W.T;
      const float s2 = ldexpf(1.f, W.lin_sh - 1);
      auto build_win = [&](int seg, uint32_t buf) {
        const int r0 = g.tau_lo + seg * kSegTau;
        const int nrow = kRows + min(kSegTau, g.tau_hi - r0 + 1);
        if (tid < nrow) {
          const int p = g.jA + kP * (r0 + tid);
          const bool in = p >= 0 && p + kP <= L, any = p < L && p + kP > 0;
          uint32_t b0, b1;
          load64(bits, L, p, b0, b1);
#pragma unroll
          for (int x = 0; x < 8; x++) {
            uint4 o = any ? pm1_f16((x < 4 ? b0 : b1) >> (8 * (x & 3))) : make_uint4(0u, 0u, 0u, 0u);
            if (!in) clip8(o, L, p + 8 * x);
            sts128(win_s + buf * kWinBytes + (uint32_t)(x * kWinPlane + tid * 16), o);
          }
        }
        fence_proxy_async();
        mbar_arrive(win_b(buf));
      };
      const int nseg = (g.tau_hi - g.tau_lo) / kSegTau + 1;
      build_win(0, sg & 1u);  // its buffer was drained with the segment before last
      named_sync<1, 32 * kLinEpiWarps>();  // (read below; later windows are ordered by the draining)
      long long acc[32];
#pragma unroll
      for (int q = 0; q < 32; q++) acc[q] = 0;
      const int half = warp >> 2;
      const int b = 32 * (warp & 3) + lane, x0 = kP * b + (half == 0 ? 32 : 0);  // first offset of the thread
      const bool first = it.kc == 0;
      long long *Y = lin_y(W);
      auto win_index = [&](int j) {
        const int i = j - (int)W.start - 1;
        return i < 0 ? i + L : i;
      };
      // the shares of a split tile add up; a whole tile stores, then adds to what it stored itself
      auto add_y = [&](int i, long long v, bool again) {
        if (it.pad > 1)
          atomicAdd(reinterpret_cast<unsigned long long *>(Y + i), (unsigned long long)v);
        else
          Y[i] = again ? Y[i] + v : v;
      };
      const uint32_t tm0 = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(half * 4 * 8 * kDig);
      for (int seg = 0; seg < nseg; seg++, sg++) {
        const uint32_t buf = sg & 1u;
        if (seg + 1 < nseg) build_win(seg + 1, buf ^ 1u);
        // the S tiles of the segment's chunks whose rows differ: rows of one kind, the others zero, copied
        // from the segment's window
        const int ta = g.tau_lo + seg * kSegTau, tb = min(g.tau_hi, ta + kSegTau - 1);
        for (int part = 0; part < 2; part++) {
          const int t_lo = max(part == 0 ? g.b_lo : max(g.b_lo, g.d_hi), ta);
          const int t_hi = min(part == 0 ? min(g.b_hi, g.d_lo) : g.b_hi, tb);
          for (int t = t_lo; ok && t <= t_hi; t++) {
            const int pipe = (t - g.tau_lo) & 1, row = tid & (kRows - 1), xh = tid / kRows;  // a thread: half a row
            const bool is_b = row >= t - g.qa && row <= t + g.rmax;
            const uint32_t src = win_s + buf * kWinBytes + (uint32_t)(4 * xh * kWinPlane + (t - ta + row) * 16);
            const uint32_t dst = stile_s + (uint32_t)(pipe * kSTiles) * kSTileBytes + (uint32_t)(4 * xh * kSPlane + row * 16);
            uint4 o[4];
#pragma unroll
            for (int x = 0; x < 4; x++) o[x] = lds128(src + (uint32_t)(x * kWinPlane));
            uint32_t &n_s = pipe ? sq[1] : sq[0];  // chunks with S tiles: B's tile, then D's
            for (int dk = 0; dk < 2; dk++) {
              if (n_s > 0) ok = ok && warp_wait(sempty_b(pipe, dk), (n_s - 1u) & 1u, err, 20);
#pragma unroll
              for (int x = 0; x < 4; x++)
                sts128(dst + (uint32_t)(dk * kSTileBytes + x * kSPlane), is_b == (dk == 0) ? o[x] : make_uint4(0u, 0u, 0u, 0u));
              fence_proxy_async();
              mbar_arrive(sfull_b(pipe, dk));
            }
            n_s++;
          }
        }
        if (seg == 0) {
          // While the products run: sum E over (kin, kout] of every position, into Y.  First this item's
          // share of the sum for the tile's first position
          long long es = 0;
          const int k0 = min(g.jA, L - 1 - g.jA) + 1, k1 = max(g.jA, L - 1 - g.jA);
          const int per = (k1 - k0) / g.shares + 1;
          const int ka = k0 + (int)it.kc * per, kb = min(k1, ka + per - 1);
#pragma unroll 8
          for (int k = ka + tid; k <= kb; k += 32 * kLinEpiWarps) es += e_fixed(T, k, s2);
          // then, in the first share of a split tile, the others relative to it: each warp takes 1024
          // consecutive positions, sums their steps, and on a second pass their running sums
          const int w0 = warp * (kTilePos / kLinEpiWarps);
          long long e = 0;
          if (first) {
#pragma unroll 4
            for (int x = w0 + lane; x < w0 + kTilePos / kLinEpiWarps; x += 32)
              if (x > 0 && x < g.cnt) e += e_step(T, g.jA + x, L, s2);
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            es += __shfl_xor_sync(0xffffffffu, es, o);
            e += __shfl_xor_sync(0xffffffffu, e, o);
          }
          if (lane == 0) s.red[warp] = es, s.seg[warp] = e;
          named_sync<1, 32 * kLinEpiWarps>();
          long long run = 0;
          for (int w = 0; w < kLinEpiWarps; w++) run += s.red[w] + (w < warp ? s.seg[w] : 0);
#pragma unroll 4
          for (int x = w0 + lane; x - lane < min(w0 + kTilePos / kLinEpiWarps, g.cnt); x += 32) {
            long long v = first && x > 0 && x < g.cnt ? e_step(T, g.jA + x, L, s2) : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const long long y = __shfl_up_sync(0xffffffffu, v, o);
              if (lane >= o) v += y;
            }
            const int i = win_index(g.jA + x);
            if (x < g.cnt) add_y(i, run + v, false);
            run += __shfl_sync(0xffffffffu, v, 31);
          }
          __threadfence_block();  // the sums are read back by other threads of the block, after the barrier below
        }
        for (int pipe = 0; pipe < kPipes; pipe++)
          ok = ok && warp_wait(accf_b(pipe), sg & 1u, err, 100, *(volatile int *)&s.limit);
        ok = !named_any(1, 32 * kLinEpiWarps, !ok);  // one decision for all eight warps
        if (!ok) break;
        tc_fence_after();
        // (a segment of one chunk has nothing in the odd chunks' accumulators; the sum of both pipes'
        // is at most 2^24, still exact)
#pragma unroll
        for (int h = 0; h < 4; h++) {
          uint32_t d[2][kDig][8];
          const uint32_t t = tm0 + (uint32_t)(h * 8 * kDig);
#pragma unroll
          for (int m = 0; m < kDig; m++) {
            tmem_ld8(d[0][m], t + 8 * m);
            tmem_ld8(d[1][m], t + kAccCols + 8 * m);
          }
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 8; c++) {
            int v[kDig];
#pragma unroll
            for (int m = 0; m < kDig; m++)
              v[m] = __float2int_rn(__uint_as_float(d[0][m][c]) + (tb > ta ? __uint_as_float(d[1][m][c]) : 0.f));
            acc[8 * h + c] += (long long)v[0] + ((long long)v[1] << 12) + ((long long)v[2] << 24);
          }
        }
        tc_fence_before();
        mbar_arrive(acce_b());
      }
      if (!ok) break;
#pragma unroll
      for (int q = 0; q < 32; q++) {
        // column 32 half + q' holds a = 63 - (32 half + q'): ascending positions are descending columns
        const int x = x0 + q, j = g.jA + x, i = win_index(j);
        if (x < g.cnt) add_y(i, getbit(bits, j) ? -acc[31 - q] : acc[31 - q], true);
      }
      named_sync<1, 32 * kLinEpiWarps>();  // s.seg and s.red are free for the next item
    }
    if (ok && tid == 0) s.at = nitems;
  } else if (warp < kLinEpiWarps + kLinBuilders) {
    // ---------------- build G: a chunk per warp ----------------
    const int pipe = (warp - kLinEpiWarps) / kPipeBuilders, bw = (warp - kLinEpiWarps) % kPipeBuilders;
    uint32_t q0 = 0, c0 = 0;  // the pipe's products, and its chunks modulo its builders, of the items before
    bool ok = true;
    for (uint32_t n = s.first; ok && n < nitems; n += gridDim.x) {
      const HotItem it = items[n];
      const WalkDev &W = hdr[it.slot];
      const LinTile g = lin_tile(W, it);
      if (!g.ok) continue;
      const int L = g.L;
      const float2 *__restrict__ T = reinterpret_cast<const float2 *>(W.T);
      const float s4 = ldexpf(1.f, W.lin_sh - 2);
      // per-k values of a product: coefficient i = 2 pair + d of chunk t is that of u = 64 t - 63 + i, for
      // pairs lane and lane + 32 (127 coefficients)
      auto fetch = [&](int t, int dk, float2 (&v)[4]) {
#pragma unroll
        for (int d = 0; d < 4; d++) {
          const int i = 2 * (lane + 32 * (d >> 1)) + (d & 1), u = kP * t - (kP - 1) + i, k = u < 0 ? -u : u;
          v[d] = (k >= 1 && k < L && i < 2 * kP - 1) ? __ldg(T + 2 * k + dk) : make_float2(0.f, 0.f);
        }
      };
      float2 v[4];
      constexpr int kStep = kPipes * kPipeBuilders;
      int t = g.tau_lo + pipe + kPipes * ((bw + kPipeBuilders - (int)c0) % kPipeBuilders);
      if (t <= g.tau_hi) fetch(t, lin_kinds(g, t) == 2, v);
      for (; t <= g.tau_hi; t += kStep) {
        const int kinds = lin_kinds(g, t);
        uint32_t q = q0 + (uint32_t)(((t - g.tau_lo) >> 1) + lin_doubles(g, t, pipe));
        for (int dk = kinds == 2 ? 1 : 0; dk <= (kinds >> 1); dk++, q++) {
          // three digits of each coefficient, packed in pairs; w[r][m]: digit m of pair lane + 32 r
          uint32_t w[2][kDig], wo[2][kDig];
          const float sc = dk ? 2.f * s4 : s4;
#pragma unroll
          for (int r = 0; r < 2; r++) {
            float d[2][kDig];
#pragma unroll
            for (int e = 0; e < 2; e++) lin_digits(v[2 * r + e].y * sc, v[2 * r + e].x * sc, d[e]);
#pragma unroll
            for (int m = 0; m < kDig; m++)
              asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(w[r][m]) : "f"(d[1][m]), "f"(d[0][m]));
          }
          // the next product's values are on their way while this one is stored
          if (dk < (kinds >> 1))
            fetch(t, 1, v);
          else if (t + kStep <= g.tau_hi)
            fetch(t + kStep, lin_kinds(g, t + kStep) == 2, v);
          // the same digits one coefficient on (for the odd copies)
#pragma unroll
          for (int m = 0; m < kDig; m++) {
            const uint32_t na = __shfl_sync(0xffffffffu, lane == 0 ? w[1][m] : w[0][m], (lane + 1) & 31);
            const uint32_t nb = __shfl_down_sync(0xffffffffu, w[1][m], 1);
            wo[0][m] = __funnelshift_r(w[0][m], na, 16);
            wo[1][m] = __funnelshift_r(w[1][m], nb, 16);
          }
          const uint32_t st = q % kStages;
          if (q >= kStages) ok = warp_wait(empty_b(pipe, st), (q / kStages - 1u) & 1u, err, 100);
          ok = !__any_sync(0xffffffffu, !ok);
          if (!ok) break;
          // copy c of unit y holds coefficients 8 y + c ..: pair `pr` is the word at element
          // x = 2 pr - 2 c' of the copies 2 c' (as it is) and 2 c' + 1 (one coefficient on)
          const uint32_t h0 = h_s + (uint32_t)(pipe * kStages + st) * kHBytes;
#pragma unroll
          for (int r = 0; r < 2; r++)
#pragma unroll
            for (int c = 0; c < 4; c++) {
              const int x = 2 * (lane + 32 * r) - 2 * c;
              if (x >= 0 && x < 8 * kHCh) {
                const uint32_t a = h0 + (uint32_t)((x >> 3) * kHUnit + (x & 7) * 2 + 32 * c);
#pragma unroll
                for (int m = 0; m < kDig; m++) {
                  sts32(a + (uint32_t)(kHDig * m), w[r][m]);
                  sts32(a + (uint32_t)(kHDig * m + 16), wo[r][m]);
                }
              }
            }
          fence_proxy_async();
          mbar_arrive(full_b(pipe, st));
        }
        if (!ok) break;
      }
      const int nc = (g.tau_hi - g.tau_lo + kPipes - pipe) / kPipes;  // the pipe's chunks
      c0 = (c0 + (uint32_t)nc) % kPipeBuilders;
      q0 += (uint32_t)(nc + lin_doubles(g, g.tau_hi + 1, pipe));
    }
  } else if (lane == 0) {
    // ---------------- issue a pipe's products ----------------
    const int pipe = warp - kLinEpiWarps - kLinBuilders;
    const uint32_t d = tmem + (uint32_t)pipe * kAccCols, hp_s = h_s + (uint32_t)(pipe * kStages) * kHBytes,
                   sp_s = stile_s + (uint32_t)(pipe * kSTiles) * kSTileBytes;
    uint32_t st = 0, ph = 0, ss = 0, sph = 0, sg = 0;  // stage and S tile with their phases, segment
    uint32_t nacc = 0;                                 // segments announced
    bool ok = true, ready = false;                     // the stage is full
    for (uint32_t n = s.first; ok && n < nitems; n += gridDim.x) {
      const HotItem it = items[n];
      const LinTile g = lin_tile(hdr[it.slot], it);
      if (!g.ok) continue;
      for (int t0 = g.tau_lo; ok && t0 <= g.tau_hi; t0 += kSegTau, sg++) {
        const uint32_t buf = sg & 1u;
        if (sg >= 1) ok = wait_or_err(acce_b(), (sg - 1u) & 1u, err);
        if (ok) ok = wait_or_err(win_b(buf), (sg >> 1) & 1u, err);
        if (!ok) break;
        bool acc = false;
        const int t1 = min(g.tau_hi, t0 + kSegTau - 1);
        uint32_t aw = win_s + buf * kWinBytes + 16u * (uint32_t)pipe;
        for (int t = t0 + pipe; ok && t <= t1; t += kPipes, aw += 16u * kPipes) {
          const bool both = lin_kinds(g, t) == 3;
          for (int rep = both ? 2 : 1; ok && rep > 0; rep--) {
            const uint32_t a0 = both ? sp_s + ss * kSTileBytes : aw, lbo = both ? kSPlane : kWinPlane;
            const uint64_t da = smem_desc(a0, lbo, 128u), db = smem_desc(hp_s + st * kHBytes, kHUnit, kHDig);
            if (!ready) ok = wait_or_err(full_b(pipe, st), ph, err);
            if (ok && both) ok = wait_or_err(sfull_b(pipe, ss), sph, err);
            if (!ok) break;
            tc_fence_after();
            const uint32_t st0 = st, ss0 = ss;
            mma_f16(d, da, db, acc);
            mma_f16(d, da + (2u * lbo >> 4), db + (2u * kHUnit >> 4), true);
            // while these run: is the next stage of G there already?
            if (++st == kStages) st = 0, ph ^= 1u;
            ready = mbar_try_wait(full_b(pipe, st), ph);
            mma_f16(d, da + 2u * (2u * lbo >> 4), db + 2u * (2u * kHUnit >> 4), true);
            mma_f16(d, da + 3u * (2u * lbo >> 4), db + 3u * (2u * kHUnit >> 4), true);
            acc = true;
            mma_commit(empty_b(pipe, st0));
            if (both) {
              mma_commit(sempty_b(pipe, ss0));
              if (++ss == kSTiles) ss = 0, sph ^= 1u;
            }
          }
        }
        if (ok && !g.stall) mma_commit(accf_b(pipe)), nacc++;
      }
    }
    // nothing is in flight when the accumulators are given back or the barriers set up again: no product, and no
    // arrival of a commit (the last one on each barrier; a parity that no commit has reached yet reads complete)
    mma_commit(drain_b(pipe));
    bool done = mbar_wait_bounded(drain_b(pipe), 0) && mbar_wait_bounded(accf_b(pipe), (nacc - 1u) & 1u);
    for (uint32_t q = 0; q < kStages; q++) done = done && mbar_wait_bounded(empty_b(pipe, q), q < st ? ph : ph ^ 1u);
    for (uint32_t q = 0; q < kSTiles; q++) done = done && mbar_wait_bounded(sempty_b(pipe, q), q < ss ? sph : sph ^ 1u);
    if (!done) s.pending = s.err = 1;
  }
  __syncwarp();
}

}  // namespace

__global__ void __launch_bounds__(kLinThreads, 1) k_lin(WalkDev *hdr, const HotItem *all_items, const Schedule *sched) {
  if (threadIdx.x == 0) {
    lin_init_bars();
    s_lin.first = blockIdx.x;
  }
  const bool alloc = threadIdx.x / 32 == kLinEpiWarps + kLinBuilders;
  if (alloc) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(&s_lin.tmem))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const HotItem *items = all_items + sched->nitems + sched->nquad;
  const uint32_t nitems = sched->nlin;
  for (;;) {  // (a second time only after a wait ran out)
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    lin_items(hdr, items, nitems);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (!s_lin.err) break;
    const uint32_t at = s_lin.at;
    const bool pending = s_lin.pending != 0;
    if (threadIdx.x == 0)
      for (uint32_t n = at; n < nitems && (pending || n == at); n += gridDim.x)
        hdr[items[n].slot].error = (uint32_t)-5;  // PSL_ETIMEOUT of the library header
    __syncthreads();  // every thread has read the flags
    if (pending) break;
    if (threadIdx.x == 0) {
      for (uint32_t b = 0; b < kLinBars; b++) mbar_inval(lin_bars() + 8u * b);
      lin_init_bars();
      s_lin.first = at + gridDim.x;
    }
  }
  if (alloc)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(s_lin.tmem) : "memory");
}

// ------------------------------------------------------------------------------------
// k_quad: sum_{k <= kin} A_k [s_{j+k} = s_{j-k}] by subset-sum tables, the correction of the B / D
// boundary, and the final score.  The structure is that of k_hot_pc: two producer warps stage each
// tile of 32 super-blocks (30 shifts) by TMA and build its tables (one per group of five shifts,
// 768 bytes per super-block, entries swizzled by the super-block as there), scorer warps look up.
// ------------------------------------------------------------------------------------
namespace {

constexpr int kQWarps = 14;                 // scorer warps: 448 window positions per item
constexpr int kQProducers = 2;
constexpr int kQThreads = 32 * (kQWarps + kQProducers);
constexpr int kQNsb = 32;                   // super-blocks per tile
constexpr int kQTileK = kQNsb * kSbK;
constexpr int kQSbb = 6 * 128;              // table bytes per super-block
constexpr int kQFb = 8;                     // super-blocks per block sum
constexpr size_t kQSmem = 128 + 2 * ((size_t)kQNsb * kQSbb + (size_t)kQTileK * 16);
static_assert(32 * kQWarps == (int)kQuadPos, "positions per item shared with the host's item list");

enum QFlags : uint32_t { kQFirst = 1, kQLast = 2, kQEmpty = 4, kQSkip = 8 };
constexpr uint32_t kQEnd = 0xffffffffu;
struct QTile {
  uint32_t item;
  int32_t kt0;
  uint32_t flags, pad;
};

// table of one group: entry b holds the sum of A over the shifts of b
__device__ __forceinline__ void quad_build(float *tab, int sb, int q, const float4 *Ts, int kt0, int kg, int L) {
  float a[5];
#pragma unroll
  for (int t = 0; t < 5; t++) {
    a[t] = 0.f;
    if (kg + t < L) {
      const float2 v = *reinterpret_cast<const float2 *>(Ts + (kg + t - kt0));
      a[t] = 0.5f * (v.x + v.y);
    }
  }
  const float lo[4] = {0.f, a[0], a[1], a[0] + a[1]};
  const float p = a[2] + a[3];
  const float hi[8] = {0.f, a[2], a[3], p, a[4], a[2] + a[4], a[3] + a[4], p + a[4]};
  float *base = tab + sb * (kQSbb / 4) + q * 32;
  const int sw = sb & 31;
#pragma unroll
  for (int b = 0; b < 32; b++) base[b ^ sw] = lo[b & 3] + hi[b >> 2];
}

// X holds the 30 shifts' bits from bit 2 on (the partner windows are read two positions early), so that
// field q is a table's byte offset after one shift by 5 q.  The sums go in pairs (add.f32x2).
__device__ __forceinline__ void quad_lookup(float2 &a, uint32_t X, uint32_t bsw) {
  const float v0 = lds_at<0>((X & 0x7Cu) ^ bsw), v1 = lds_at<128>(((X >> 5) & 0x7Cu) ^ bsw);
  a = __fadd2_rn(a, make_float2(v0, v1));
  const float v2 = lds_at<256>(((X >> 10) & 0x7Cu) ^ bsw), v3 = lds_at<384>(((X >> 15) & 0x7Cu) ^ bsw);
  a = __fadd2_rn(a, make_float2(v2, v3));
  const float v4 = lds_at<512>(((X >> 20) & 0x7Cu) ^ bsw), v5 = lds_at<640>(((X >> 25) & 0x7Cu) ^ bsw);
  a = __fadd2_rn(a, make_float2(v4, v5));
}

// sum over p in [lo, hi) of (B - D)_{|p-j|} s_p, flushed every 16 terms
__device__ __forceinline__ float band_sum(const uint32_t *__restrict__ bits, const float4 *__restrict__ T, int j, int lo,
                                          int hi) {
  float sum = 0.f, c = 0.f, blk = 0.f;
  for (int p = lo; p < hi; p++) {
    const float4 v = __ldg(T + (p > j ? p - j : j - p));
    const float d = 0.25f * (v.y - v.x) - 0.5f * (v.w - v.z);
    blk += getbit(bits, p) ? -d : d;
    if (((p - lo) & 15) == 15) flush_block(sum, c, blk);
  }
  flush_block(sum, c, blk);
  return sum + c;
}

// k_lin takes B for a partner of row j0 (64 positions) and chunk p0 iff 2 j0 - (L-1) <= p0 <= 2 j0;
// the exact condition is 2j - (L-1) <= p <= 2j.  The terms where the two differ, times s_j:
__device__ __forceinline__ float band_fix(const uint32_t *__restrict__ bits, const float4 *__restrict__ T, int j, int j0,
                                          int L) {
  const int hi_t = min(2 * j, L - 1), hi_r = min(j0 + kP * floor_div64(j0) + kP - 1, L - 1);
  const int lo_t = max(2 * j - (L - 1), 0), lo_r = max(j0 - kP * floor_div64(L - 1 - j0), 0);
  float r = hi_t > hi_r ? band_sum(bits, T, j, hi_r + 1, hi_t + 1) : -band_sum(bits, T, j, hi_t + 1, hi_r + 1);
  r += lo_t < lo_r ? band_sum(bits, T, j, lo_t, lo_r) : -band_sum(bits, T, j, lo_r, lo_t);
  return getbit(bits, j) ? -r : r;
}

}  // namespace

__global__ void __launch_bounds__(kQThreads, 2) k_quad(WalkDev *hdr, const HotItem *items, Schedule *sched) {
  extern __shared__ __align__(128) float smem_q[];
  items += sched->nitems;
  const uint32_t nquad = sched->nquad;
  __shared__ __align__(8) uint64_t s_bar[6];  // full[2], empty[2], copy[2]
  __shared__ QTile s_hdr[2];
  __shared__ uint32_t s_item;
  __shared__ int s_pflag, s_prun, s_pstall;
  const uint32_t raw_s = (uint32_t)__cvta_generic_to_shared(smem_q);
  const uint32_t tab_s0 = (raw_s + 127u) & ~127u;
  float *tab0 = smem_q + (tab_s0 - raw_s) / 4;
  float4 *stage0 = reinterpret_cast<float4 *>(tab0 + 2 * kQNsb * (kQSbb / 4));
  const uint32_t stage_s0 = tab_s0 + 2 * kQNsb * kQSbb;
  const uint32_t bar_s = (uint32_t)__cvta_generic_to_shared(s_bar);
  auto full_b = [&](int b) { return bar_s + 8u * (uint32_t)b; };
  auto empty_b = [&](int b) { return bar_s + 16u + 8u * (uint32_t)b; };
  auto copy_b = [&](int b) { return bar_s + 32u + 8u * (uint32_t)b; };
  const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; b++) {
      mbar_init(full_b(b), 1);
      mbar_init(empty_b(b), kQWarps);
      mbar_init(copy_b(b), 1);
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp >= kQWarps) {
    // ---------------------------------- producer ----------------------------------
    const int ptid = (int)threadIdx.x - 32 * kQWarps;
    auto psync = [] { named_sync<1, 32 * kQProducers>(); };
    uint32_t s = 0;                     // tile sequence number (buffer s & 1, use s >> 1)
    uint32_t ncopy0 = 0u, ncopy1 = 0u;  // copies issued into each staging buffer
    bool ok = true;
    // a bounded wait decided by one producer thread, so that both warps take the same branch
    auto pwait = [&](uint32_t mbar, uint32_t parity, int limit) {
      if (ptid == 0) s_pflag = mbar_wait_bounded(mbar, parity, limit) ? 1 : 0;
      psync();
      const bool r = s_pflag != 0;
      if (r && ptid != 0) mbar_wait_bounded(mbar, parity, 1 << 20);
      psync();
      return r;
    };
    auto publish = [&](uint32_t item, int kt0, uint32_t flags) {
      const int b = (int)(s & 1u);
      if (ptid == 0) {
        s_hdr[b].item = item;
        s_hdr[b].kt0 = kt0;
        s_hdr[b].flags = flags;
        mbar_arrive(full_b(b));
      }
      s++;
    };
    auto claim = [&]() {
      const int b = (int)(s & 1u);
      return s < 2 || pwait(empty_b(b), ((s >> 1) - 1u) & 1u, 1 << 20);
    };
    for (;;) {
      if (ptid == 0) {
        const uint32_t nx = atomicAdd(&sched->quad_next, 1u);
        s_item = nx;
        s_prun = 0, s_pstall = 0;
        if (nx < nquad) {
          WalkDev &Wn = hdr[items[nx].slot];
          if (Wn.error) Wn.status = kError;  // k_lin ran out a wait over the walk
          s_prun = Wn.status == kRunning ? 1 : 0;
          s_pstall = Wn.inject_stall ? 1 : 0;
        }
      }
      psync();
      const uint32_t item = s_item;
      const bool run = s_prun != 0, stall = s_pstall != 0;
      psync();
      if (item >= nquad) break;
      const HotItem it = items[item];
      WalkDev &W = hdr[it.slot];
      if (!run) {
        if (!(ok = claim())) break;
        publish(item, 0, kQFirst | kQLast | kQEmpty | kQSkip);
        continue;
      }
      const int L = (int)W.L, N = (int)W.N;
      // largest kin over the item's positions start + i0 .. start + min(i0 + 447, N), modulo L
      const int a = (int)(((uint64_t)W.start + (uint64_t)it.i0) % (uint64_t)L);
      const int cnt = min((int)it.i0 + 32 * kQWarps - 1, N) - (int)it.i0 + 1;
      auto seg_kin = [&](int x, int y) {
        const int m = min(max((L - 1) / 2, x), y);
        return max(min(m, L - 1 - m), max(min(x, L - 1 - x), min(y, L - 1 - y)));
      };
      const int kmax = a + cnt - 1 < L ? seg_kin(a, a + cnt - 1) : max(seg_kin(a, L - 1), seg_kin(0, a + cnt - 1 - L));
      const int per = (int)W.kchunk_sb / kQNsb;  // tiles per k-chunk
      const int tile_lo = W.ksplit > 1 ? (int)it.kc * per : 0;
      const int tiles = (kmax + kQTileK - 1) / kQTileK;
      const int ntiles = max(0, (W.ksplit > 1 ? min(tiles, tile_lo + per) : tiles) - tile_lo);
      if (ntiles == 0) {
        // the test hook lets one wait run out even where there is nothing to copy
        const bool dead = stall && (!pwait(copy_b(0), ncopy0 & 1u, 64));
        if (dead && ptid == 0) {
          W.error = (uint32_t)-5;
          W.status = kError;
        }
        if (!(ok = claim())) break;
        publish(item, 0, kQFirst | kQLast | kQEmpty | (dead ? kQSkip : 0u));
        continue;
      }
      bool failed = false;
      for (int tile = 0; tile < ntiles; tile++) {
        const int kt0 = 1 + (tile_lo + tile) * kQTileK;
        const uint32_t flags = (tile == 0 ? kQFirst : 0u) | (tile + 1 == ntiles ? kQLast : 0u);
        if (!(ok = claim())) break;
        const int b = (int)(s & 1u);
        if (failed) {
          publish(item, kt0, flags | kQEmpty | kQSkip);
          continue;
        }
        if (ptid == 0 && !stall) {
          const uint32_t bytes = 16u * (uint32_t)min(kQTileK, L - kt0);
          fence_proxy_async();
          mbar_expect_tx(copy_b(b), bytes);
          tma_load_1d(stage_s0 + (uint32_t)b * (kQTileK * 16), W.T + kt0, bytes, copy_b(b));
        }
        if (!stall) (b ? ncopy1 : ncopy0)++;
        const uint32_t nc = b ? ncopy1 : ncopy0;
        const bool got = stall ? pwait(copy_b(b), nc & 1u, 64) : pwait(copy_b(b), (nc - 1u) & 1u, 1 << 20);
        if (!got) {
          if (ptid == 0) {
            W.error = (uint32_t)-5;  // PSL_ETIMEOUT of the library header
            W.status = kError;
          }
          if (!stall) {  // a copy that may still be in flight: stop using this block
            ok = false;
            break;
          }
          failed = true;
          publish(item, kt0, flags | kQEmpty | kQSkip);
          continue;
        }
        const float4 *Ts = stage0 + b * kQTileK;
        for (int g = ptid; g < 6 * kQNsb; g += 32 * kQProducers) {
          const int sb = g % kQNsb, q = g / kQNsb, ka = kt0 + sb * kSbK;
          if (ka <= kmax) quad_build(tab0 + b * kQNsb * (kQSbb / 4), sb, q, Ts, kt0, ka + 5 * q, L);
        }
        psync();
        publish(item, kt0, flags);
      }
      if (!ok) break;
    }
    if (ok && claim()) {
      publish(kQEnd, 0, 0);
    } else if (ptid == 0) {
      for (int b = 0; b < 2; b++) {
        s_hdr[b].item = kQEnd;
        mbar_arrive(full_b(b));
      }
    }
    return;
  }

  // ---------------------------------- scorers ----------------------------------
  uint32_t s = 0, cur = kQEnd;
  WalkDev *Wp = nullptr;
  int i = 0, j = 0, kin = 0, kin_lo = 0, kin_hi = 0, L = 0, N = 0;
  bool live = false, skip = false;
  float hi = 0.f, lo = 0.f;
  float2 a = make_float2(0.f, 0.f);
  for (;;) {
    const int b = (int)(s & 1u);
    const bool got = mbar_wait_bounded(full_b(b), (s >> 1) & 1u);
    if (__any_sync(0xffffffffu, !got)) {
      if (cur != kQEnd && lane == 0 && Wp) {
        Wp->error = (uint32_t)-5;
        Wp->status = kError;
      }
      break;
    }
    const QTile h = s_hdr[b];
    if (h.item == kQEnd) break;
    if (h.flags & kQFirst) {
      cur = h.item;
      const HotItem it = items[cur];
      Wp = hdr + it.slot;
      skip = false;
      hi = lo = a.x = a.y = 0.f;
      if (!(h.flags & kQSkip)) {
        const WalkDev &W = *Wp;
        L = (int)W.L, N = (int)W.N;
        i = (int)it.i0 + 32 * warp + lane;
        live = i <= N;
        j = (int)(((uint64_t)W.start + (uint64_t)min(i, N)) % (uint64_t)L);
        kin = min(j, L - 1 - j);
        const bool warp_live = (int)it.i0 + 32 * warp <= N;
        kin_lo = __reduce_min_sync(0xffffffffu, kin);
        kin_hi = warp_live ? __reduce_max_sync(0xffffffffu, kin) : 0;
      }
    }
    if (h.flags & kQSkip) skip = true;
    if (!(h.flags & kQEmpty) && !skip) {
      const uint32_t *__restrict__ win_f = Wp->win_f;
      const uint32_t *__restrict__ win_r = Wp->win_r;
      const int kt0 = h.kt0;
      const int n_all = sb_count(kin_hi, kt0, 0, kQNsb);
      const int n_int = min(sb_count(kin_lo, kt0, kSbK - 1, kQNsb), n_all);
      uint32_t bsw = tab_s0 + (uint32_t)b * (kQNsb * kQSbb);
      int sb = 0;
      const uint32_t *wu = win_f + (j + kt0 - 2), *wv = win_r + (j - kt0 + 2);
      // every lane has both partners; at most 24 additions into either accumulator per flush
      for (; sb + kQFb - 1 < n_int; sb += kQFb) {
#pragma unroll
        for (int u = 0; u < kQFb; u++)
          quad_lookup(a, ~(__ldg(wu + u * kSbK) ^ __ldg(wv - u * kSbK)), bsw + u * (kQSbb + 4));
        flush2(hi, lo, a.x, a.y);
        wu += kQFb * kSbK, wv -= kQFb * kSbK, bsw += kQFb * (kQSbb + 4);
      }
      // the rest masked to each lane's k <= kin: the empty subset's entry is 0
      for (; sb < n_all; sb++) {
        const int ka = kt0 + sb * kSbK;
        const uint32_t U = __ldg(win_f + min(j + ka, L) - 2), V = __ldg(win_r + max(j - ka, -1) + 2);
        const int nk = min(kSbK, max(0, kin - ka + 1));
        quad_lookup(a, ~(U ^ V) & (((1u << nk) - 1u) << 2), bsw);
        if ((sb & 7) == 7) flush2(hi, lo, a.x, a.y);
        bsw += kQSbb + 4;
      }
      flush2(hi, lo, a.x, a.y);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(empty_b(b));  // this warp is done with the buffer
    if ((h.flags & kQLast) && !skip && live) {
      WalkDev &W = *Wp;
      const uint32_t kc = items[cur].kc;
      if (W.ksplit <= 1 || kc == W.kc_psl) {
        // the boundary terms and k_lin's sum (cleared for the next step's shares)
        const int f = ((int)W.start + 1) % L;
        const int off = N == L ? j : (j >= f ? j - f : j);  // offset in the row grid of k_lin's tiles
        float fix = band_fix(W.bits, W.T, j, j - (off & (kP - 1)), L);
        flush_block(hi, lo, fix);
        long long *Y = lin_y(W) + (i - 1);
        const long long y = *Y;
        *Y = 0;
        const float sc = ldexpf(1.f, -W.lin_sh);
        const float y0 = __ll2float_rn(y);
        float y1 = y0 * sc;
        flush_block(hi, lo, y1);
        lo += __ll2float_rn(y - __float2ll_rn(y0)) * sc;
        // exact neighbour PSL, only when some neighbour may beat psl_best
        int pj = INT_MAX;
        if (W.ktau_on) pj = neighbour_psl(W, W.ktau, (int)W.nktau, j, L, getbit(W.bits, j) ? -1 : 1, W.psl - 8, 0);
        W.pslj[i - 1] = pj;
      }
      if (W.ksplit > 1)
        W.score_part[(size_t)kc * N + (i - 1)] = hi + lo;
      else
        W.score[i - 1] = hi + lo;
    }
    s++;
  }
}

static uint32_t g_quad_per_sm = 1;

cudaError_t prepare_lin_kernels() {
  cudaError_t e = cudaFuncSetAttribute(k_lin, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLinSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_quad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQSmem);
  int nb = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_quad, kQThreads, kQSmem);
  g_quad_per_sm = (uint32_t)(nb > 0 ? nb : 1);
  return e;
}

cudaError_t launch_hot_lin(const LaunchCtx &c) {
  k_lin<<<c.sm_count, kLinThreads, kLinSmem, c.stream>>>(c.hdr, c.items, c.sched);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_quad<<<g_quad_per_sm * c.sm_count, kQThreads, kQSmem, c.stream>>>(c.hdr, c.items, c.sched);
  return cudaGetLastError();
}

}  // namespace psl
