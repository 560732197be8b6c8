// Error-free split-BF16 ladder (LADDER_OZAKI): the two-pass form of the
// tensor-core path with an error-free splitting of every operand, after the
// scheme of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012), so that
// R and E_L come out with FP64-class accuracy from BF16 tensor-core products.
//
// R_ij^ab = sum_cd (ac|bd) tau_ij^cd (Eq. pp-Ladder-0), (ac|bd) = sum_P
// B^P_ac B^P_bd (Eq. RIM), in the slot form of the symmetric / antisymmetric
// pair scheme (Sec. II.C) used by the other tensor-core kernels: virtual
// indices in blocks of 8, block pairs k <= l, V+-_ab[(c,d)] = (ac|bd) +-
// (ad|bc), R+- = sum T+- V+-.
//
// Splitting.  A row x of an operand (the K index running along it) is held as
// S slices of fixed-point numbers under one power-of-two scale per row:
//   x = scale * sum_s x_s 2^(-8 s),  x_0 in [-256, 256], x_s in [-128, 128],
// each x_s an integer, stored as the BF16 number x_s 2^(-8 s) (exact: at most
// 8 significant bits).  A product of slices p and q is exact in FP32 and is an
// integer multiple of 2^(-8 (p + q)) below 2^16 of that unit.
//
// Accumulation.  The tensor core rounds its FP32 accumulator with a bias, so a
// sum of products is exact only while every partial sum is representable.  A
// TMEM accumulator here receives products of one slice order p + q only
// (orders 0, 1 and 2 each in their own, orders >= 3 together, 2^-24 below the
// result where rounding no longer matters), over an exactness window short
// enough that its partial sums stay below 2^24 units:
//   GEMM1 (K = aux functions): windows of 192 (6 K-steps of 32; order 2 sums at
//         most 2 x 256 x 128 + 128 x 128 = 81920 units per function, so 204
//         would do); every row of B has one scale over all P, so windows add
//         without rescaling.  Against windows of 128 a third fewer drains:
//         o=10, v=120, N=480 1414 -> 1395 us a step, o=16, v=200, N=800 with
//         general B 22.1 -> 21.4 ms;
//   GEMM2 (K = slots): one block pair (64 slots) per window; V+- and tau+-
//         rows have one scale per block pair, applied when the window's four
//         accumulators are drained.
// The conversion warps drain each window's four accumulators into a
// double-single sum (an FP32 pair kept with TwoSum, about 48 bits).
//
// Pass 1 (oz_vstore_kernel): per (ab tile, block pair): X = (ac|bd) and
// Y = (ad|bc) windows alternate and take two TMEM halves in turn (X drains while
// Y's MMAs run, and on a diagonal block pair, which has no Y, X's own next ones:
// o=16, v=200 with general B 21.2 -> 20.6 ms); at the end V+- = X +- Y' (Y transposed across lanes), cut into S
// fixed-point slices with one scale per (ab row, block pair), stored to the
// workspace with their scales.  Pass 2 (oz_gemm2_kernel): per (tile, chunk of
// <= 128 occupied pairs of one sign, block-pair range): the S x S slice
// products of every 16-slot piece with p + q < S, issued and drained by order
// group so that draining one group overlaps the MMAs of the other.  The unpack kernel of the two-pass form then writes R.
//
// Warp roles (576 threads): warp 0 TMA producer, warp 1 MMA issuer (in step, one
// elected lane), warps 2-17 conversion (four per TMEM lane quadrant, each owning a
// quarter of the columns).
#include <algorithm>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace ladder {
namespace {
using namespace tc;

constexpr int kThreads = 576;
constexpr int kEpi = 512;
constexpr int KSTEP = 32;                             // aux functions per GEMM1 stage
constexpr uint32_t A_TILE = 128u * KSTEP * 2u;        // 8 KB: rows (a,c), 64-byte rows
constexpr uint32_t B_TILE = 64u * KSTEP * 2u;         // 4 KB: rows (b,d)
constexpr int TPIECE = 16;                            // slots per GEMM2 piece
constexpr uint32_t VP_PLANE = 128u * TPIECE * 2u;     // 4 KB: 128 ab rows x 16 slots
constexpr uint32_t kSmemBudget = 230400u;             // ring bytes available per CTA

// s + e = a + b exactly (Knuth's TwoSum), two FP32 lanes at once (f32x2), each
// rounded exactly like the scalar instruction
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e) {
  s = add2(a, b);
  const float2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}
// The same where a is a multiple of the last place of b: three operations do
// (Dekker's Fast2Sum; if a is the smaller one, the sum is rounded by at most one
// last place of b, so s - a is a representable multiple of it)
__device__ __forceinline__ void fast_two_sum2(float2 a, float2 b, float2 &s, float2 &e) {
  s = add2(a, b);
  e = sub2(b, sub2(s, a));
}
// (H, L) += (h, l), two accumulators at once (as ds_acc)
__device__ __forceinline__ void ds_acc2(float2 &H, float2 &L, float2 h, float2 l) {
  float2 s, e;
  two_sum2(H, h, s, e);
  H = s;
  L = add2(L, add2(l, e));
}
// One exactness window of pass 1 into the double-single sums of 16 columns,
// two columns per f32x2 instruction.  The window's value comes from its four
// order accumulators g0..g3 (TMEM columns cbase + 64 g) as a double-single
// (h, l) with |l| <= ulp(h) / 2.  In units of the order-0 products, g0 is an
// integer and |g1| < 2^16, so h0 + e = g0 + g1 exactly (Fast2Sum); e is a
// multiple of 2^-8 of at most 1/2 and g2 one of 2^-16 of at most 240 (192 x
// 81920 units), so e + g2 is exact in FP32, and h0, a multiple of 2^-8, of its
// last place: the second Fast2Sum leaves a remainder of at most ulp(h) / 2, to
// which the tail orders (2^-24 below h) are added with a rounding 2^-48 below h.
// (Adding g2 straight into the low word would round it 2^-40 below h.)  (h, l)
// then goes into the running sum as ds_acc2 does.  The FP32 pipe bounds the
// drains: 17 operations for two columns (23 with TwoSum throughout).
__device__ __forceinline__ void drain_window(uint32_t cbase, float2 (&acc)[16]) {
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    float g0[4], g1[4], g2[4], g3[4];
    const uint32_t c0 = cbase + 4u * h;
    tmem_ld4(c0, g0);
    tmem_ld4(c0 + 64u, g1);
    tmem_ld4(c0 + 128u, g2);
    tmem_ld4(c0 + 192u, g3);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 4; e += 2) {
      float2 h0, er, hh, ll;
      fast_two_sum2(make_float2(g0[e], g0[e + 1]), make_float2(g1[e], g1[e + 1]), h0, er);
      fast_two_sum2(h0, add2(er, make_float2(g2[e], g2[e + 1])), hh, ll);
      ll = add2(ll, make_float2(g3[e], g3[e + 1]));
      float2 H = make_float2(acc[4 * h + e].x, acc[4 * h + e + 1].x);
      float2 L = make_float2(acc[4 * h + e].y, acc[4 * h + e + 1].y);
      ds_acc2(H, L, hh, ll);
      acc[4 * h + e] = make_float2(H.x, L.x);
      acc[4 * h + e + 1] = make_float2(H.y, L.y);
    }
  }
}

// 2^e as a float for -126 <= e <= 127
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// Exponent E with m < 2^E for m > 0 (m finite, normal).
__device__ __forceinline__ int exp_above(float m) { return ((__float_as_int(m) >> 23) & 0xff) - 126; }

// 8x8 transpose across the 8 lanes of a group (lane x holds row x on entry,
// column x on exit).
__device__ __forceinline__ void transpose8(float (&r)[8], int x) {
#pragma unroll
  for (int s = 1; s < 8; s <<= 1) {
    const bool up = (x & s) != 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j & s) continue;
      const float send = up ? r[j] : r[j ^ s];
      const float recv = __shfl_xor_sync(0xffffffffu, send, s);
      if (up)
        r[j] = recv;
      else
        r[j ^ s] = recv;
    }
  }
}

__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo_bytes, uint32_t layout) {
  return ((sbo_bytes >> 4) & 0x3FFFu) | (1u << 14) | (layout << 29);
}
__device__ __forceinline__ uint64_t desc64(uint32_t saddr, uint32_t hi) {
  return ((uint64_t)hi << 32) | (uint64_t)(((saddr >> 4) & 0x3FFFu) | (1u << 16));
}

struct DrainWatch {
  int zero = 0;
  Watchdog wd;
  __device__ DrainWatch(int *status, uint64_t deadline) : wd{status, &zero, deadline} {}
};

// Work unit (tile, chunk, range) as in the other tensor-core kernels: tile =
// (a 16-block iA, b 8-block jB >= 2 iA), range [p0, p1) of block pairs.
struct Item {
  int tile, ch, A0, B0, p0, p1;
  TcChunk CH;
  float2 *racc;
};
__device__ __forceinline__ Item decode(const OzArgs &A, int slot, int nchunks) {
  Item I;
  const int ksl = slot % A.ksplit;
  const int tc = slot / A.ksplit;
  const int tile = tc / nchunks;
  I.ch = tc % nchunks;
  int iA = 0, t = tile + A.tile0;  // tile0: first tile of the plan's range
  while (t >= A.nB8 - 2 * iA) {
    t -= A.nB8 - 2 * iA;
    ++iA;
  }
  I.tile = tile;
  I.A0 = iA * 16;
  I.B0 = (2 * iA + t) * CB;
  I.CH = A.chunks[I.ch];
  I.p0 = (int)((long long)A.nbp * ksl / A.ksplit);
  I.p1 = (int)((long long)A.nbp * (ksl + 1) / A.ksplit);
  I.racc = A.racc ? A.racc + (size_t)slot * 128 * A.racc_cols : nullptr;
  return I;
}

// The molecule's arguments and the local unit index of work unit u: a single
// molecule reads them from the launch parameters, a batch from its device table.
template <bool kBatch>
__device__ __forceinline__ const OzArgs &oz_args(const OzLaunch &Lp, int u, int &local) {
  if constexpr (!kBatch) {
    local = u;
    return Lp.one;
  } else {
    const int2 w = Lp.items[u];
    local = w.y;
    return Lp.mols[w.x];
  }
}
// Pass 1 units walk range-major (unit u: range u / tiles of tile u % tiles) so
// the resident CTAs share B panels in L2; pass 2 likewise over (tile, chunk).
__device__ __forceinline__ int vstore_slot(const OzArgs &A, int u) {
  return (u % A.ntiles) * A.ksplit + u / A.ntiles;
}
__device__ __forceinline__ int gemm2_slot(const OzArgs &A, int u) {
  const int tcs = A.ntiles * A.nchunks;
  return (u % tcs) * A.ksplit + u / tcs;
}

struct Bars {
  uint32_t base;
  int stages;
  __device__ uint32_t full(int s) const { return base + 8u * s; }
  __device__ uint32_t empty(int s) const { return base + 8u * (stages + s); }
  __device__ uint32_t cfull(int b) const { return base + 8u * (2 * stages + b); }
  __device__ uint32_t cfree(int b) const { return base + 8u * (2 * stages + 3 + b); }
  __device__ uint32_t done() const { return base + 8u * (2 * stages + 6); }
  static constexpr int kCount = 7;  // + 2 * stages
};

template <int S>
struct Cfg1 {
  static constexpr uint32_t kStage = (uint32_t)S * (A_TILE + B_TILE);
  static constexpr int kStages = (int)(kSmemBudget / kStage);
  static constexpr uint32_t kRing = kStage * kStages;
  static constexpr uint32_t kSmem = kRing + 256 + 1024;
};
// Pass 2's ring, in two parts: slices 0..2 (L) and 3..S-1 (H) of a 16-slot
// piece of V+- (4 KB a slice) and of the chunk's sc rows of tau+-.  The stages
// are as small as the chunk allows: n of H and n + 1 of L.
template <int S>
struct Cfg2 {
  static constexpr int kLow = 3, kHigh = S - kLow;
  static constexpr int kMaxL = 10;
  static constexpr uint32_t kRing = 229376u;  // n = 5 at S = 5, n = 4 at S = 6 for 128 rows
  static constexpr uint32_t kBars = 8u * (4 * kMaxL + 7);
  static constexpr uint32_t kSmem = kRing + 512 + 1024;
};
struct Ring2 {
  uint32_t lbytes, hbytes, hbase;  // stage sizes, start of H in the ring
  int nL, nH;
  template <int S>
  __device__ static Ring2 of(uint32_t sc) {
    using C = Cfg2<S>;
    Ring2 r;
    const uint32_t slice = VP_PLANE + sc * 32u;
    r.lbytes = C::kLow * slice;
    r.hbytes = C::kHigh * slice;
    r.nH = min(C::kMaxL - 1, (int)((C::kRing - r.lbytes) / (r.lbytes + r.hbytes)));
    r.nL = r.nH + 1;
    r.hbase = r.nL * r.lbytes;
    return r;
  }
};
struct Bars2 {
  uint32_t base;
  static constexpr int kMax = 10;
  __device__ uint32_t fullL(int s) const { return base + 8u * s; }
  __device__ uint32_t emptyL(int s) const { return base + 8u * (kMax + s); }
  __device__ uint32_t fullH(int s) const { return base + 8u * (2 * kMax + s); }
  __device__ uint32_t emptyH(int s) const { return base + 8u * (3 * kMax + s); }
  __device__ uint32_t cfull(int b) const { return base + 8u * (4 * kMax + b); }
  __device__ uint32_t cfree(int b) const { return base + 8u * (4 * kMax + 3 + b); }
  __device__ uint32_t done() const { return base + 8u * (4 * kMax + 6); }
};

// V+- = X +- Y' of one ab row (double-single, renormalised; this lane holds
// the 8 slots (c = x_l, d = 0..7) of it in Xj and Yj, two columns per f32x2
// instruction), then per sign the row's scale (a power of two above the
// largest of its 64 slots, taken over the 8 lanes x_l) and the S fixed-point
// slices, stored to the row of the stored planes.
//
// The FP32 pipe bounds this (and with it the V+- formation), so the slices are
// cut with four additions each and no renormalisation: adding and subtracting
// 1.5 2^(23 - 8 s) rounds to the multiple of 2^(-8 s) that slice s stores, and
// the remainder is exact.  hi, below 2^8, holds whole multiples of 2^-16 once
// slices 0 and 1 are off, or less of it if it is smaller, so lo joins at slice 2
// exactly to 2^-42 (13 f32x2 instructions per slice before: the formation at
// v = 120 534 -> 418 us).  Five slices end at 2^-33, far above that; of six, which
// end at 2^-41, the last takes the rounding error of that sum along (without it
// slices are off by up to 1.44 x 2^-41, 0.69 rms; with it 0.94 and 0.58).
template <int S>
__device__ __forceinline__ void vpm_store(const float2 *Xj, const float2 *Yj, __nv_bfloat16 *vbase, float *sbase,
                                          int row, int x_l) {
  float2 Vp[8], Vm[8];  // (hi, lo) of columns e, e + 1: hi pair at [e], lo pair at [e + 1]
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    const float2 xh = make_float2(Xj[e].x, Xj[e + 1].x), xl = make_float2(Xj[e].y, Xj[e + 1].y);
    const float2 yh = make_float2(Yj[e].x, Yj[e + 1].x), yl = make_float2(Yj[e].y, Yj[e + 1].y);
    // TwoSum of the high words, then Dekker's Fast2Sum with what is left (where
    // the high words cancel below it, its error is 2^-47 of them, far under the
    // last slice)
    float2 s, t, er;
    two_sum2(xh, yh, s, er);
    t = add2(add2(xl, yl), er);
    Vp[e] = add2(s, t);
    Vp[e + 1] = sub2(t, sub2(Vp[e], s));
    s = sub2(xh, yh);
    const float2 bb = sub2(s, xh);
    er = sub2(sub2(xh, sub2(s, bb)), add2(yh, bb));
    t = add2(sub2(xl, yl), er);
    Vm[e] = add2(s, t);
    Vm[e + 1] = sub2(t, sub2(Vm[e], s));
  }
#pragma unroll
  for (int sg = 0; sg < 2; ++sg) {
    const float2 *V = sg ? Vm : Vp;
    float m = 0.f;
#pragma unroll
    for (int e = 0; e < 8; e += 2) m = fmaxf(m, fmaxf(fabsf(V[e].x), fabsf(V[e].y)));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 4));
    // rows below 2^-119 (far under any integral of interest) count as zero,
    // which keeps both powers of two normal floats
    float inv = 0.f, scale = 0.f;
    const int E = exp_above(m);
    if (m > 0.f && E >= -118) {
      inv = pow2f(8 - E);
      scale = pow2f(E - 8);
    }
    uint4 out[S];
    const float2 inv2 = make_float2(inv, inv);
#pragma unroll
    for (int e2 = 0; e2 < 4; ++e2) {
      float2 r = mul2(V[2 * e2], inv2);
      const float2 lo = mul2(V[2 * e2 + 1], inv2);
      float2 er = make_float2(0.f, 0.f);  // of r + lo (r is zero or a multiple of more than lo)
#pragma unroll
      for (int s = 0; s < S; ++s) {
        if (s == 5) r = add2(r, er);
        const float mg = 12582912.0f * pow2f(-8 * s);
        const float2 magic = make_float2(mg, mg);
        const float2 x = sub2(add2(s == 2 ? add2(r, lo) : r, magic), magic);
        r = sub2(r, x);
        if (s == 2) fast_two_sum2(r, lo, r, er);
        const __nv_bfloat162 b2 = __floats2bfloat162_rn(x.x, x.y);
        (&out[s].x)[e2] = *reinterpret_cast<const uint32_t *>(&b2);
      }
    }
#pragma unroll
    for (int s = 0; s < S; ++s)
      __stcs(reinterpret_cast<uint4 *>(vbase + (size_t)(sg * S + s) * (128 * SLOTS) + row * SLOTS + x_l * CB),
             out[s]);
    if (x_l == 0) sbase[sg * 128 + row] = scale;
  }
}

// The slice products of one K-step (two K16) into the four order blocks of a
// TMEM half: for slice pa <= 3 of A the slices q <= 3 - pa of B sit back to
// back, so one MMA of N = 64 (4 - pa) puts order pa + q into block pa + q; the
// products of order >= 4 go into block 3 one by one.  first: the window's first
// K-step.  (Descriptor low words are address / 16 with a fixed bit; shared
// addresses stay below 2^18, so the constant offsets never carry into it.)
template <int S>
__device__ __forceinline__ void mma_window(uint32_t dT, uint32_t a_smem, uint32_t b_smem, bool first) {
  const uint64_t hi = (uint64_t)desc_hi(512, kSwizzle64) << 32;
  const uint32_t a = (a_smem >> 4) | (1u << 16), b = (b_smem >> 4) | (1u << 16);
#pragma unroll
  for (int kk = 0; kk < KSTEP / 16; ++kk)
#pragma unroll
    for (int pa = 0; pa < S; ++pa) {
      const uint64_t ad = hi | (a + pa * (A_TILE >> 4) + kk * 2);
      if (pa <= 3)
        mma_bf16_warp(dT + 64u * pa, ad, hi | (b + kk * 2), idesc_bf16(128, 64 * (4 - pa)),
                      kk == 0 && pa == 0 && first ? 0u : 1u);
#pragma unroll
      for (int q = (pa <= 4 ? 4 - pa : 0); q <= S - 1 - pa; ++q)
        mma_bf16_warp(dT + 192u, ad, hi | (b + q * (B_TILE >> 4) + kk * 2), idesc_bf16(128, 64), 1u);
    }
}

// ============================================================================ pass 1
// GEMM1 of every (tile, block pair) in exact windows, V+- = X +- Y', fixed-point
// slices of V+- to the workspace.  Work units walk range-major (unit u: range
// u / tiles of tile u % tiles) so the resident CTAs share B panels in L2.
template <int S, bool kBatch>
__global__ void __launch_bounds__(kThreads, 1) oz_vstore_kernel(const __grid_constant__ OzLaunch Lp) {
  using C = Cfg1<S>;
  static_assert(C::kStages >= 3 && 8 * (2 * C::kStages + Bars::kCount) + 8 <= 256, "ring");
  static_assert(S >= 4 && S <= 6, "slices");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
  uint8_t *smem = smem_raw + pad;
  const uint32_t ring = raw + pad;
  Bars bars{ring + C::kRing, C::kStages};
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + C::kRing + 8 * (2 * C::kStages + Bars::kCount));
  int *abort_flag = reinterpret_cast<int *>(tmem_holder + 1);
  const int warp = (int)uniform(threadIdx.x / 32), lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(bars.full(s), 1);
      mbar_init(bars.empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bars.cfull(b), 1);
      mbar_init(bars.cfree(b), kEpi);
    }
    mbar_init(bars.done(), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_holder), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  dep_sync();
  const uint32_t tmem = *tmem_holder;
  const Watchdog wd{Lp.status, abort_flag, Lp.timeout_ns};

  if (warp == 0) {
    // ================================================================ TMA producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0, armed = 0, armed_par = 0;
      bool ok = true;
      for (int u = blockIdx.x; ok && u < Lp.nitems; u += gridDim.x) {
        int local;
        const OzArgs &A = oz_args<kBatch>(Lp, u, local);
        const Item I = decode(A, vstore_slot(A, local), 1);
        const int nwin = (A.nks + kOzKc - 1) / kOzKc;
        tma_prefetch_desc(&A.tmA);
        tma_prefetch_desc(&A.tmB);
        for (int p = I.p0; ok && p < I.p1; ++p) {
          int k, l;
          pair_of(p, k, l);
          const int ntile = (k == l) ? 1 : 2;
          for (int w = 0; ok && w < nwin; ++w)
            for (int tt = 0; ok && tt < ntile; ++tt)
              for (int ks = w * kOzKc; ok && ks < min(A.nks, (w + 1) * kOzKc); ++ks) {
                if (!(ok = mbar_wait(bars.empty(stage), phase ^ 1u, wd, kSiteTmaEmpty))) break;
                const uint32_t dst = ring + (uint32_t)stage * C::kStage;
                mbar_arrive_expect_tx(bars.full(stage), C::kStage);
                armed |= 1u << stage;
                armed_par = (armed_par & ~(1u << stage)) | (phase << stage);
                // X: rows (a, c in block k) x (b, d in block l); Y: the blocks swapped
                const int ca = (tt == 0 ? k : l) * CB, cb = (tt == 0 ? l : k) * CB;
                tma_load_4d(dst, &A.tmA, bars.full(stage), ks * KSTEP, ca, I.A0, 0);
                tma_load_4d(dst + S * A_TILE, &A.tmB, bars.full(stage), ks * KSTEP, cb, I.B0, 0);
                if (++stage == C::kStages) {
                  stage = 0;
                  phase ^= 1u;
                }
              }
        }
      }
      if (!ok) {
        DrainWatch dw(Lp.status, Lp.timeout_ns);
        for (int s = 0; s < C::kStages; ++s)
          if (armed & (1u << s)) mbar_wait(bars.full(s), (armed_par >> s) & 1u, dw.wd, kSiteTmaFull);
      }
    }
  } else if (warp == 1) {
    // ================================================================ MMA issuer
    // the whole warp runs in step (see mma_bf16_warp)
    const uint32_t utm = uniform(tmem), uring = uniform(ring);
    const Bars ub{uring + C::kRing, C::kStages};
    int stage = 0;
    uint32_t phase = 0, use = 3u, acc = 0;  // windows take the accumulators in turn; use: the parity that each is free at
    bool ok = true;
    for (int u = blockIdx.x; ok && u < Lp.nitems; u += gridDim.x) {
      int local;
      const OzArgs &A = oz_args<kBatch>(Lp, u, local);
      const Item I = decode(A, vstore_slot(A, local), 1);
      const int nks = (int)uniform(A.nks), nwin = (nks + kOzKc - 1) / kOzKc;
      const int p0 = (int)uniform(I.p0), p1 = (int)uniform(I.p1);
      for (int p = p0; ok && p < p1; ++p) {
        int k, l;
        pair_of(p, k, l);
        const int ntile = (int)uniform(k == l ? 1 : 2);
        for (int w = 0; ok && w < nwin; ++w)
          for (int tt = 0; ok && tt < ntile; ++tt) {
              if (!(ok = mbar_wait_warp(ub.cfree(acc), (use >> acc) & 1u, wd, kSiteXYFree))) break;
              tc_fence_after();
              const uint32_t dT = utm + 256u * acc;
              const int ks0 = w * kOzKc;
              for (int ks = ks0; ok && ks < min(nks, ks0 + kOzKc); ++ks) {
                if (!(ok = mbar_wait_warp(ub.full(stage), phase, wd, kSiteTmaFull))) break;
                const uint32_t st = uring + (uint32_t)stage * C::kStage;
                mma_window<S>(dT, st, st + S * A_TILE, ks == ks0);
                mma_commit_warp(ub.empty(stage));
                if (++stage == C::kStages) {
                  stage = 0;
                  phase ^= 1u;
                }
              }
              if (!ok) break;
              mma_commit_warp(ub.cfull(acc));
              use ^= 1u << acc;
              acc ^= 1u;
          }
      }
    }
    mma_commit_warp(ub.done());
    DrainWatch dw(Lp.status, Lp.timeout_ns);
    mbar_wait(ub.done(), 0, dw.wd, kSiteRFull);
  } else {
    // ================================================================ conversion warps
    const int quad = warp & 3;
    const int qw = (warp - 2) >> 2;      // columns 16 qw .. 16 qw + 15 of each block: b = 2 qw + j
    const int L = quad * 32 + lane;      // TMEM lane = A row (a, c): a = A0 + L / 8, c = 8 k + L % 8
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + 16u * qw;
    const int a_l = L >> 3, x_l = L & 7;
    uint32_t use = 0, acc = 0;  // as the issuer's
    bool ok = true;
    for (int u = blockIdx.x; ok && u < Lp.nitems; u += gridDim.x) {
      int local;
      const OzArgs &A = oz_args<kBatch>(Lp, u, local);
      const Item I = decode(A, vstore_slot(A, local), 1);
      const int nwin = (A.nks + kOzKc - 1) / kOzKc;
      const int a = I.A0 + a_l;
      for (int p = I.p0; ok && p < I.p1; ++p) {
        int k, l;
        pair_of(p, k, l);
        const bool diag = (k == l);
        float2 X[16], Y[16];  // (hi, lo) sums of columns (b = 2 qw + j, d = 0..7), j = e / 8
#pragma unroll
        for (int e = 0; e < 16; ++e) X[e] = Y[e] = make_float2(0.f, 0.f);
        for (int w = 0; ok && w < nwin; ++w)
          for (int tt = 0; tt < (diag ? 1 : 2); ++tt) {
            if (!(ok = mbar_wait(bars.cfull(acc), (use >> acc) & 1u, wd, kSiteXYFull))) break;
            use ^= 1u << acc;
            tc_fence_after();
            if (tt == 0)
              drain_window(tl + 256u * acc, X);
            else
              drain_window(tl + 256u * acc, Y);
            tc_fence_before();
            mbar_arrive(bars.cfree(acc));
            acc ^= 1u;
          }
        if (!ok) break;
        // scale to B units: X[(a, c), (b, d)] by scale(a, c) scale(b, d), c = 8k + x_l, d = 8l + e;
        // Y[(a, d'), (b, c')] with d' = 8l + x_l, c' = 8k + e
        const float rX = A.rsB[(size_t)a * A.vp + k * CB + x_l];
        const float rY = A.rsB[(size_t)a * A.vp + l * CB + x_l];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int b = I.B0 + 2 * qw + j;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float sx = rX * A.rsB[(size_t)b * A.vp + l * CB + e];
            X[8 * j + e].x *= sx;
            X[8 * j + e].y *= sx;
            if (!diag) {
              const float sy = rY * A.rsB[(size_t)b * A.vp + k * CB + e];
              Y[8 * j + e].x *= sy;
              Y[8 * j + e].y *= sy;
            }
          }
        }
        // Y' : lane (a, c = 8k + x_l) gets (ad|bc) for d = 8l + e (transpose across the 8 lanes)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          float rh[8], rl[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            rh[e] = diag ? X[8 * j + e].x : Y[8 * j + e].x;
            rl[e] = diag ? X[8 * j + e].y : Y[8 * j + e].y;
          }
          transpose8(rh, x_l);
          transpose8(rl, x_l);
#pragma unroll
          for (int e = 0; e < 8; ++e) Y[8 * j + e] = make_float2(rh[e], rl[e]);
        }
        __nv_bfloat16 *vbase = A.Vst + (size_t)(I.tile * A.nbp + p) * 2 * S * (128 * SLOTS);
        float *sbase = A.sV + (size_t)(I.tile * A.nbp + p) * 2 * 128;
#pragma unroll
        for (int j = 0; j < 2; ++j) vpm_store<S>(X + 8 * j, Y + 8 * j, vbase, sbase, a_l * 8 + 2 * qw + j, x_l);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ============================================================================ symmetric B
// With B^P_ac = B^P_ca for every P (the RI factors of real orbitals) the
// integral (ac|bd) = sum_P B^P_ac B^P_bd depends only on the unordered pairs
// {a, c} and {b, d}, and on them in either order.  Rows (a, c) of B with a in
// virtual block alpha and c in block gamma, alpha <= gamma, form the row block
// pair r = (alpha, gamma) (numbered as the block pairs of the slot scheme);
// the distinct integrals are the 64 x 64 tiles
//   X'(r, q)[(i' % 8) * 8 + j' % 8][(i % 8) * 8 + j % 8] = sum_P B^P_ij B^P_i'j',
// i in alpha, j in gamma, i' in beta, j' in lambda, q = (beta, lambda), r <= q,
// both orders of a diagonal block pair present.  They are computed once each
// (about a quarter of the general pass 1's GEMM1) in the same exact windows
// and kept as double-single sums in B units; the formation kernel then builds
// V+- of every (ab tile, block pair) from them and slices it as pass 1 does.

// Tile (r, q), r <= q, of the distinct integrals in row-major triangular order.
__device__ __forceinline__ size_t xtri(int r, int q, int nbp) {
  return (size_t)r * nbp - (size_t)r * (r - 1) / 2 + (size_t)(q - r);
}

// Pass 1 of the symmetric form.  Row tile m of 128 rows (a in the 16-block iA, c
// in block kk >= 2 iA) holds the row block pairs (2 iA, kk) and (2 iA + 1, kk); in
// the order of xtile the pairs' numbers rise with m, so the 128 x 128 tiles (m,
// n) with m <= n cover the distinct integrals.  A work unit (xunits[u] = (iA, kk,
// n0, n1)) is one row tile against the column tiles n0 .. n1 - 1.  Block pairs r
// > q within a tile are computed but not stored, and nor is the half (2 iA + 1,
// 2 iA) of the tile kk = 2 iA (the tile kk = 2 iA + 1 holds it).
//
// Bound by shared memory, which gives 128 bytes a clock: per K16 the MMAs read
// 112 KB and 40 KB come in, 1,216 clocks for 960 of MMAs.  (128 x 64 tiles, X's
// and Y's halves of TMEM in turn as in the general pass 1, take 768 for half the
// tile, and their MMAs of 64 columns run at two thirds of the rate: 419 us at v =
// 120, N = 480, 24.3 ms at v = 300, N = 1200, against 366 us and 20.8 ms.)  The four
// order accumulators of 128 columns fill TMEM, so a window's drain overlaps the
// next window's products of orders >= 3, 9 of 15, which run ahead on the first
// K32 steps; their own short drain overlaps the window's last head products.
__host__ __device__ inline void xtile(int n, int &iA, int &kk) {  // n = (kk + 1)^2 / 4 + iA, iA <= kk / 2
  int k = (int)(2.0f * sqrtf((float)n)) - 1;
  if (k < 0) k = 0;
  while ((k + 2) * (k + 2) / 4 <= n) ++k;
  while ((k + 1) * (k + 1) / 4 > n) --k;
  kk = k;
  iA = n - (k + 1) * (k + 1) / 4;
}
// Ring stages are the 128 rows of both operands of a K32 step, in two rings: L
// slices 0..2, H slices 3.. .  H goes back as soon as the tail products (orders
// >= 3) of a step are issued, L is held for the others, so that the steps after
// the ones that ran ahead are there in time (one ring of all slices: 1,000
// clocks a window lost; 400 us against 366 at v = 120, N = 480).  Rows of 64
// bytes: TMA takes about a row a clock, and rows of 32 bytes bounded the pass.
template <int S>
struct CfgX {
  static constexpr int kLow = 3, kHigh = S - kLow;
  static constexpr uint32_t kStageL = 2u * kLow * A_TILE, kStageH = 2u * kHigh * A_TILE;
  static constexpr int kH = 2, kL = (int)((kSmemBudget - kH * kStageH) / kStageL);
  static constexpr uint32_t kBaseH = kL * kStageL, kRing = kBaseH + kH * kStageH;
  static constexpr uint32_t kSmem = kRing + 256 + 1024;
  static constexpr int kAhead = kL - 1;  // K32 steps whose tail products run ahead
};
struct BarsX {
  uint32_t base;
  int nl, nh;
  __device__ uint32_t fullL(int s) const { return base + 8u * s; }
  __device__ uint32_t emptyL(int s) const { return base + 8u * (nl + s); }
  __device__ uint32_t fullH(int s) const { return base + 8u * (2 * nl + s); }
  __device__ uint32_t emptyH(int s) const { return base + 8u * (2 * nl + nh + s); }
  __device__ uint32_t cfull(int b) const { return base + 8u * (2 * (nl + nh) + b); }
  __device__ uint32_t cfree(int b) const { return base + 8u * (2 * (nl + nh) + 2 + b); }
  __device__ uint32_t done() const { return base + 8u * (2 * (nl + nh) + 4); }
  static constexpr int kCount = 5;  // + 2 (nl + nh)
};
// A step's slices in shared memory (in units of 16 bytes, as descriptors): slice
// s of either operand at l or h.
template <int S>
struct XStep {
  uint64_t l, h;
  __device__ __forceinline__ uint64_t a(int s) const { return s < 3 ? l + s * (A_TILE >> 4) : h + (s - 3) * (A_TILE >> 4); }
  __device__ __forceinline__ uint64_t b(int s) const {
    return s < 3 ? l + (3 + s) * (A_TILE >> 4) : h + (S - 3 + s - 3) * (A_TILE >> 4);
  }
};
// The products of orders >= 3 and of orders 0 to 2 of one K32 step into the order
// blocks of 128 columns at d.
template <int S>
__device__ __forceinline__ void xsym_tail(uint32_t d, const XStep<S> &x, bool first) {
#pragma unroll
  for (int kk = 0; kk < 2; ++kk)
#pragma unroll
    for (int pa = 0; pa < S; ++pa)
#pragma unroll
      for (int q = (pa < 3 ? 3 - pa : 0); q < S - pa; ++q)
        mma_bf16_warp(d + 384u, x.a(pa) + 2 * kk, x.b(q) + 2 * kk, idesc_bf16(128, 128),
                      first && kk == 0 && pa == 0 && q == 3 ? 0u : 1u);
}
template <int S>
__device__ __forceinline__ void xsym_head(uint32_t d, const XStep<S> &x, bool first) {
  constexpr uint32_t id = idesc_bf16(128, 128), id2 = idesc_bf16(128, 256);
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    const uint32_t acc = first && kk == 0 ? 0u : 1u;
    mma_bf16_warp(d, x.a(0) + 2 * kk, x.b(0) + 2 * kk, id2, acc);
    mma_bf16_warp(d + 256u, x.a(0) + 2 * kk, x.b(2) + 2 * kk, id, acc);
    mma_bf16_warp(d + 128u, x.a(1) + 2 * kk, x.b(0) + 2 * kk, id2, 1u);
    mma_bf16_warp(d + 256u, x.a(2) + 2 * kk, x.b(0) + 2 * kk, id, 1u);
  }
}

template <int S, bool kBatch>
__global__ void __launch_bounds__(kThreads, 1) oz_xsym_kernel(const __grid_constant__ OzLaunch Lp) {
  using C = CfgX<S>;
  constexpr int kBars = 2 * (C::kL + C::kH) + BarsX::kCount;
  static_assert(C::kAhead >= 1 && 8 * kBars + 8 <= 256, "ring");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
  uint8_t *smem = smem_raw + pad;
  const uint32_t ring = raw + pad;
  BarsX bars{ring + C::kRing, C::kL, C::kH};
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + C::kRing + 8 * kBars);
  int *abort_flag = reinterpret_cast<int *>(tmem_holder + 1);
  const int warp = (int)uniform(threadIdx.x / 32), lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kL; ++s) {
      mbar_init(bars.fullL(s), 1);
      mbar_init(bars.emptyL(s), 1);
    }
    for (int s = 0; s < C::kH; ++s) {
      mbar_init(bars.fullH(s), 1);
      mbar_init(bars.emptyH(s), 1);
    }
    for (int b = 0; b < 2; ++b) {  // 0: orders 0 to 2, 1: orders >= 3
      mbar_init(bars.cfull(b), 1);
      mbar_init(bars.cfree(b), kEpi);
    }
    mbar_init(bars.done(), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_holder), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  dep_sync();
  const uint32_t tmem = *tmem_holder;
  const Watchdog wd{Lp.status, abort_flag, Lp.timeout_ns};

  if (warp == 0) {
    // ================================================================ TMA producer
    if (lane == 0) {
      uint32_t nl = 0, nh = 0;  // stages filled so far
      bool ok = true;
      for (int u = blockIdx.x; ok && u < Lp.nitems; u += gridDim.x) {
        int local;
        const OzArgs &A = oz_args<kBatch>(Lp, u, local);
        const int4 U = A.xunits[local];
        tma_prefetch_desc(&A.tmXl);
        tma_prefetch_desc(&A.tmXh);
        for (int t = U.z; ok && t < U.w; ++t) {
          int jB, ll;
          xtile(t, jB, ll);
          for (int k = 0; k < A.nks; ++k) {
            // rows (a in 16-block iA, c in block kk), then rows (b in 16-block jB, d in block ll)
            uint32_t st = nl % C::kL, dst = ring + st * C::kStageL;
            if (!(ok = mbar_wait(bars.emptyL(st), (nl / C::kL + 1) & 1u, wd, kSiteTmaEmpty))) break;
            mbar_arrive_expect_tx(bars.fullL(st), C::kStageL);
            tma_load_4d(dst, &A.tmXl, bars.fullL(st), k * KSTEP, U.y * CB, U.x * 16, 0);
            tma_load_4d(dst + C::kStageL / 2, &A.tmXl, bars.fullL(st), k * KSTEP, ll * CB, jB * 16, 0);
            ++nl;
            st = nh % C::kH, dst = ring + C::kBaseH + st * C::kStageH;
            if (!(ok = mbar_wait(bars.emptyH(st), (nh / C::kH + 1) & 1u, wd, kSiteTmaEmpty))) break;
            mbar_arrive_expect_tx(bars.fullH(st), C::kStageH);
            tma_load_4d(dst, &A.tmXh, bars.fullH(st), k * KSTEP, U.y * CB, U.x * 16, C::kLow);
            tma_load_4d(dst + C::kStageH / 2, &A.tmXh, bars.fullH(st), k * KSTEP, ll * CB, jB * 16, C::kLow);
            ++nh;
          }
        }
      }
      if (!ok) {  // the copies in flight land before the CTA leaves: the last fill of every stage
        DrainWatch dw(Lp.status, Lp.timeout_ns);
        for (uint32_t q = nl > C::kL ? nl - C::kL : 0; q < nl; ++q)
          mbar_wait(bars.fullL(q % C::kL), (q / C::kL) & 1u, dw.wd, kSiteTmaFull);
        for (uint32_t q = nh > C::kH ? nh - C::kH : 0; q < nh; ++q)
          mbar_wait(bars.fullH(q % C::kH), (q / C::kH) & 1u, dw.wd, kSiteTmaFull);
      }
    }
  } else if (warp == 1) {
    // ================================================================ MMA issuer
    // the whole warp runs in step (see mma_bf16_warp)
    const uint32_t utm = uniform(tmem), uring = uniform(ring);
    const BarsX ub{uring + C::kRing, C::kL, C::kH};
    const uint64_t hi = (uint64_t)desc_hi(512, kSwizzle64) << 32;
    uint32_t n = 0, g = 0;  // steps used (both rings), windows begun
    bool ok = true;
    auto at = [&](uint32_t q) {
      XStep<S> x;
      x.l = hi | (((uring + q % C::kL * C::kStageL) >> 4) | (1u << 16));
      x.h = hi | (((uring + C::kBaseH + q % C::kH * C::kStageH) >> 4) | (1u << 16));
      return x;
    };
    // tail products of step q, then its slices 3.. go back
    auto tail = [&](uint32_t q, bool first) {
      if (!mbar_wait_warp(ub.fullL(q % C::kL), (q / C::kL) & 1u, wd, kSiteTmaFull) ||
          !mbar_wait_warp(ub.fullH(q % C::kH), (q / C::kH) & 1u, wd, kSiteTmaFull))
        return false;
      xsym_tail<S>(utm, at(q), first);
      mma_commit_warp(ub.emptyH(q % C::kH));
      return true;
    };
    auto head = [&](uint32_t q, bool first) {
      xsym_head<S>(utm, at(q), first);
      mma_commit_warp(ub.emptyL(q % C::kL));
    };
    for (int u = blockIdx.x; ok && u < Lp.nitems; u += gridDim.x) {
      int local;
      const OzArgs &A = oz_args<kBatch>(Lp, u, local);
      const int4 U = A.xunits[local];
      const int nk = (int)uniform(A.nks), t0 = (int)uniform(U.z), t1 = (int)uniform(U.w);
      for (int t = t0; ok && t < t1; ++t)
        for (int k0 = 0; ok && k0 < nk; k0 += kOzKc, ++g) {
          const int nw = min(kOzKc, nk - k0), ahead = min(C::kAhead, nw);
          if (!(ok = mbar_wait_warp(ub.cfree(1), (g & 1u) ^ 1u, wd, kSiteXYFree))) break;
          tc_fence_after();
          for (int i = 0; ok && i < ahead; ++i) ok = tail(n + i, i == 0);
          if (ok && ahead == nw) mma_commit_warp(ub.cfull(1));
          if (!ok || !(ok = mbar_wait_warp(ub.cfree(0), (g & 1u) ^ 1u, wd, kSiteXYFree))) break;
          tc_fence_after();
          for (int i = 0; i < ahead; ++i) head(n + i, i == 0);
          // a step's tail products first, so that their last drain overlaps the last head products
          for (int i = ahead; ok && i < nw; ++i) {
            if (!(ok = tail(n + i, false))) break;
            if (i == nw - 1) mma_commit_warp(ub.cfull(1));
            head(n + i, false);
          }
          if (!ok) break;
          n += nw;
          mma_commit_warp(ub.cfull(0));
        }
    }
    mma_commit_warp(ub.done());
    DrainWatch dw(Lp.status, Lp.timeout_ns);
    mbar_wait(ub.done(), 0, dw.wd, kSiteRFull);
  } else {
    // ================================================================ conversion warps
    const int quad = warp & 3;
    const int qw = (warp - 2) >> 2;  // columns 32 qw .. 32 qw + 31: b = 16 jB + 4 qw + j, d % 8 = e
    const int L = quad * 32 + lane;  // TMEM lane = row (a, c): a = 16 iA + L / 8, c = 8 kk + L % 8
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + 32u * qw;
    uint32_t g = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < Lp.nitems; u += gridDim.x) {
      int local;
      const OzArgs &A = oz_args<kBatch>(Lp, u, local);
      const int4 U = A.xunits[local];
      const int nwin = (A.nks + kOzKc - 1) / kOzKc, h = L >> 6;
      const int r = ppos(U.y) + 2 * U.x + h;  // row block pair (2 iA + h, kk)
      const bool dup = h == 1 && U.y == 2 * U.x;
      const float ra = A.rsB[(size_t)(U.x * 16 + (L >> 3)) * A.vp + U.y * CB + (L & 7)];
      for (int t = U.z; ok && t < U.w; ++t) {
        float2 H[16], Lo[16];  // (hi, lo) sums of columns 2 k and 2 k + 1 (as .x and .y)
#pragma unroll
        for (int e = 0; e < 16; ++e) H[e] = Lo[e] = make_float2(0.f, 0.f);
        for (int w = 0; w < nwin; ++w, ++g) {
          if (!(ok = mbar_wait(bars.cfull(1), g & 1u, wd, kSiteXYFull))) break;
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float g3[8];
            tmem_ld4(tl + 384u + 8u * c, *reinterpret_cast<float(*)[4]>(g3));
            tmem_ld4(tl + 388u + 8u * c, *reinterpret_cast<float(*)[4]>(g3 + 4));
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 4; ++e) Lo[4 * c + e] = add2(Lo[4 * c + e], make_float2(g3[2 * e], g3[2 * e + 1]));
          }
          tc_fence_before();
          mbar_arrive(bars.cfree(1));
          if (!(ok = mbar_wait(bars.cfull(0), g & 1u, wd, kSiteXYFull))) break;
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < 8; ++c) {  // as drain_window
            float g0[4], g1[4], g2[4];
            tmem_ld4(tl + 4u * c, g0);
            tmem_ld4(tl + 128u + 4u * c, g1);
            tmem_ld4(tl + 256u + 4u * c, g2);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              float2 h0, er, hh, lo;
              fast_two_sum2(make_float2(g0[2 * e], g0[2 * e + 1]), make_float2(g1[2 * e], g1[2 * e + 1]), h0, er);
              fast_two_sum2(h0, add2(er, make_float2(g2[2 * e], g2[2 * e + 1])), hh, lo);
              ds_acc2(H[2 * c + e], Lo[2 * c + e], hh, lo);
            }
          }
          tc_fence_before();
          mbar_arrive(bars.cfree(0));
        }
        if (!ok) break;
        int jB, ll;
        xtile(t, jB, ll);
        const int g8 = qw >> 1, q = ppos(ll) + 2 * jB + g8;  // column block pair (2 jB + g8, ll)
        if (dup || r > q || (g8 == 1 && ll == 2 * jB)) continue;
        // column-major, so that a warp's 32 rows are 256 bytes of every store: 16 bytes per row
        // of a row-major tile took 20,000 clocks for 128 columns, during which the tensor cores
        // ran dry (492 -> 430 us in all at v = 120, N = 480)
        float2 *dst = A.Xs + xtri(r, q, A.nbp) * 4096 + (size_t)((qw & 1) * 32 * 64 + (L & 63));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float *rb = A.rsB + (size_t)(jB * 16 + 4 * qw + j) * A.vp + ll * CB;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float sc = ra * rb[e];
            const float2 x = H[4 * j + e / 2], y = Lo[4 * j + e / 2];
            dst[(8 * j + e) * 64] = e & 1 ? make_float2(x.y * sc, y.y * sc) : make_float2(x.x * sc, y.x * sc);
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// V+- of every (ab tile, block pair) of the plan's tile range from the
// distinct integral tiles: X[(a, c), (b, d)] = (ac|bd) and Y'[(a, c), (b, d)]
// = (ad|bc) read straight from them, then vpm_store as in pass 1.  Local work
// unit (of a molecule of a batch, or of `one`) = (local tile / nbp, block
// pair % nbp); 512 threads, each the ab rows
// (a = A0 + L / 8, b = B0 + 2 qw + j) and the slot row c = 8 k + L % 8, as
// pass 1's conversion warps.
// Where the integrals (p q | r s) of four 8-blocks lie in the distinct tiles:
// place = base + p' sp + q' sq + r' sr + s' ss with the indices inside their
// blocks, since which tile holds them and in which orientation depends on the
// blocks alone.
struct VfMap {
  const float2 *base;
  int sp, sq, sr, ss;
};
__device__ __forceinline__ VfMap vf_map(const float2 *Xs, int nbp, int bp, int bq, int br, int bs) {
  VfMap m;
  int r, q;
  if (bp <= bq) {
    r = ppos(bq) + bp;
    m.sp = 8, m.sq = 1;
  } else {
    r = ppos(bp) + bq;
    m.sp = 1, m.sq = 8;
  }
  if (br <= bs) {
    q = ppos(bs) + br;
    m.sr = 8, m.ss = 1;
  } else {
    q = ppos(br) + bs;
    m.sr = 1, m.ss = 8;
  }
  if (r <= q) {
    m.base = Xs + xtri(r, q, nbp) * 4096;
    m.sr *= 64, m.ss *= 64;
  } else {
    m.base = Xs + xtri(q, r, nbp) * 4096;
    m.sp *= 64, m.sq *= 64;
  }
  return m;
}
// X = (a c | b d) and Y = (a d | b c) at b, b + 1 for the eight d of a block:
// p points at (b, d = 0), sb and sd are the distances in b and d.  16-byte
// loads where d or b runs contiguously, else 8-byte ones.
__device__ __forceinline__ void vf_gather(const float2 *__restrict__ p, int sb, int sd, float2 (&v)[2][8]) {
  if (sd == 1) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 t = __ldg(reinterpret_cast<const float4 *>(p + j * sb) + i);
        v[j][2 * i] = make_float2(t.x, t.y);
        v[j][2 * i + 1] = make_float2(t.z, t.w);
      }
  } else if (sb == 1) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float4 t = __ldg(reinterpret_cast<const float4 *>(p + e * sd));
      v[0][e] = make_float2(t.x, t.y);
      v[1][e] = make_float2(t.z, t.w);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 8; ++e) v[j][e] = __ldg(p + j * sb + e * sd);
  }
}

template <int S, bool kBatch>
__global__ void __launch_bounds__(512) oz_vform_kernel(const __grid_constant__ OzLaunch Lp) {
  dep_sync();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int L = (warp & 3) * 32 + lane, qw = warp >> 2;
  const int a_l = L >> 3, x_l = L & 7;
  for (int u = blockIdx.x; u < Lp.nitems; u += gridDim.x) {
    int local;
    const OzArgs &A = oz_args<kBatch>(Lp, u, local);
    if (A.forder) local = A.forder[local];
    const int t = local / A.nbp, p = local - t * A.nbp;
    int iA = 0, tr = t + A.tile0;
    while (tr >= A.nB8 - 2 * iA) {
      tr -= A.nB8 - 2 * iA;
      ++iA;
    }
    const int ba = 2 * iA + ((warp & 3) >> 1), bb = 2 * iA + tr;  // this warp's a block, the b block
    int k, l;
    pair_of(p, k, l);
    float2 X[2][8], Y[2][8];
    const VfMap mx = vf_map(A.Xs, A.nbp, ba, k, bb, l);  // (a c | b d)
    const VfMap my = vf_map(A.Xs, A.nbp, ba, l, bb, k);  // (a d | b c)
    vf_gather(mx.base + (a_l & 7) * mx.sp + x_l * mx.sq + 2 * qw * mx.sr, mx.sr, mx.ss, X);
    vf_gather(my.base + (a_l & 7) * my.sp + x_l * my.ss + 2 * qw * my.sr, my.sr, my.sq, Y);
    __nv_bfloat16 *vbase = A.Vst + (size_t)(t * A.nbp + p) * 2 * S * (128 * SLOTS);
    float *sbase = A.sV + (size_t)(t * A.nbp + p) * 2 * 128;
#pragma unroll
    for (int j = 0; j < 2; ++j) vpm_store<S>(X[j], Y[j], vbase, sbase, a_l * 8 + 2 * qw + j, x_l);
  }
}

// ============================================================================ pass 2
// GEMM2 of one (tile, chunk of <= 128 occupied pairs of one sign, block-pair
// range), one CTA per work unit: per block pair the slice products V_p T_q^T
// (p + q < S) of its four 16-slot pieces into the four order accumulators
// (columns 0, sc, 2 sc and 3 sc), issued and drained in two groups with the
// pair's row scales into double-single sums in registers.  Work units walk
// range-major (unit u: range u / (tiles * chunks)).
//
// Issue.  A pair takes 56 MMAs (S = 5), and issuing them was what bounded the
// pass: 5,500 of 6,860 clocks a pair at o = 10, v = 120 (chunks of 64 and 48
// columns) went into the issuing thread.  The MMA warp now runs in step with
// all its operands in uniform registers.
//
// Order of the groups.  Shared memory holds little more than one pair's
// operands (160 of 224 KB at 128 columns), so a stage should be refilled long
// before it is needed again.  Orders >= 3, which read all slices and take 9 of
// the 15 products, go first: they need a piece only every ninth MMA, and give
// slices 3.. back at once; orders 0 to 2 then run on slices 0..2 alone, which go
// back one piece after the other well before the next pair's second piece.
// Their drain, the heavy one, overlaps the next pair's longer group.  The FP32
// pipe bounds it, so the three orders are drained together (17 operations for
// two columns; order 2 in a group of its own took 25 in all): 38.8 -> 35.4 ms at
// o = 28, v = 300, N = 1200, 312 -> 303 us at o = 10, v = 120.  The latter reads
// V+- at 5.4 TB/s.
template <int S, bool kBatch>
__global__ void __launch_bounds__(kThreads, 1) oz_gemm2_kernel(const __grid_constant__ OzLaunch Lp) {
  using C = Cfg2<S>;
  static_assert(C::kMaxL == Bars2::kMax && C::kBars + 8 <= 512, "barriers");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
  uint8_t *smem = smem_raw + pad;
  const uint32_t ring = raw + pad;
  const Bars2 bars{ring + C::kRing};
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + C::kRing + C::kBars);
  int *abort_flag = reinterpret_cast<int *>(tmem_holder + 1);
  const int warp = (int)uniform(threadIdx.x / 32), lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kMaxL; ++s) {
      mbar_init(bars.fullL(s), 1);
      mbar_init(bars.emptyL(s), 1);
      mbar_init(bars.fullH(s), 1);
      mbar_init(bars.emptyH(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bars.cfull(b), 1);
      mbar_init(bars.cfree(b), kEpi);
    }
    mbar_init(bars.done(), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_holder), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  dep_sync();
  const uint32_t tmem = *tmem_holder;
  const Watchdog wd{Lp.status, abort_flag, Lp.timeout_ns};
  constexpr int kPieces = SLOTS / TPIECE;
  int local;
  const OzArgs &A = oz_args<kBatch>(Lp, (int)blockIdx.x, local);
  const Item I = decode(A, gemm2_slot(A, local), A.nchunks);
  const uint32_t sc = (uint32_t)(I.CH.nps + I.CH.nms);
  const int sg = I.CH.nps > 0 ? 0 : 1;
  const Ring2 R = Ring2::of<S>(sc);

  if (warp == 0) {
    // ================================================================ TMA producer
    if (lane == 0) {
      int sl = 0, sh = 0;
      uint32_t pl = 0, ph = 0, armedL = 0, parL = 0, armedH = 0, parH = 0;
      bool ok = true;
      tma_prefetch_desc(&A.tmVl);
      tma_prefetch_desc(&A.tmVh);
      const uint32_t tlow = C::kLow * sc * 32u, thigh = C::kHigh * sc * 32u;
      const uint8_t *t2 = A.T2 + I.CH.t2off + (size_t)I.p0 * kPieces * (tlow + thigh);
      for (int p = I.p0; ok && p < I.p1; ++p) {
        const int plane0 = ((I.tile * A.nbp + p) * 2 + sg) * S;
        for (int piece = 0; piece < kPieces; ++piece, t2 += tlow + thigh) {
          if (!(ok = mbar_wait(bars.emptyL(sl), pl ^ 1u, wd, kSiteTmaEmpty))) break;
          uint32_t dst = ring + sl * R.lbytes;
          mbar_arrive_expect_tx(bars.fullL(sl), R.lbytes);
          armedL |= 1u << sl;
          parL = (parL & ~(1u << sl)) | (pl << sl);
          tma_load_3d(dst, &A.tmVl, bars.fullL(sl), piece * TPIECE, 0, plane0);
          bulk_load(dst + C::kLow * VP_PLANE, t2, tlow, bars.fullL(sl));
          if (++sl == R.nL) {
            sl = 0;
            pl ^= 1u;
          }
          if (!(ok = mbar_wait(bars.emptyH(sh), ph ^ 1u, wd, kSiteTmaEmpty))) break;
          dst = ring + R.hbase + sh * R.hbytes;
          mbar_arrive_expect_tx(bars.fullH(sh), R.hbytes);
          armedH |= 1u << sh;
          parH = (parH & ~(1u << sh)) | (ph << sh);
          tma_load_3d(dst, &A.tmVh, bars.fullH(sh), piece * TPIECE, 0, plane0 + C::kLow);
          bulk_load(dst + C::kHigh * VP_PLANE, t2 + tlow, thigh, bars.fullH(sh));
          if (++sh == R.nH) {
            sh = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) {  // the copies in flight land before the CTA leaves
        DrainWatch dw(Lp.status, Lp.timeout_ns);
        for (int s = 0; s < C::kMaxL; ++s) {
          if (armedL & (1u << s)) mbar_wait(bars.fullL(s), (parL >> s) & 1u, dw.wd, kSiteTmaFull);
          if (armedH & (1u << s)) mbar_wait(bars.fullH(s), (parH >> s) & 1u, dw.wd, kSiteTmaFull);
        }
      }
    }
  } else if (warp == 1) {
    // ================================================================ MMA issuer
    // The instructions around the MMAs count: the low descriptor words of a piece
    // (address / 16 and the fixed bit; shared addresses stay below 2^18, so
    // adding offsets never carries into it) are sums of two registers, and the
    // piece loops stay rolled.
    {
      const uint32_t usc = uniform(sc), utm = uniform(tmem), ulb = uniform(R.lbytes), uhb = uniform(R.hbytes), uhbase = uniform(R.hbase);
      const int unL = (int)uniform(R.nL), unH = (int)uniform(R.nH), up0 = (int)uniform(I.p0), up1 = (int)uniform(I.p1);
      const uint32_t uring = uniform(ring);
      const Bars2 bars{uring + C::kRing};
      int sl = 0, sh = 0;
      uint32_t pl = 0, ph = 0, g = 0;
      const uint64_t hi32 = (uint64_t)desc_hi(256, kSwizzle32) << 32;
      const uint32_t id = idesc_bf16(128, (int)usc), id2 = idesc_bf16(128, 2 * (int)usc);
      const bool wide3 = 3 * usc <= 256;
      const uint32_t id3 = idesc_bf16(128, wide3 ? 3 * (int)usc : 16);
      const uint32_t d1 = utm + usc, d2 = d1 + usc, d3 = d2 + usc;
      constexpr uint32_t vplane = VP_PLANE >> 4;
      const uint32_t trow = usc * 2u;  // bytes of one tau+- slice / 16
      const uint32_t tl0 = C::kLow * vplane, th0 = C::kHigh * vplane;
      bool ok = true;
      for (int p = up0; ok && p < up1; ++p, ++g) {
        // orders >= 3, waiting for each piece's operands; slices 3.. go back after them
        const int sl0 = sl;
        if (!(ok = mbar_wait_warp(bars.cfree(1), (g & 1u) ^ 1u, wd, kSiteRFree))) break;
        tc_fence_after();
#pragma unroll 1
        for (int piece = 0; piece < kPieces; ++piece) {
          if (!(ok = mbar_wait_warp(bars.fullL(sl), pl, wd, kSiteTmaFull))) break;
          if (!(ok = mbar_wait_warp(bars.fullH(sh), ph, wd, kSiteTmaFull))) break;
          const uint32_t lo = ((uring + sl * ulb) >> 4) | (1u << 16);
          const uint32_t hi = ((uring + uhbase + sh * uhb) >> 4) | (1u << 16);
          uint32_t v[S], t[S];
#pragma unroll
          for (int s = 0; s < S; ++s) {
            v[s] = s < C::kLow ? lo + s * vplane : hi + (s - C::kLow) * vplane;
            t[s] = s == 0 ? lo + tl0 : s == C::kLow ? hi + th0 : t[s - 1] + trow;
          }
          uint32_t acc3 = piece ? 1u : 0u;
#pragma unroll
          for (int pa = 0; pa < S; ++pa)
#pragma unroll
            for (int q = (pa < 3 ? 3 - pa : 0); q < S - pa; ++q) {
              mma_bf16_warp(d3, hi32 | v[pa], hi32 | t[q], id, acc3);
              acc3 = 1u;
            }
          mma_commit_warp(bars.emptyH(sh));
          if (++sl == unL) {
            sl = 0;
            pl ^= 1u;
          }
          if (++sh == unH) {
            sh = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        mma_commit_warp(bars.cfull(1));
        // orders 0 to 2: slice 0 of V+- against slices 0, 1 (and 2) of tau+- and slice 1 against
        // 0 and 1 as one MMA each; a piece's slices 0..2 go back after them
        if (!(ok = mbar_wait_warp(bars.cfree(0), (g & 1u) ^ 1u, wd, kSiteRFree))) break;
        tc_fence_after();
        int si = sl0;
#pragma unroll 1
        for (int piece = 0; piece < kPieces; ++piece) {
          const uint32_t v0 = ((uring + si * ulb) >> 4) | (1u << 16), t0 = v0 + tl0;
          if (wide3) {
            mma_bf16_warp(utm, hi32 | v0, hi32 | t0, id3, piece ? 1u : 0u);
          } else {
            mma_bf16_warp(utm, hi32 | v0, hi32 | t0, id2, piece ? 1u : 0u);
            mma_bf16_warp(d2, hi32 | v0, hi32 | (t0 + 2 * trow), id, piece ? 1u : 0u);
          }
          mma_bf16_warp(d1, hi32 | (v0 + vplane), hi32 | t0, id2, 1u);
          mma_bf16_warp(d2, hi32 | (v0 + 2 * vplane), hi32 | t0, id, 1u);
          mma_commit_warp(bars.emptyL(si));
          if (++si == unL) si = 0;
        }
        mma_commit_warp(bars.cfull(0));
      }
      mma_commit_warp(bars.done());
      DrainWatch dw(Lp.status, Lp.timeout_ns);
      mbar_wait(bars.done(), 0, dw.wd, kSiteRFull);
    }
  } else {
    // ================================================================ drains -> sums
    // As the MMA issuer commits them: orders >= 3 (2^-24 below the window) fused
    // into the low words, where the rounding is 2^-48 of the window; then orders
    // 0 to 2 joined as in pass 1 and scaled by the pair's row scales (exact
    // powers of two), one TwoSum into the double-single sums; two columns per
    // f32x2 instruction.
    const int quad = warp & 3;
    const int cw = (int)sc / 4, ng = cw / 4;  // this warp's columns and their groups of four
    const int col0 = ((warp - 2) >> 2) * cw;
    const int L = quad * 32 + lane;  // TMEM lane = ab row of the tile
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)col0;
    uint32_t g = 0;
    bool ok = true;
    float2 H[16], Lo[16];  // (hi, lo) sums of columns col0 + 2k and 2k + 1 (as .x and .y)
#pragma unroll
    for (int e = 0; e < 16; ++e) H[e] = Lo[e] = make_float2(0.f, 0.f);
    for (int p = I.p0; ok && p < I.p1; ++p, ++g) {
      const float *svp = A.sV + ((size_t)(I.tile * A.nbp + p) * 2 + sg) * 128 + L;
      const float *st = A.sT + ((size_t)I.ch * A.nbp + p) * kOzMaxCols + col0;
      // this pair's scales into L1 while its MMAs run
      asm volatile("prefetch.global.L1 [%0];" ::"l"(st));
      asm volatile("prefetch.global.L1 [%0];" ::"l"(svp));
      if (!(ok = mbar_wait(bars.cfull(1), g & 1u, wd, kSiteRFull))) break;
      tc_fence_after();
      const float sv = *svp;
      const float2 sv2 = make_float2(sv, sv);
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        if (h < ng) {
          float g3[4];
          tmem_ld4(tl + 4u * h + 3 * sc, g3);
          const float4 t0 = *reinterpret_cast<const float4 *>(st + 4 * h);
          tmem_ld_wait();
          const float2 s01 = mul2(sv2, make_float2(t0.x, t0.y)), s23 = mul2(sv2, make_float2(t0.z, t0.w));
          Lo[2 * h] = fma2(make_float2(g3[0], g3[1]), s01, Lo[2 * h]);
          Lo[2 * h + 1] = fma2(make_float2(g3[2], g3[3]), s23, Lo[2 * h + 1]);
        }
      }
      tc_fence_before();
      mbar_arrive(bars.cfree(1));
      if (!(ok = mbar_wait(bars.cfull(0), g & 1u, wd, kSiteRFull))) break;
      tc_fence_after();
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        if (h < ng) {
          float g0[4], g1[4], g2[4];
          const uint32_t c0 = tl + 4u * h;
          tmem_ld4(c0, g0);
          tmem_ld4(c0 + sc, g1);
          tmem_ld4(c0 + 2 * sc, g2);
          const float4 t0 = *reinterpret_cast<const float4 *>(st + 4 * h);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float2 s2 = mul2(sv2, e ? make_float2(t0.z, t0.w) : make_float2(t0.x, t0.y));
            float2 h0, er, hh, ll;
            fast_two_sum2(make_float2(g0[2 * e], g0[2 * e + 1]), make_float2(g1[2 * e], g1[2 * e + 1]), h0, er);
            fast_two_sum2(h0, add2(er, make_float2(g2[2 * e], g2[2 * e + 1])), hh, ll);
            ds_acc2(H[2 * h + e], Lo[2 * h + e], mul2(hh, s2), mul2(ll, s2));
          }
        }
      }
      tc_fence_before();
      mbar_arrive(bars.cfree(0));
    }
    // this unit's sums, [col][lane]
    if (ok)
#pragma unroll
      for (int h = 0; h < 8; ++h)
        if (h < ng)
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const size_t c = (size_t)(col0 + 4 * h + 2 * k);
            I.racc[c * 128 + L] = make_float2(H[2 * h + k].x, Lo[2 * h + k].x);
            I.racc[(c + 1) * 128 + L] = make_float2(H[2 * h + k].y, Lo[2 * h + k].y);
          }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ============================================================================ preparation
// The scale 2^(E - 8) of a row whose largest magnitude has the bit pattern mb
// (finite), 2^E the least power of two above it; 0 for a zero row, and below
// FP32's range.
__device__ __forceinline__ float row_scale(unsigned long long mb) {
  if (mb == 0) return 0.f;
  const int e = (int)(mb >> 52);
  const int E = e ? e - 1022 : -1010 - __clzll((long long)mb);  // subnormal: units of 2^-1074
  if (E - 8 > 127) return __int_as_float(0x7f800000);
  if (E - 8 >= -126) return pow2f(E - 8);
  return E - 8 >= -149 ? __int_as_float(1 << (E - 8 + 149)) : 0.f;
}
// log2 of a row scale (a positive power of two)
__device__ __forceinline__ int scale_exp(float s) {
  const int b = __float_as_int(s);
  return b >> 23 ? (b >> 23) - 127 : 31 - __clz(b) - 149;
}

// First launch of the preparation: row scales of B, and where B is declared
// symmetric the check of it, in blocks of their own (as the slices of B and of
// tau+- below: two launches for four, 92 -> 78 us a step at o=4, v=24).
//
// Scales: the smallest E with max_P |B^P_ac| < 2^E gives row (a, c) its scale
// 2^(E - 8) (0 for a zero row or a padding row).  One block per 32 rows (a,
// c0 .. c0 + 31), its 16 warps sharing the P: one read of B at HBM rate, where
// one thread per row left most of the chip idle (125 -> 22 us at v = 120,
// N = 480).  A NaN or infinite element records kSiteNonFinite.
//
// Check: B^P_ac = B^P_ca for every P and a, c < v (bitwise) on 32 x 32 tiles of
// the upper triangle; a mismatch records kSiteAsymmetric.
constexpr int kScaleWarps = 16;
constexpr int kCheckP = 4;  // auxiliary functions per checking block (1, 4, 16: 34, 31, 40 us at v = 120, 550, 486, 487 at v = 300)
__global__ void __launch_bounds__(32 * kScaleWarps, 3)
    oz_scale_kernel(int N, int v, int vp, const double *__restrict__ B, float *__restrict__ rs, int *status, int nscale,
                    int nsym) {
  dep_sync();
  __shared__ double buf[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if ((int)blockIdx.x >= nscale) {
    const int blk = (int)blockIdx.x - nscale, ntri = ppos((v + 31) / 32);
    int ta, tc;
    pair_of(blk % ntri, ta, tc);
    bool bad = false;
    for (int P = blk / ntri; P < N; P += nsym / ntri) {
      const double *Bp = B + (size_t)P * v * v;
      __syncthreads();
      for (int y = ty; y < 32; y += kScaleWarps) {
        const int a = tc * 32 + y, c = ta * 32 + tx;
        if (a < v && c < v) buf[y][tx] = Bp[(size_t)a * v + c];
      }
      __syncthreads();
      for (int y = ty; y < 32; y += kScaleWarps) {
        const int a = ta * 32 + y, c = tc * 32 + tx;
        if (a < v && c < v) bad |= __double_as_longlong(Bp[(size_t)a * v + c]) != __double_as_longlong(buf[tx][y]);
      }
    }
    if (bad) record_status(status, kSiteAsymmetric);
    return;
  }
  unsigned long long(*red)[33] = reinterpret_cast<unsigned long long(*)[33]>(buf);
  const int nx = (vp + 31) / 32, a = (int)blockIdx.x / nx, c = ((int)blockIdx.x % nx) * 32 + tx;
  // the largest |B^P_ac| as the largest magnitude bit pattern (the order of
  // non-negative doubles; NaN and infinity have an all-ones exponent), on the
  // integer pipe
  unsigned long long mb = 0;
  if (a < v && c < v) {
    const double *p = B + (size_t)a * v + c;
    const size_t step = (size_t)v * v;
#pragma unroll 4
    for (int P = ty; P < N; P += kScaleWarps)
      mb = max(mb, (unsigned long long)__double_as_longlong(__ldg(p + P * step)) & 0x7fffffffffffffffull);
  }
  red[ty][tx] = mb;
  __syncthreads();
  if (ty || c >= vp) return;
#pragma unroll
  for (int w = 1; w < kScaleWarps; ++w) mb = max(mb, red[w][tx]);
  const bool bad = mb >= 0x7ff0000000000000ull;
  if (bad) record_status(status, kSiteNonFinite);
  rs[(size_t)a * vp + c] = bad ? 0.f : row_scale(mb);
}

// The S fixed-point slices of x (|x| < 2^E, step = 2^(E - 8 S), the unit of
// the last slice): x rounded to the nearest multiple of the step, as balanced
// base-256 digits x_0 in [-256, 256], x_s in [-128, 127], digit s stored as
// the BF16 number x_s 2^(-8 s) (exact).  Integer arithmetic throughout: the
// FP64 pipe (four instructions per element before) was what bound the slicing.
template <int S>
__device__ __forceinline__ void fixed_slices(double x, int step_exp, float (&out)[S]) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((unsigned long long)b >> 52) & 0x7ff;
  long long m = b & 0xfffffffffffffll;
  if (e) m |= 1ll << 52;
  const int s = max(e, 1) - 1075 - step_exp;  // x = m 2^(e - 1075)
  if (s >= 0)
    m = s < 11 ? m << s : 0;  // s <= 8 S - 52 for |x| < 2^E
  else if (s > -55)
    m = (m + (1ll << (-s - 1))) >> (-s);
  else
    m = 0;
  if (b < 0) m = -m;
#pragma unroll
  for (int q = S - 1; q > 0; --q) {
    const int d = (int)(signed char)(m & 0xff);
    out[q] = (float)d * pow2f(-8 * q);
    m = (m - d) >> 8;
  }
  out[0] = (float)(int)m;
}

// Bt[s][a][c][P] = slice s of B^P_ac / scale(a, c), 64 (P) x 32 (c) tiles
// through shared memory (read c fastest, write P fastest, 128 bytes per warp);
// zero beyond v and N.  Bound by HBM: 8 B read and 2 S B written per element
// (77 -> 42 us at v = 120, N = 480, S = 5).
template <int S>
__device__ __forceinline__ void split_B(int blk, int N, int v, int vp, int Np, const double *__restrict__ B,
                                        const float *__restrict__ rs, __nv_bfloat16 *__restrict__ Bt) {
  __shared__ double tile[32][65];
  const int nx = (vp + 31) / 32, ny = (Np + 63) / 64, a = blk / (nx * ny);
  const int c0 = blk % nx * 32, P0 = blk / nx % ny * 64;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
#pragma unroll
  for (int r = ty; r < 64; r += 8) {
    const int P = P0 + r, c = c0 + tx;
    tile[tx][r] = (P < N && c < v && a < v) ? __ldg(B + ((size_t)P * v + a) * v + c) : 0.0;
  }
  __syncthreads();
  const size_t slice = (size_t)vp * vp * Np;
  const int P = P0 + 2 * tx;
  if (P >= Np) return;
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int c = c0 + r;
    if (c >= vp) break;
    const float sc = rs[(size_t)a * vp + c];
    float x[S], y[S];
    if (sc > 0.f) {
      const int step = scale_exp(sc) - 8 * (S - 1);
      fixed_slices<S>(tile[r][2 * tx], step, x);
      fixed_slices<S>(tile[r][2 * tx + 1], step, y);
    } else {
#pragma unroll
      for (int q = 0; q < S; ++q) x[q] = y[q] = 0.f;
    }
    const size_t off = ((size_t)a * vp + c) * Np + P;
#pragma unroll
    for (int q = 0; q < S; ++q)
      *reinterpret_cast<__nv_bfloat162 *>(Bt + q * slice + off) = __floats2bfloat162_rn(x[q], y[q]);
  }
}

// GEMM2 operand: for chunk c, 16-slot piece x (block pair x / 4) and slice s,
// the chunk's rows (lambda+ rows, padding, lambda- rows, padding) of 32 bytes,
// stored [x][s][row] in the 32-byte-swizzled order of shared memory, as
// pack_t2 does.  Eight threads share one (row, block pair): thread cl takes
// c = 8k + cl, d = 8l + 0..7 (piece cl / 2, half cl % 2), the group's maximum
// gives the row's scale for the pair, written to sT[c][pair][row].
//   tau+ = w (tau^cd + tau^dc),  tau- = w (tau^cd - tau^dc),  w = 1/4 (k = l), 1/2.
template <int S>
__device__ __forceinline__ void pack_t2(int bx, int nx, int chunk, const OzPackArgs &a) {
  const TcChunk CH = a.chunks[chunk];
  const int ncol = CH.nps + CH.nms;
  const size_t groups = (size_t)ncol * a.nbp;
  uint4 *dst = reinterpret_cast<uint4 *>(a.T2 + CH.t2off);
  const int cl = threadIdx.x & 7;
  const size_t g0 = ((size_t)bx * 256 + threadIdx.x) >> 3;
  const size_t gstep = ((size_t)nx * 256) >> 3;
  const size_t vv = (size_t)a.v * a.v;
  // every thread runs the same number of iterations (the shuffles below take
  // the whole warp)
  const size_t niter = (groups + gstep - 1) / gstep;
  for (size_t it = 0; it < niter; ++it) {
    const size_t gi = g0 + it * gstep;
    const bool live_g = gi < groups;
    const int row = live_g ? (int)((unsigned)gi % (unsigned)ncol) : 0;
    const int p = live_g ? (int)((unsigned)gi / (unsigned)ncol) : 0;
    int k, l;
    pair_of(p, k, l);
    int i = 0, j = 0;
    bool live = false, plus = true;
    if (live_g && row < CH.np) {
      lam_plus(CH.lp0 + row, i, j);
      live = true;
    } else if (live_g && row >= CH.nps && row - CH.nps < CH.nm) {
      lam_minus(CH.lm0 + (row - CH.nps), i, j);
      live = true;
      plus = false;
    }
    const int c = k * CB + cl;
    const double *tij = a.tau + ((size_t)i * a.o + j) * vv;
    // tau_cd +- tau_dc; the weight w is a power of two and goes into the scale
    double val[8];
    unsigned long long mb = 0;
    bool bad = false;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int d = l * CB + e;
      double x = 0.0;
      if (live && c < a.v && d < a.v) {
        const double t_cd = tij[(size_t)c * a.v + d], t_dc = tij[(size_t)d * a.v + c];
        x = plus ? t_cd + t_dc : t_cd - t_dc;
        // (an overflowing sum of finite elements counts as a zero row below)
        if (((unsigned long long)__double_as_longlong(x) & 0x7ff0000000000000ull) == 0x7ff0000000000000ull)
          bad |= !(isfinite(t_cd) && isfinite(t_dc));
      }
      val[e] = x;
      mb = max(mb, (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull);
    }
    if (bad) record_status(a.status, kSiteNonFinite);
    mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 1));
    mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 2));
    mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, 4));
    if (!live_g) continue;
    const float sc = mb < 0x7ff0000000000000ull ? row_scale(mb) : 0.f;
    const float scale = sc * (k == l ? 0.25f : 0.5f);
    uint32_t sl[S][4];
    const int step = sc > 0.f ? scale_exp(sc) - 8 * (S - 1) : 0;
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      float xs[S], ys[S];
      fixed_slices<S>(sc > 0.f ? val[e] : 0.0, step, xs);
      fixed_slices<S>(sc > 0.f ? val[e + 1] : 0.0, step, ys);
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const __nv_bfloat162 b2 = __floats2bfloat162_rn(xs[s], ys[s]);
        sl[s][e / 2] = *reinterpret_cast<const uint32_t *>(&b2);
      }
    }
    const size_t x = (size_t)p * 4 + cl / 2;
    const int h = cl & 1;
#pragma unroll
    for (int s = 0; s < S; ++s)
      dst[((x * S + s) * ncol + row) * 2 + (h ^ ((row >> 2) & 1))] = make_uint4(sl[s][0], sl[s][1], sl[s][2], sl[s][3]);
    if (cl == 0) a.sT[((size_t)chunk * a.nbp + p) * kOzMaxCols + row] = scale;
  }
}

// Second launch of the preparation: the slices of B and of tau+-, in blocks of
// their own (either may be left out).
struct OzSliceArgs {
  const double *B;
  const float *rs;
  __nv_bfloat16 *Bt;
  int N, v, vp, Np, nsplit, npack;
  OzPackArgs pk;
};
template <int S>
__global__ void __launch_bounds__(256, 6) oz_slices_kernel(const __grid_constant__ OzSliceArgs a) {
  dep_sync();
  if ((int)blockIdx.x < a.nsplit) {
    split_B<S>(blockIdx.x, a.N, a.v, a.vp, a.Np, a.B, a.rs, a.Bt);
  } else {
    const int blk = (int)blockIdx.x - a.nsplit;
    pack_t2<S>(blk % a.npack, a.npack, blk / a.npack, a.pk);
  }
}

}  // namespace

void launch_oz_scale(int N, int v, int vp, const double *B, bool check, float *rs, int *status, cudaStream_t s) {
  const int nscale = (vp + 31) / 32 * vp, ntri = ppos((v + 31) / 32);
  const int nsym = check ? ntri * std::min((N + kCheckP - 1) / kCheckP, 4096) : 0;
  launch_dep(oz_scale_kernel, nscale + nsym, 32 * kScaleWarps, 0, s, N, v, vp, B, rs, status, nscale, nsym);
}

void launch_oz_slices(int N, int v, int vp, int Np, int nslices, const double *B, const float *rs, __nv_bfloat16 *Bt,
                      const OzPackArgs *pk, cudaStream_t s) {
  OzSliceArgs a{};
  a.B = B;
  a.rs = rs;
  a.Bt = Bt;
  a.N = N;
  a.v = v;
  a.vp = vp;
  a.Np = Np;
  a.nsplit = B ? (vp + 31) / 32 * ((Np + 63) / 64) * vp : 0;
  int blocks = a.nsplit;
  if (pk) {
    a.pk = *pk;
    // eight threads per (row, block pair), at most 512 blocks a chunk
    a.npack = std::min(512, (kOzMaxCols * pk->nbp * 8 + 255) / 256);
    blocks += a.npack * pk->nchunks;
  }
  if (nslices == 5)
    launch_dep(oz_slices_kernel<5>, blocks, 256, 0, s, a);
  else
    launch_dep(oz_slices_kernel<6>, blocks, 256, 0, s, a);
}

uint32_t oz_smem_bytes(int pass, int nslices) {
  if (pass == 1) return nslices == 5 ? Cfg1<5>::kSmem : Cfg1<6>::kSmem;
  return nslices == 5 ? Cfg2<5>::kSmem : Cfg2<6>::kSmem;
}

template <int S>
cudaError_t oz_attrs() {
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(oz_vstore_kernel<S, false>, at, (int)Cfg1<S>::kSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(oz_vstore_kernel<S, true>, at, (int)Cfg1<S>::kSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(oz_gemm2_kernel<S, false>, at, (int)Cfg2<S>::kSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(oz_gemm2_kernel<S, true>, at, (int)Cfg2<S>::kSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(oz_xsym_kernel<S, false>, at, (int)CfgX<S>::kSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(oz_xsym_kernel<S, true>, at, (int)CfgX<S>::kSmem);
  return e;
}

cudaError_t oz_init_attributes(int nslices) { return nslices == 5 ? oz_attrs<5>() : oz_attrs<6>(); }

// one CTA per work unit
cudaError_t launch_oz_vstore(const OzLaunch &L, int nslices, cudaStream_t s) {
  if (L.nitems <= 0) return cudaSuccess;
  const bool b = L.mols != nullptr;
  if (nslices == 5) {
    if (b)
      launch_dep(oz_vstore_kernel<5, true>, L.nitems, kThreads, Cfg1<5>::kSmem, s, L);
    else
      launch_dep(oz_vstore_kernel<5, false>, L.nitems, kThreads, Cfg1<5>::kSmem, s, L);
  } else {
    if (b)
      launch_dep(oz_vstore_kernel<6, true>, L.nitems, kThreads, Cfg1<6>::kSmem, s, L);
    else
      launch_dep(oz_vstore_kernel<6, false>, L.nitems, kThreads, Cfg1<6>::kSmem, s, L);
  }
  return cudaGetLastError();
}

cudaError_t launch_oz_gemm2(const OzLaunch &L, int nslices, cudaStream_t s) {
  if (L.nitems <= 0) return cudaSuccess;
  const bool b = L.mols != nullptr;
  if (nslices == 5) {
    if (b)
      launch_dep(oz_gemm2_kernel<5, true>, L.nitems, kThreads, Cfg2<5>::kSmem, s, L);
    else
      launch_dep(oz_gemm2_kernel<5, false>, L.nitems, kThreads, Cfg2<5>::kSmem, s, L);
  } else {
    if (b)
      launch_dep(oz_gemm2_kernel<6, true>, L.nitems, kThreads, Cfg2<6>::kSmem, s, L);
    else
      launch_dep(oz_gemm2_kernel<6, false>, L.nitems, kThreads, Cfg2<6>::kSmem, s, L);
  }
  return cudaGetLastError();
}

// one CTA per work unit of the distinct integral tiles
cudaError_t launch_oz_xsym(const OzLaunch &L, int nslices, cudaStream_t s) {
  if (L.nitems <= 0) return cudaSuccess;
  const bool b = L.mols != nullptr;
  if (nslices == 5) {
    if (b)
      launch_dep(oz_xsym_kernel<5, true>, L.nitems, kThreads, CfgX<5>::kSmem, s, L);
    else
      launch_dep(oz_xsym_kernel<5, false>, L.nitems, kThreads, CfgX<5>::kSmem, s, L);
  } else {
    if (b)
      launch_dep(oz_xsym_kernel<6, true>, L.nitems, kThreads, CfgX<6>::kSmem, s, L);
    else
      launch_dep(oz_xsym_kernel<6, false>, L.nitems, kThreads, CfgX<6>::kSmem, s, L);
  }
  return cudaGetLastError();
}

// one block per SM, each walking the units in their order, so that the units under
// way share integral tiles in L2 (two blocks per SM need 64 registers a thread and
// spill: 418 -> 743 us at v = 120)
cudaError_t launch_oz_vform(const OzLaunch &L, int nslices, int sm_count, cudaStream_t s) {
  if (L.nitems <= 0) return cudaSuccess;
  const int grid = std::min(L.nitems, sm_count);
  const bool b = L.mols != nullptr;
  if (nslices == 5) {
    if (b)
      launch_dep(oz_vform_kernel<5, true>, grid, 512, 0, s, L);
    else
      launch_dep(oz_vform_kernel<5, false>, grid, 512, 0, s, L);
  } else {
    if (b)
      launch_dep(oz_vform_kernel<6, true>, grid, 512, 0, s, L);
    else
      launch_dep(oz_vform_kernel<6, false>, grid, 512, 0, s, L);
  }
  return cudaGetLastError();
}

}  // namespace ladder
