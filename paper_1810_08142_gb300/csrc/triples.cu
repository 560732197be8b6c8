// Perturbative triples (Sec. II.A): the energy kernels.
//
//   E(T) = sum_ijk sum_abc (4 W_ijk^abc + W_ijk^bca + W_ijk^cab)
//                          (V_ijk^abc - V_ijk^cba) / (3 D_ijk^abc)
//   V_ijk^abc = W_ijk^abc + v_jk^bc t_i^a + v_ik^ac t_j^b + v_ij^ab t_k^c
//   D_ijk^abc = e_i + e_j + e_k - e_a - e_b - e_c
//
// W_ijk^abc itself (the permutation operator P over the six orderings of the
// two contractions of Sec. II.A, one two-segment GEMM per ordering) is
// accumulated by the CUDA-core GEMM of dress.cu or the tensor-core GEMMs of
// triples_tc.cu (BF16X6) and crt_gemm.cu (FP64), for a range of the sorted
// triples i >= j >= k at a time, into W[triple][a][b][c].  These kernels read
// that W, form V from it and the integrals v_jk^bc = (bj|ck) (stored
// [j][k][b][c]), and reduce the energy of the sorted triples in a fixed order:
//   triples_energy_kernel   one partial sum per (sorted triple, block of abc)
//   triples_sum_kernel      the partials of one triple
//   triples_final_kernel    the sums of all triples, one block
#include <algorithm>
#include <type_traits>

#include "kernels.h"

namespace ladder {
namespace {

constexpr int kTE = 256;  // threads per energy block
constexpr int kTriplesMaxBlocks = 1024;  // energy blocks per k (each walks several orbits)
constexpr int kTC = 8;    // edge of the (a, b, c) cube of one block

// Sorted triples.  W and V are symmetric under a simultaneous permutation of
// (i, j, k) and (a, b, c), and D is symmetric in each, so the energy of a
// permuted triple is the sum over abc of the same tensors with permuted
// virtual indices.  Relabelling the sum, the factor
//   Z^abc = 4 W^abc + W^bca + W^cab
// is unchanged (the two 3-cycles are conjugate to each other), and V^cba
// becomes V with one of the three transpositions of (a, b, c) applied.  Over
// the six orderings of a triple each transposition comes twice, so
//   sum over the distinct orderings of (i, j, k) of E_ijk
//     = m_ijk sum_abc Z^abc (3 V^abc - V^acb - V^bac - V^cba) / (3 D^abc)
// with m = 2 for i > j > k, 1 for two equal indices, 1/3 for i = j = k.  The
// W contractions then run only for i >= j >= k (a sixth of the triples).
//
// Blocks over (orbits of 8-wide index blocks, k <= j), each block walking
// orbits blockIdx.x, blockIdx.x + gridDim.x, ... (at most kTriplesMaxBlocks
// blocks per k, so the partials stay bounded).  An orbit is a
// sorted block triple A0 <= B0 <= C0 with its distinct orderings (6, 3 or
// 1): the elements (a, b, c) of every ordering's 8x8x8 cube need W only at
// the six index permutations of (a, b, c), and those lie in the cubes of the
// same orbit.  The block therefore copies each of the orbit's cubes of W[k]
// into shared memory once (coalesced rows of 8) and reads every permuted W
// from there, so W is read from memory once per k instead of six times.
// One partial sum per block, reduced in a fixed order.
template <typename T>
__global__ void __launch_bounds__(kTE) triples_energy_kernel(const TriplesArgs a, const T *__restrict__ W,
                                                             double *__restrict__ part, int per) {
  constexpr int kCube = kTC * kTC * kTC;
  __shared__ double red[kTE / 32];
  // dynamic shared memory: six cubes, then t1 of i, j, k and e_vir (v each)
  extern __shared__ __align__(16) unsigned char tri_smem[];
  T(*cube)[kTC][kTC][kTC + 1] = reinterpret_cast<T(*)[kTC][kTC][kTC + 1]>(tri_smem);
  int i, j, k;
  triple_of(a.t0 + (int)blockIdx.y, i, j, k);
  const int v = a.v, o = a.o;
  const int nc = (v + kTC - 1) / kTC;
  T *sti = reinterpret_cast<T *>(tri_smem) + 6 * kTC * kTC * (kTC + 1);
  T *stj = sti + v, *stk = stj + v, *sev = stk + v;
  const long long vv = (long long)v * v, v3 = vv * v;
  const T *Wk = W + (long long)blockIdx.y * v3;
  const T *oovv = static_cast<const T *>(a.oovv);
  const T *Ijk = oovv + ((long long)j * o + k) * vv;  // v_jk^bc at [b][c]
  const T *Iik = oovv + ((long long)i * o + k) * vv;  // v_ik^ac at [a][c]
  const T *Iij = oovv + ((long long)i * o + j) * vv;  // v_ij^ab at [a][b]
  // terms in T (FP32 mode: the FP64 pipe is scarce on this part, so the
  // singles and orbital energies are converted once per block), sums in FP64
  for (int x = threadIdx.x; x < v; x += kTE) {
    sti[x] = (T)a.t1[(long long)i * v + x];
    stj[x] = (T)a.t1[(long long)j * v + x];
    stk[x] = (T)a.t1[(long long)k * v + x];
    sev[x] = (T)a.e_vir[x];
  }
  const T eijk = (T)(a.e_occ[i] + a.e_occ[j] + a.e_occ[k]);
  // V^xyz = W^xyz + v_jk^yz t_i^x + v_ik^xz t_j^y + v_ij^xy t_k^z
  auto singles = [&](int x, int y, int z) -> T {
    return Ijk[y * v + z] * sti[x] + Iik[x * v + z] * stj[y] + Iij[x * v + y] * stk[z];
  };
  auto on_singles = [&](T s, int x, int y, int z) -> T {  // one multiply-add each
    s += Ijk[y * v + z] * sti[x];
    s += Iik[x * v + z] * stj[y];
    return s + Iij[x * v + y] * stk[z];
  };
  // the thread's sum: FP64 for T = double; for T = float a double-single
  // (hi, lo) kept with TwoSum on the FP32 pipe (about 48 bits), widened once
  double s = 0.0;
  float sh = 0.f, sl = 0.f;
  const int norb = nc * (nc + 1) * (nc + 2) / 6;
  for (int orb = blockIdx.x; orb < norb; orb += gridDim.x) {
    __syncthreads();  // the previous orbit's cubes are no longer read
    // orbit -> sorted block triple A <= B <= C (every thread for itself), its
    // distinct orderings pos[] and the cubes of (A,B,C), (B,C,A), (C,A,B),
    // (A,C,B), (B,A,C), (C,B,A) among them, four bits each
    int A, B, C;
    triple_of(orb, C, B, A);
    const int n = A == C ? 1 : (A == B || B == C) ? 3 : 6;
    // orderings as index digits (0 A, 1 B, 2 C), two bits each, first index lowest
    auto code = [](int x, int y, int z) { return x | y << 2 | z << 4; };
    const unsigned cid = n == 6 ? 0x521430u : n == 1 ? 0u : A == B ? 0x201210u : 0x210120u;
    auto position = [&](int p, int &X, int &Y, int &Z) {
      // n = 6: ABC ACB BAC BCA CAB CBA; A == B: AAC ACA CAA; B == C: ABB BAB BBA
      const int six[6] = {code(0, 1, 2), code(0, 2, 1), code(1, 0, 2), code(1, 2, 0), code(2, 0, 1), code(2, 1, 0)};
      const int aac[3] = {code(0, 0, 2), code(0, 2, 0), code(2, 0, 0)};
      const int abb[3] = {code(0, 1, 1), code(1, 0, 1), code(1, 1, 0)};
      const int w = n == 6 ? six[p] : p >= 3 ? 0 : A == B ? aac[p] : abb[p];
      auto pick = [&](int d) { return d == 0 ? A : d == 1 ? B : C; };
      X = pick(w & 3);
      Y = pick((w >> 2) & 3);
      Z = pick(w >> 4);
    };
    // the orbit's cubes: thread t copies elements t and t + 256 of each
#pragma unroll
    for (int p = 0; p < 6; ++p) {
      if (p >= n) break;
      int X0, Y0, Z0;
      position(p, X0, Y0, Z0);
#pragma unroll
      for (int h = 0; h < kCube / kTE; ++h) {
        const int e = threadIdx.x + h * kTE;
        const int x = e / (kTC * kTC), y = (e / kTC) % kTC, z = e % kTC;
        const int X = X0 * kTC + x, Y = Y0 * kTC + y, Z = Z0 * kTC + z;
        cube[p][x][y][z] = (X < v && Y < v && Z < v) ? Wk[(long long)X * vv + (long long)Y * v + Z] : T(0);
      }
    }
    __syncthreads();
    // One element (a, b, c) of the first cube at a time with all six index
    // permutations, so that each w, V and integral is read once instead of up
    // to six times.  In FP64 they share D, and with the even permutations (abc,
    // bca, cab) and the odd ones (acb, bac, cba) the sum of their terms is
    //   sum_p (3 w_p + sum of its parity's w) (3 V_p - sum of the other parity's V) / (3 D)
    //     = (sum_p w_p r_p + (w_even - w_odd) (V_even - V_odd)) / D,  r_p the second factor
    // (w_even and the like: sums), which knows w and V only up to a constant each: both
    // are taken less the first one's.  Of i = j = k they agree in all permutations,
    // and where one occupied orbital dominates what rounding leaves of its triple
    // exceeds E(T) (with factors of 2^-5 and 2^-10 between the occupied orbitals
    // errors of up to 1e-12 and 4e-8 with w and V as they are, 2e-16 so).
    // An orbit of two (one) distinct blocks visits every ordering twice (six
    // times).  At o = 10, v = 120 (FP32) 3.90 -> 1.8 ms in all, at o = 8, v = 60
    // (FP64, bound by the FP64 pipe) 3.44 -> 1.10 ms.
    const int X0 = A * kTC, Y0 = B * kTC, Z0 = C * kTC;
    const int c0 = cid & 15, c1 = (cid >> 4) & 15, c2 = (cid >> 8) & 15, c3 = (cid >> 12) & 15, c4 = (cid >> 16) & 15,
              c5 = cid >> 20;
    const T share = n == 6 ? T(1) : n == 3 ? T(0.5) : T(1) / T(6);
#pragma unroll
    for (int h = 0; h < kCube / kTE; ++h) {
      const int e = threadIdx.x + h * kTE;
      const int al = e / (kTC * kTC), bl = (e / kTC) % kTC, cl = e % kTC;
      const int aa = X0 + al, bb = Y0 + bl, cc = Z0 + cl;
      if (aa >= v || bb >= v || cc >= v) continue;
      const T w0 = cube[c0][al][bl][cl], w1 = cube[c1][bl][cl][al], w2 = cube[c2][cl][al][bl];
      const T w3 = cube[c3][al][cl][bl], w4 = cube[c4][bl][al][cl], w5 = cube[c5][cl][bl][al];
      if constexpr (std::is_same<T, float>::value) {
        const T x0 = w0 + singles(aa, bb, cc), x1 = w1 + singles(bb, cc, aa), x2 = w2 + singles(cc, aa, bb);
        const T x3 = w3 + singles(aa, cc, bb), x4 = w4 + singles(bb, aa, cc), x5 = w5 + singles(cc, bb, aa);
        // FP32: the six terms one by one, each rounded as it stands (their
        // common factors, taken out as below, would move E(T) by 3e-8)
        const float weight = n == 3 ? 0.5f : 1.f;  // n = 1: the first alone
        float ts[6];
        auto term = [&](float w, float wn, float wp, float x, float xa, float xb, float xc, int i1, int i2, int i3) {
          const float D = eijk - sev[i1] - sev[i2] - sev[i3];
          return (4.f * w + wn + wp) * (3.f * x - xa - xb - xc) / (3.f * D);
        };
        ts[0] = term(w0, w1, w2, x0, x3, x4, x5, aa, bb, cc);
        ts[1] = term(w1, w2, w0, x1, x4, x5, x3, bb, cc, aa);
        ts[2] = term(w2, w0, w1, x2, x5, x3, x4, cc, aa, bb);
        ts[3] = term(w3, w5, w4, x3, x0, x2, x1, aa, cc, bb);
        ts[4] = term(w4, w3, w5, x4, x1, x0, x2, bb, aa, cc);
        ts[5] = term(w5, w4, w3, x5, x2, x1, x0, cc, bb, aa);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          if (q && n == 1) break;
          const float y = weight * ts[q], x = __fadd_rn(sh, y), bp = __fsub_rn(x, sh);
          sl = __fadd_rn(sl, __fadd_rn(__fsub_rn(sh, __fsub_rn(x, bp)), __fsub_rn(y, bp)));
          sh = x;
        }
      } else {
        const T v1 = w1 - w0, v2 = w2 - w0, v3 = w3 - w0, v4 = w4 - w0, v5 = w5 - w0;
        // V minus the first one's
        const T s0 = singles(aa, bb, cc);
        const T y1 = on_singles(v1 - s0, bb, cc, aa), y2 = on_singles(v2 - s0, cc, aa, bb);
        const T y3 = on_singles(v3 - s0, aa, cc, bb), y4 = on_singles(v4 - s0, bb, aa, cc);
        const T y5 = on_singles(v5 - s0, cc, bb, aa);
        const T ye = y1 + y2, yo = y3 + y4 + y5;
        T t = (v1 + v2 - v3 - v4 - v5) * (ye - yo);
        t += v1 * (T(3) * y1 - yo);
        t += v2 * (T(3) * y2 - yo);
        t += v3 * (T(3) * y3 - ye);
        t += v4 * (T(3) * y4 - ye);
        t += v5 * (T(3) * y5 - ye);
        s += (double)(t * share / (eijk - sev[aa] - sev[bb] - sev[cc]));
      }
    }
  }  // orbits
  if constexpr (std::is_same<T, float>::value) s = (double)sh + (double)sl;
  // fixed-order reduction: warp shuffles, then the warps' sums in order
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kTE / 32; ++w) t += red[w];
    // multiplicity of the sorted triple (i >= j >= k)
    const double m = (i == k) ? 1.0 / 3.0 : (i == j || j == k) ? 1.0 : 2.0;
    part[(long long)(a.t0 + (int)blockIdx.y) * per + blockIdx.x] = m * t;
  }
}

// t2 in the GEMMs' element type (t2c, skipped when null) and with the two
// virtual indices exchanged (t2T[i][j][b][a] = t2[i][j][a][b]).
template <typename T>
__global__ void triples_t2_kernel(long long n, int v, const double *__restrict__ t2, T *__restrict__ t2c,
                                  T *__restrict__ t2T) {
  const long long vv = (long long)v * v;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const double x = t2[e];
    const long long ij = e / vv, ab = e % vv;
    if (t2c) t2c[e] = (T)x;
    t2T[ij * vv + (ab % v) * v + ab / v] = (T)x;
  }
}

// dst[g][x][y][d] = src[g][y][x][d]; consecutive threads take consecutive d
template <typename T>
__global__ void triples_swap12_kernel(const T *__restrict__ src, T *__restrict__ dst, long long n, int v) {
  const long long vv = (long long)v * v;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const long long g = e / (vv * v), r = e % (vv * v);
    const long long x = r / vv, y = (r / v) % v, d = r % v;
    dst[e] = src[g * vv * v + (y * v + x) * v + d];
  }
}

template <typename T>
__global__ void triples_negate_kernel(T *__restrict__ x, long long n) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    x[e] = -x[e];
}

// The `per` partials of triple blockIdx.x into its first: thread t sums
// partials t, t + 256, ... in order, then a tree.  (One block over all
// partials took 203 us of a 10.6 ms call at o = 10, v = 120.)
__global__ void __launch_bounds__(256) triples_sum_kernel(double *__restrict__ part, int per) {
  __shared__ double red[256];
  double *p = part + (long long)blockIdx.x * per;
  double s = 0.0;
  for (int q = threadIdx.x; q < per; q += 256) s += p[q];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) p[0] = red[0];
}

// One block: thread t sums the triples t, t + 1024, ... in order, then a tree.
// A nonzero *status (a bounded wait of a tensor-core W kernel ran out) makes
// the result NaN.
__global__ void __launch_bounds__(1024) triples_final_kernel(const double *__restrict__ part, int n, int per,
                                                             double *__restrict__ E, const int *status) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int q = threadIdx.x; q < n; q += 1024) s += part[(long long)q * per];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *E = (status && *status) ? __longlong_as_double(0x7ff8000000000000LL) : red[0];
}

// dynamic shared memory of the energy kernel for v virtual orbitals
template <typename T>
size_t triples_energy_smem(int v) {
  return (6 * kTC * kTC * (kTC + 1) + 4 * (size_t)v) * sizeof(T);
}

}  // namespace

// orbits of sorted 8-wide block triples
int triples_energy_blocks(int v) {
  const int nc = (v + kTC - 1) / kTC;
  return std::min(nc * (nc + 1) * (nc + 2) / 6, kTriplesMaxBlocks);
}

template <typename T>
cudaError_t launch_triples_energy(const TriplesArgs &a, const T *W, int nt, double *part, cudaStream_t s) {
  // about four waves of blocks, each walking several orbits: a block per orbit
  // spent most of its time setting up.  The partials beyond the grid stay zero.
  const int most = triples_energy_blocks(a.v), per = std::max(1, 152 * 24 / std::max(nt, 1));
  const dim3 grid((unsigned)std::min(most, per), (unsigned)nt);
  const size_t smem = triples_energy_smem<T>(a.v);
  if (smem > 48 * 1024) {  // FP64 at large v only; set on the current device
    const cudaError_t e =
        cudaFuncSetAttribute(triples_energy_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  triples_energy_kernel<T><<<grid, kTE, smem, s>>>(a, W, part, most);
  return cudaGetLastError();
}
template cudaError_t launch_triples_energy<double>(const TriplesArgs &, const double *, int, double *, cudaStream_t);
template cudaError_t launch_triples_energy<float>(const TriplesArgs &, const float *, int, double *, cudaStream_t);

template <typename T>
cudaError_t launch_triples_t2(int o, int v, const double *t2, T *t2c, T *t2T, cudaStream_t s) {
  const long long n = (long long)o * o * v * v;
  const long long blocks = std::min<long long>((n + 255) / 256, 8192);
  triples_t2_kernel<T><<<(unsigned)blocks, 256, 0, s>>>(n, v, t2, t2c, t2T);
  return cudaGetLastError();
}
template cudaError_t launch_triples_t2<double>(int, int, const double *, double *, double *, cudaStream_t);
template cudaError_t launch_triples_t2<float>(int, int, const double *, float *, float *, cudaStream_t);

namespace {
__global__ void triples_narrow_kernel(const double *__restrict__ x, float *__restrict__ y, long long n) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    y[e] = (float)x[e];
}
}  // namespace
cudaError_t launch_triples_narrow(const double *x, float *y, long long n, cudaStream_t s) {
  const long long blocks = std::max<long long>(1, std::min<long long>((n + 255) / 256, 152 * 16));
  triples_narrow_kernel<<<(unsigned)blocks, 256, 0, s>>>(x, y, n);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_triples_swap12(const T *src, T *dst, int G, int v, cudaStream_t s) {
  const long long n = (long long)G * v * v * v;
  const long long blocks = std::min<long long>((n + 255) / 256, 152 * 64);
  if (blocks > 0) triples_swap12_kernel<T><<<(unsigned)blocks, 256, 0, s>>>(src, dst, n, v);
  return cudaGetLastError();
}
template cudaError_t launch_triples_swap12<double>(const double *, double *, int, int, cudaStream_t);
template cudaError_t launch_triples_swap12<float>(const float *, float *, int, int, cudaStream_t);

template <typename T>
cudaError_t launch_triples_negate(T *x, long long n, cudaStream_t s) {
  const long long blocks = std::min<long long>((n + 255) / 256, 8192);
  if (blocks > 0) triples_negate_kernel<T><<<(unsigned)blocks, 256, 0, s>>>(x, n);
  return cudaGetLastError();
}
template cudaError_t launch_triples_negate<double>(double *, long long, cudaStream_t);
template cudaError_t launch_triples_negate<float>(float *, long long, cudaStream_t);

cudaError_t launch_triples_final(double *part, int n, int per, double *E, cudaStream_t s, const int *status) {
  triples_sum_kernel<<<n, 256, 0, s>>>(part, per);
  triples_final_kernel<<<1, 1024, 0, s>>>(part, n, per, E, status);
  return cudaGetLastError();
}

}  // namespace ladder
