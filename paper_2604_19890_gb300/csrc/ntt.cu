// NTT / inverse NTT over RNS limbs (Section 2.1 ring arithmetic), for the
// cyclotomic rings X^N + 1 (m = 2N) and X^N - X^(N/2) + 1 (m = 3N).
//
// Forward: merged-twist Cooley-Tukey with twiddles psi^bitrev(m+i); natural
// coefficients in, evaluation form out with word j = a(psi^(2 bitrev(j)+1)).
// Inverse: Gentleman-Sande with psi^-bitrev(m+i), then times N^-1.
// m = 3N: the same trees with node 1 replaced by the split into
// X^(N/2) - rho and X^(N/2) - rho^5 (R3 kernels) and the subtree twiddles of
// those two factors; word h N/2 + j = a(omega^(e_h + 6 bitrev(j))).
//
// A length-N transform is split N = N1 * N2. Its first log2(N1) stages act on
// the N2 columns (stride N2) independently, the remaining log2(N2) stages on
// the N1 contiguous chunks of N2 words. Each phase is one kernel whose CTAs hold
// tiles of 2048 or 4096 words in registers and shared memory. N <= 4096 runs in
// one phase.
// Three forms, by size and prime width:
//  * N >= 8192, primes below 2^55: k_ntt16_cols / k_ntt16_rows (products by
//    halves, below). One GB300, 328 limbs of 2^16 words: 0.565 us a limb forward
//    and 0.573 inverse, where the Shoup form takes 0.751 and 0.870.
//  * N >= 8192, wider primes: k_ntt16 (Shoup products: halves need nine spare bits).
//  * N <= 4096: k_ntt, one phase in shared memory with Harvey's lazy butterflies.
#include "launch.cuh"
#include "modarith.cuh"
#include "ss_internal.h"

namespace ss {

namespace {

__device__ __forceinline__ void cp16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}

constexpr int TILE = 4096;  // words per CTA tile (32 KiB of shared memory)

// resident CTAs per SM the radix-16 phases are compiled for (forward, inverse)
#ifndef SS_NTT_PREFETCH
#define SS_NTT_PREFETCH 1  // inverse chunk phase: first-stage twiddles loaded before the staging
#endif
#ifndef SS_NTT_MINB_F
#define SS_NTT_MINB_F 3
#endif
#ifndef SS_NTT_MINB_I
#define SS_NTT_MINB_I 3
#endif
// resident CTAs of 128 threads per SM that the phases of products by halves are compiled for (72 registers, 64 in
// the large column tiles and the fused inner product; they spill 4 to 60 bytes a thread for it. 328 limbs of 2^16
// words, us a limb forward / inverse at 5, 6, 7, 8 CTAs: 0.579/0.607, 0.569/0.593, 0.565/0.573, 0.576/0.587)
#ifndef SS_COLS_F
#define SS_COLS_F 7
#endif
#ifndef SS_COLS_I
#define SS_COLS_I 7
#endif
#ifndef SS_COLS_BIG
#define SS_COLS_BIG 4  // of 256 threads
#endif
#ifndef SS_ROWS_F
#define SS_ROWS_F 7
#endif
#ifndef SS_ROWS_I
#define SS_ROWS_I 7
#endif
#ifndef SS_ROWS_IP
#define SS_ROWS_IP 4  // CTAs of 256 threads
#endif
#ifndef SS_NTT_MINB_R5
#define SS_NTT_MINB_R5 3  // m = 5N/2 column phases (the factored split fits the same 80 registers)
#endif

struct NttArgs {
  u64* base;
  long outer_stride;
  int n_outer, nl, q0, nq, L, N;
  int skip_w, skip_mod, skip_level;
  const Modulus* mods;
  const u64* tw;     // per prime 4N words: twiddle word pairs forward, then inverse ((w, w') or (w_0, w_1), TwRow)
  const u32* tp;     // products by halves: the half-quotients (p_0, p_1) beside A.tw's pairs; else null
  int tws;           // products by halves: slots per prime and direction, N + N1 (half_tw)
  const u64* ninv;   // per prime (N^-1, shoup, N^-1 psi^(-N/2), shoup, m = 3N: (2 rho - 1)^-1 N^-1, shoup)
  const u64* split;  // m = 5N/2: per prime 12 (value, shoup) pairs of the four-way split (split4_fwd/inv)
  const u64* src;    // out-of-place first phase: polynomial (o, i) is read at src + o src_os + i N
  long src_os;
  int pre_w1;        // forward, X^N + 1: upper halves already carry psi^(N/2) (PolySet::pre_w1)
  int post_scale;    // inverse, X^N + 1: last stage without its products (PolySet::post_scale)
};

// Blocks walk the polynomials limb-major (all outer copies of limb 0, then of
// limb 1, ...) so consecutive blocks share a prime and its twiddles stay in L2.
__device__ __forceinline__ bool poly_of(const NttArgs& A, int poly, u64*& ptr, int& pidx) {
  int i = poly / A.n_outer, o = poly % A.n_outer;
  if (A.skip_w > 0) {
    int j = o % A.skip_mod;
    int lo = j * A.skip_w, hi = min(lo + A.skip_w, A.skip_level);
    if (i >= lo && i < hi && i < A.nq) return false;
  }
  ptr = A.base + (long)o * A.outer_stride + (long)i * A.N;
  pidx = i < A.nq ? A.q0 + i : A.L + (i - A.nq);
  return true;
}

// Shared-memory word for linear tile index `lin`: one pad word per 8, which
// spreads the strided round accesses over all banks.
__device__ __forceinline__ int swz(int lin) { return lin + (lin >> 3); }

#ifndef SS_NTT_XSWZ
#define SS_NTT_XSWZ 1  // chunk phases of the radix-16 kernels: XOR swizzle instead of the padded one
#endif
// Chunk tiles of the radix-16 kernels: within every aligned group of 16 words
// the low four index bits are XORed with the next four. A half-warp then hits
// 16 distinct bank pairs both when it touches 16 consecutive words (rounds of
// spacing >= 16, the linear staging loops: the XOR is one permutation of the
// group) and when it touches one word of each of 16 consecutive groups
// (rounds of spacing 1: thread B holds words 16B .. 16B+15), where the padded
// swizzle left two threads on each bank pair. It needs no padding.
template <bool COLS>
__device__ __forceinline__ int swz16(int lin) {
  if (COLS || !SS_NTT_XSWZ) return swz(lin);
  return lin ^ ((lin >> 4) & 15);
}

// Slot of node `widx` of a stage of half-distance 2^logt. In the round of
// spacing 1 neighbouring threads hold neighbouring groups G of 16 words, and a
// stage of half-distance below 8 has 2^(3 - logt) twiddles per group: stored
// group by group, one load of a warp would touch a line per thread (340
// wavefronts of the L1 path a round and warp, which then bounded the chunk
// phases at 90 % of its rate). So those stages store, for each block of 2^wb
// groups, first every group's first twiddle, then every group's second, and so on.
__host__ __device__ __forceinline__ int tw_slot(int widx, int logt, int wb) {
  if (logt >= 3) return widx;
  const int g = widx >> (3 - logt), i = widx & ((1 << (3 - logt)) - 1);
  return ((g >> wb) << (wb + 3 - logt)) + (i << wb) + (g & ((1 << wb) - 1));
}

// Tables of products by halves, per prime and direction: slots [0, N1) hold the
// column phase's nodes, slots N1 + c N2 + l node l of chunk c's own subtree.
template <bool FWD>
__device__ __forceinline__ const ulonglong2* half_tw(const NttArgs& A, int pidx) {
  return reinterpret_cast<const ulonglong2*>(A.tw) + (size_t)(2 * pidx + (FWD ? 0 : 1)) * A.tws;
}
template <bool FWD>
__device__ __forceinline__ const uint2* half_tp(const NttArgs& A, int pidx) {
  return reinterpret_cast<const uint2*>(A.tp) + (size_t)(2 * pidx + (FWD ? 0 : 1)) * A.tws;
}

// v < 64q  ->  v mod q. The quotient estimate k = floor(t * mq / 2^24) from
// t = floor(v / 2^(kb-8)) and mq = floor(2^(kb+16) / q) satisfies
// v/q - 2 < k <= v/q, so v - k q lies in [0, 2q) and one subtraction ends it.
__device__ __forceinline__ u64 reduce_lazy(u64 v, u64 q, int kb, uint32_t mq) {
  const uint32_t t = (uint32_t)(v >> (kb - 8));
  const uint32_t k = (t * mq) >> 24;
  const u64 r = v - (u64)k * q;
  return r >= q ? r - q : r;
}

// Products by halves: per-prime constants of the reductions.
struct HalfMod {
  u64 q, nq2;     // q, -2q mod 2^64
  u32 n0, n1;     // -q mod 2^64
  u32 mq, s1, s2; // floor(2^(kb+16) / q); v >> (kb - 6) as a funnel shift by s1 <= 32 and a shift by s2
};
__device__ __forceinline__ HalfMod half_mod(const Modulus& m) {
  HalfMod h;
  h.q = m.q;
  h.nq2 = 0 - 2 * m.q;
  h.n0 = (u32)(0 - m.q);
  h.n1 = (u32)((0 - m.q) >> 32);
  h.mq = (u32)(m.mu >> 47);
  const int s = m.kbits - 6;
  h.s1 = s < 32 ? s : 32;
  h.s2 = s < 32 ? 0 : s - 32;
  return h;
}
// v < 512q (q below 2^55)  ->  v mod q in [0, 2q): the quotient estimate
// k = floor(t mq / 2^22) from t = floor(v / 2^(kb-6)), t mq <= (v / q) 2^22 < 2^31;
// the truncations leave v/q - k below 1 + 2^-5 + 2^-7.
__device__ __forceinline__ u64 reduce_half(u64 v, const HalfMod& m) {
  const u32 lo = (u32)v, hi = (u32)(v >> 32);
  const u32 k = ((__funnelshift_rc(lo, hi, m.s1) >> m.s2) * m.mq) >> 22;
  u32 r0, r1;
  asm("mad.lo.cc.u32 %0, %2, %3, %5;\n\tmadc.hi.u32 %1, %2, %3, %6;\n\tmad.lo.u32 %1, %2, %4, %1;"
      : "=&r"(r0), "=&r"(r1)
      : "r"(k), "r"(m.n0), "r"(m.n1), "r"(lo), "r"(hi));
  return ((u64)r1 << 32) | r0;
}

// m = 5N/2: the four-way split of Phi_10(X^(N/4)) on four words a_j (the
// quarters' words at one position), factored through the quadratics
// y^2 - c y + 1 = (y - xi^e)(y - xi^-e), c = xi^e + xi^-e, e = 1 and 3. Both
// c are roots of c^2 = c + 1 (c_1 + c_3 = 1, c_1 c_3 = -1), so a mod the
// quadratic is (a0 - a2 - c a3) + (a1 + c (a2 + a3)) y and the two
// quadratics share the products c_1 a3 and c_1 (a2 + a3); each remainder is
// then evaluated at its two roots. Forward: 6 Shoup products per 4 words,
// inputs below 4q give outputs below 16q, in the order xi^1, xi^3, xi^7, xi^9.
// Inverse (inputs below B; off a multiple of q, B <= off and B + off + 2q < 2^64:
// every difference lifted by off or off + q stays in one positive word): the
// remainders from the root values, then
// a3 = (r0 - s0) / (1 - 2 c_1), a2 + a3 = (s1 - r1) / (1 - 2 c_1),
// a1 = r1 - c_1 (a2 + a3), a0 = r0 + a2 + c_1 a3, scaled by 4/N: 10 products,
// canonical. Constants per prime (value, Shoup pairs): forward c_1, xi, xi^3,
// xi^7, xi^9; inverse (xi - xi^9)^-1, xi, (xi^3 - xi^7)^-1, xi^3,
// (1 - 2 c_1)^-1 4/N, 4/N, c_1.
constexpr int kSplitWords = 24;
__device__ __forceinline__ void split4_fwd(u64& a0, u64& a1, u64& a2, u64& a3, const ulonglong2* __restrict__ c,
                                           u64 q) {
  const ulonglong2 c1 = __ldg(c);
  const u64 t3 = shoup_lazy(a3, c1.x, c1.y, q);
  const u64 t23 = shoup_lazy(a2 + a3, c1.x, c1.y, q);
  const u64 r0 = a0 + 6 * q - a2 - t3;
  const u64 r1 = a1 + t23;
  const u64 s0 = a0 + t3 + 8 * q - a2 - a3;
  const u64 s1 = a1 + a2 + a3 + 2 * q - t23;
  const ulonglong2 x1 = __ldg(c + 1), x3 = __ldg(c + 2), x7 = __ldg(c + 3), x9 = __ldg(c + 4);
  a0 = r0 + shoup_lazy(r1, x1.x, x1.y, q);
  a3 = r0 + shoup_lazy(r1, x9.x, x9.y, q);
  a1 = s0 + shoup_lazy(s1, x3.x, x3.y, q);
  a2 = s0 + shoup_lazy(s1, x7.x, x7.y, q);
}
__device__ __forceinline__ void split4_inv(u64& b0, u64& b1, u64& b2, u64& b3, const ulonglong2* __restrict__ c,
                                           u64 q, u64 off) {
  const ulonglong2 k1 = __ldg(c + 5), x1 = __ldg(c + 6), k3 = __ldg(c + 7), x3 = __ldg(c + 8);
  const u64 r1 = shoup(b0 - b3 + off, k1.x, k1.y, q);
  const u64 r0 = b0 + q - shoup(r1, x1.x, x1.y, q);
  const u64 s1 = shoup(b1 - b2 + off, k3.x, k3.y, q);
  const u64 s0 = b1 + q - shoup(s1, x3.x, x3.y, q);
  const ulonglong2 d = __ldg(c + 9), sg = __ldg(c + 10), c1 = __ldg(c + 11);
  const u64 a3 = shoup(r0 - s0 + off + q, d.x, d.y, q);
  const u64 S = shoup(s1 - r1 + q, d.x, d.y, q);
  const u64 a2 = S >= a3 ? S - a3 : S + q - a3;
  const u64 u1 = shoup(r1, sg.x, sg.y, q), v1 = shoup(S, c1.x, c1.y, q);
  const u64 a1 = u1 >= v1 ? u1 - v1 : u1 + q - v1;
  u64 a0 = shoup(r0, sg.x, sg.y, q) + a2 + shoup(a3, c1.x, c1.y, q);
  if (a0 >= 2 * q) a0 -= 2 * q;
  if (a0 >= q) a0 -= q;
  b0 = a0;
  b1 = a1;
  b2 = a2;
  b3 = a3;
}

// One round of up to three radix-2 stages held in registers. The thread owns
// the eight words r_k = rbase + k*u (rbase = B*8u + o, o < u); the round's
// stages have half-distances t = u*2^j for j in [JLO, JHI] and pair the
// registers (k, k + 2^j). Butterflies of one 2t-block share one twiddle,
// index (mg << sg) + r/(2t), sg = logS - 1 - log2(t).
// R3 (m = 3N): node 1 (twiddle index 1) is the split of X^N - X^(N/2) + 1 into
// X^(N/2) - rho and X^(N/2) - rho^5 (rho^5 = 1 - rho): forward (U, V) ->
// (U + rho V, U + V - rho V); inverse t = (U - V)(2 rho - 1)^-1 ->
// (U + V - t, 2t), both scaled by N^-1 with the rest afterwards.
template <bool FWD, int JLO, int JHI, int RING>
__device__ __forceinline__ void ntt_round(u64 (&x)[8], int rbase, int logu, int logS, int mg,
                                          const ulonglong2* __restrict__ tw, u64 q, bool pre1) {
  const u64 q2 = 2 * q;
#pragma unroll
  for (int jj = JLO; jj <= JHI; ++jj) {
    const int j = FWD ? JHI + JLO - jj : jj;
    const int d = 1 << j;
    const int logt = logu + j;
    const int sg = logS - 1 - logt;
#pragma unroll
    for (int blk = 0; blk < 4 / d; ++blk) {
      const int k0 = blk * 2 * d;
      const int widx = (mg << sg) + ((rbase + (k0 << logu)) >> (logt + 1));
      const ulonglong2 wv = __ldg(tw + widx);
      const u64 w = wv.x, wp = wv.y;
#pragma unroll
      for (int p = 0; p < d; ++p) {
        const int k = k0 + p;
        u64 U = x[k], V = x[k + d];
        if (RING == 3 && widx == 1) {
          if (FWD) {  // residues stay below 4q
            if (U >= q2) U -= q2;
            if (V >= q2) V -= q2;
            const u64 t = shoup_lazy(V, w, wp, q);
            u64 z = V + q2 - t;
            if (z >= q2) z -= q2;
            x[k] = U + t;
            x[k + d] = U + z;
          } else {
            const u64 t = shoup_lazy(U - V + q2, w, wp, q);
            x[k] = U + V + q2 - t;
            x[k + d] = t + t;
          }
        } else if (FWD) {
          if (U >= q2) U -= q2;
          if (!(pre1 && widx == 1)) V = shoup_lazy(V, w, wp, q);  // pre1: node 1's product already applied
          x[k] = U + V;
          x[k + d] = U - V + q2;
        } else {
          u64 s = U + V;
          if (s >= q2) s -= q2;
          x[k] = s;
          x[k + d] = shoup_lazy(U - V + q2, w, wp, q);
        }
      }
    }
  }
}

template <bool FWD, int RING>
__device__ __forceinline__ void ntt_round_dispatch(int jlo, int jhi, u64 (&x)[8], int rbase, int logu, int logS, int mg,
                                                   const ulonglong2* tw, u64 q, bool pre1) {
  switch (jlo * 3 + jhi) {
    case 0: ntt_round<FWD, 0, 0, RING>(x, rbase, logu, logS, mg, tw, q, pre1); break;
    case 1: ntt_round<FWD, 0, 1, RING>(x, rbase, logu, logS, mg, tw, q, pre1); break;
    case 2: ntt_round<FWD, 0, 2, RING>(x, rbase, logu, logS, mg, tw, q, pre1); break;
    case 4: ntt_round<FWD, 1, 1, RING>(x, rbase, logu, logS, mg, tw, q, pre1); break;
    case 5: ntt_round<FWD, 1, 2, RING>(x, rbase, logu, logS, mg, tw, q, pre1); break;
    default: ntt_round<FWD, 2, 2, RING>(x, rbase, logu, logS, mg, tw, q, pre1); break;
  }
}

// One phase: the tile is CPB sub-transforms of S = 2^logS words (columns of
// stride N/S when COLS, else contiguous chunks), staged in shared memory.
// blockDim = CPB*S/8. Residues stay lazy ([0,4q) forward, [0,2q) inverse)
// except in the LAST phase, which writes canonical values (times N^-1 for
// the inverse).
template <bool FWD, bool COLS, bool LAST, int RING = 1>
__global__ void __launch_bounds__(512) k_ntt(NttArgs A, int logS, int logCPB, int m0) {
  extern __shared__ u64 sm[];
  u64* ptr;
  int pidx;
  if (!poly_of(A, blockIdx.y, ptr, pidx)) return;
  const u64 q = A.mods[pidx].q;
  const ulonglong2* tw = reinterpret_cast<const ulonglong2*>(A.tw + (size_t)pidx * 4 * A.N + (FWD ? 0 : 2 * A.N));
  const int S = 1 << logS, CPB = 1 << logCPB, W = S << logCPB;
  const int tid = threadIdx.x, T = blockDim.x;
  const int tile = blockIdx.x;
  const long colbase = (long)tile * CPB;
  const int stride = A.N >> logS;
  // global -> shared, coalesced: consecutive lin are consecutive addresses
  for (int lin = tid; lin < W; lin += T) {
    long g = COLS ? (long)(lin >> logCPB) * stride + colbase + (lin & (CPB - 1)) : (long)tile * W + lin;
    sm[swz(lin)] = ptr[g];
  }
  __syncthreads();
  // m = 5N/2 (one phase over CPB = 4 chunks, the four factors): the split
  // first, residues brought below 2q for the rounds
  const ulonglong2* spl =
      RING == 5 ? reinterpret_cast<const ulonglong2*>(A.split + (size_t)pidx * kSplitWords) : nullptr;
  if (RING == 5 && FWD) {
    const int n4 = W >> 2;
    for (int i = tid; i < n4; i += T) {
      u64 a0 = sm[swz(i)], a1 = sm[swz(i + n4)], a2 = sm[swz(i + 2 * n4)], a3 = sm[swz(i + 3 * n4)];
      split4_fwd(a0, a1, a2, a3, spl, q);
      u64* o4[4] = {&a0, &a1, &a2, &a3};
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        u64 v = *o4[h];  // below 16q
        if (v >= 8 * q) v -= 8 * q;
        if (v >= 4 * q) v -= 4 * q;
        if (v >= 2 * q) v -= 2 * q;
        sm[swz(i + h * n4)] = v;
      }
    }
    __syncthreads();
  }
  const int rounds = (logS + 2) / 3;
  for (int rho = 0; rho < rounds; ++rho) {
    // log2 of the smallest (a) and largest (b) half-distance of this round
    const int ns = min(3, logS - 3 * rho);
    const int b = FWD ? logS - 1 - 3 * rho : 3 * rho + ns - 1;
    const int a = b - ns + 1;
    const int logu = max(0, b - 2);
    int c, o, B;
    if (COLS) {
      c = tid & (CPB - 1);
      int rest = tid >> logCPB;
      o = rest & ((1 << logu) - 1);
      B = rest >> logu;
    } else {
      o = tid & ((1 << logu) - 1);
      int rest = tid >> logu;
      int logB = logS - 3 - logu;
      B = rest & ((1 << logB) - 1);
      c = rest >> logB;
    }
    const int rbase = (B << (logu + 3)) + o;
    const int mg = m0 + (COLS ? 0 : tile * CPB + c);
    u64 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      int r = rbase + (k << logu);
      x[k] = sm[swz(COLS ? (r << logCPB) + c : (c << logS) + r)];
    }
    ntt_round_dispatch<FWD, RING>(a - logu, b - logu, x, rbase, logu, logS, mg, tw, q, RING == 1 && A.pre_w1);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      int r = rbase + (k << logu);
      sm[swz(COLS ? (r << logCPB) + c : (c << logS) + r)] = x[k];
    }
    __syncthreads();
  }
  if (RING == 5 && !FWD) {  // the split last, with the 4/N scaling: canonical
    const int n4 = W >> 2;
    for (int i = tid; i < n4; i += T) {
      u64 b0 = sm[swz(i)], b1 = sm[swz(i + n4)], b2 = sm[swz(i + 2 * n4)], b3 = sm[swz(i + 3 * n4)];
      split4_inv(b0, b1, b2, b3, spl, q, 2 * q);
      sm[swz(i)] = b0;
      sm[swz(i + n4)] = b1;
      sm[swz(i + 2 * n4)] = b2;
      sm[swz(i + 3 * n4)] = b3;
    }
    __syncthreads();
  }
  u64 ni = 0, nip = 0;
  if (LAST && !FWD) { ni = A.ninv[6 * pidx]; nip = A.ninv[6 * pidx + 1]; }
  for (int lin = tid; lin < W; lin += T) {
    u64 v = sm[swz(lin)];
    if (LAST) {
      if (FWD) {
        if (v >= 2 * q) v -= 2 * q;
        if (v >= q) v -= q;
      } else if (RING != 5) {
        v = shoup(v, ni, nip, q);
      }
    }
    long g = COLS ? (long)(lin >> logCPB) * stride + colbase + (lin & (CPB - 1)) : (long)tile * W + lin;
    ptr[g] = v;
  }
}

// ---------------------------------------------------------------- radix-16 phases
// Same scheme with sixteen words per thread (four stages per register round,
// two rounds per 256-point phase) for the two-phase transforms (N >= 8192).
// Round 0 reads global memory straight into registers and the last round
// writes straight back whenever that access is coalesced (always for column
// tiles; for chunk tiles when the round's spacing u >= 16), otherwise the
// tile passes through shared memory once more.
// blockDim = CPB*S/16, S = 2^LOGS with 5 <= LOGS <= 8. Every round's stage
// range is a compile-time constant, so the sixteen words stay in registers.
// The forward butterfly here never reduces its upper input: each stage adds
// less than 2q to the bound, so inputs below 4q leave a log2 N <= 16 stage
// transform below 36q (40q with the m = 3N split, 44q with m = 5N/2's) < 64q < 2^64 (primes below
// 2^58), and the last phase brings every word back to [0, q) once (reduce_lazy).
// One CTA tile (`tile` of polynomial `poly`) of one phase; the body of the
// per-transform kernel k_ntt16 and of the persistent kernel k_ntt16_multi.
// R3 (m = 3N, column phases only): the first forward stage and the last
// inverse stage are node 1, the split of X^N - X^(N/2) + 1 (see ntt_round).
// Forward it adds up to 6q to the bound, so the transform stays below 40q.
// Inverse it is fused with N^-1: with c = (2 rho - 1)^-1 N^-1 (inverse
// twiddle word 0), high = (U - V) 2c, low = (U + V) N^-1 - (U - V) c.
template <bool FWD, bool COLS, bool LAST, int LOGS, bool SRC, int RING = 1>
__device__ __forceinline__ void ntt16_tile(const NttArgs& A, int logCPB, int m0, int tile, int poly) {
  extern __shared__ u64 sm[];
  u64* ptr;
  int pidx;
  if (!poly_of(A, poly, ptr, pidx)) return;
  const u64 q = A.mods[pidx].q;
  const ulonglong2* tw = reinterpret_cast<const ulonglong2*>(A.tw + (size_t)pidx * 4 * A.N + (FWD ? 0 : 2 * A.N));
  constexpr int S = 1 << LOGS;
  const int CPB = 1 << logCPB, W = S << logCPB;
  const int tid = threadIdx.x, T = blockDim.x;
  const int stride = A.N >> LOGS;
  u64* gbase = COLS ? ptr + (long)tile * CPB : ptr + (long)tile * W;
  const u64* gsrc = gbase;
  if (SRC) {  // same polynomial, read from the out-of-place source
    const int i = poly / A.n_outer, o = poly % A.n_outer;
    const u64* rb = A.src + (long)o * A.src_os + (long)i * A.N;
    gsrc = COLS ? rb + (long)tile * CPB : rb + (long)tile * W;
  }
  constexpr int NR = (LOGS + 3) / 4;
  constexpr int B0 = FWD ? LOGS - 1 : (LOGS < 4 ? LOGS : 4) - 1;
  constexpr int NSL = LOGS - 4 * (NR - 1);
  constexpr int BL = FWD ? LOGS - 1 - 4 * (NR - 1) : 4 * (NR - 1) + NSL - 1;
  constexpr bool DIN = COLS || (B0 - 3 >= 4);
  constexpr bool DOUT = COLS || (BL - 3 >= 4);
  // Inverse chunk phase (staged through shared memory): the first stage's
  // eight twiddles of this thread are consecutive; load them before the
  // staging so their latency overlaps it.
  constexpr bool PRE = SS_NTT_PREFETCH && !FWD && !DIN && !COLS;
  ulonglong2 pre[PRE ? 8 : 1];
  if (PRE) {
    const int logB = LOGS - 4;
    const int B = tid & ((1 << logB) - 1), c = tid >> logB;
    const int mg = m0 + tile * CPB + c;
    const ulonglong2* tp = tw + (mg << (LOGS - 1)) + (B << 3);
#pragma unroll
    for (int i = 0; i < (PRE ? 8 : 1); ++i) pre[i] = __ldg(tp + i);
  }
  if (!DIN) {
    for (int lin = tid; lin < W; lin += T) sm[swz16<COLS>(lin)] = gsrc[lin];
    __syncthreads();
  }
  u64 ni = 0, nip = 0;
  u64 wni = 0, wnip = 0;
  u64 cni = 0, cnip = 0;
  if (LAST && !FWD) {
    const u64* nv = A.ninv + 6 * pidx;
    ni = nv[0];
    nip = nv[1];
    wni = nv[2];
    wnip = nv[3];
    if (RING == 3) {
      cni = nv[4];
      cnip = nv[5];
    }
  }
  const int kb = A.mods[pidx].kbits;
  const uint32_t mq = (uint32_t)(A.mods[pidx].mu >> 47);
#pragma unroll
  for (int rho = 0; rho < NR; ++rho) {
    const int ns = (LOGS - 4 * rho) < 4 ? (LOGS - 4 * rho) : 4;
    const int b = FWD ? LOGS - 1 - 4 * rho : 4 * rho + ns - 1;
    const int a = b - ns + 1;
    const int logu = b - 3 > 0 ? b - 3 : 0;
    int c, o, B;
    if (COLS) {
      c = tid & (CPB - 1);
      int rest = tid >> logCPB;
      o = rest & ((1 << logu) - 1);
      B = rest >> logu;
    } else {
      o = tid & ((1 << logu) - 1);
      int rest = tid >> logu;
      const int logB = LOGS - 4 - logu;
      B = rest & ((1 << logB) - 1);
      c = rest >> logB;
    }
    const int rbase = (B << (logu + 4)) + o;
    const int mg = m0 + (COLS ? 0 : tile * CPB + c);
    u64 x[16];
    if (rho == 0 && DIN) {
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        int r = rbase + (k << logu);
        x[k] = COLS ? gsrc[(long)r * stride + c] : gsrc[(c << LOGS) + r];
      }
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        int r = rbase + (k << logu);
        x[k] = sm[swz16<COLS>(COLS ? (r << logCPB) + c : (c << LOGS) + r)];
      }
    }
    // stages j in [a - logu, b - logu]: d = 2^j registers apart
    const u64 q2 = 2 * q;
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int jlo = a - logu, jhi = b - logu;
      const int j = FWD ? jhi - jj : jlo + jj;
      if (jj < ns) {
        const int d = 1 << j;
        const int logt = logu + j;
        const int sg = LOGS - 1 - logt;
        // the inverse transform's last stage (one twiddle, psi^(-N/2)) also
        // applies N^-1: sums times N^-1, differences times N^-1 psi^(-N/2)
        const bool fold = LAST && !FWD && rho == NR - 1 && jj == ns - 1;
        const bool split = RING == 3 && COLS && FWD && rho == 0 && jj == 0;
        // node 1 of X^N + 1 (the column phase's first forward stage) on inputs
        // whose upper half already carries its twiddle: no product
        const bool pre1 = RING == 1 && COLS && FWD && rho == 0 && jj == 0 && A.pre_w1;
        // m = 5N/2: the first two forward stages and the last two inverse
        // stages of the column phase are the four-way split on the registers
        // k, k+4, k+8, k+12 (the quarters), k < 4
        if (RING == 5 && COLS && FWD && rho == 0 && jj < 2) {
          if (jj == 0) {
            const ulonglong2* spl = reinterpret_cast<const ulonglong2*>(A.split + (size_t)pidx * kSplitWords);
#pragma unroll
            for (int k = 0; k < 4; ++k) split4_fwd(x[k], x[k + 4], x[k + 8], x[k + 12], spl, q);
          }
          continue;
        }
        if (RING == 5 && COLS && LAST && !FWD && rho == NR - 1 && jj >= ns - 2) {
          if (jj == ns - 1) {
            const ulonglong2* spl = reinterpret_cast<const ulonglong2*>(A.split + (size_t)pidx * kSplitWords);
#pragma unroll
            for (int k = 0; k < 4; ++k) split4_inv(x[k], x[k + 4], x[k + 8], x[k + 12], spl, q, q2);
          }
          continue;
        }
#pragma unroll
        for (int blk = 0; blk < 8; ++blk) {
          if (blk < 8 / d) {
            const int k0 = blk * 2 * d;
            u64 w = wni, wp = wnip;
            if (PRE && rho == 0 && jj == 0) {
              w = pre[PRE ? blk : 0].x;
              wp = pre[PRE ? blk : 0].y;
            } else if (!fold && !pre1) {
              const int widx = (mg << sg) + ((rbase + (k0 << logu)) >> (logt + 1));
              const ulonglong2 wv = __ldg(tw + widx);
              w = wv.x;
              wp = wv.y;
            }
#pragma unroll
            for (int p = 0; p < 8; ++p) {
              if (p < d) {
                const int k = k0 + p;
                u64 U = x[k], V = x[k + d];
                if (fold && RING == 3) {
                  const u64 dv = U - V + q2;
                  const u64 lo = shoup(U + V, ni, nip, q), cr = shoup(dv, cni, cnip, q);
                  x[k] = lo >= cr ? lo - cr : lo + q - cr;
                  x[k + d] = shoup(dv, w, wp, q);
                } else if (fold && A.post_scale) {  // N^-1 and N^-1 psi^(-N/2) left to the consumer
                  x[k] = U + V;
                  x[k + d] = U - V + q2;
                } else if (fold) {
                  x[k] = shoup(U + V, ni, nip, q);
                  x[k + d] = shoup(U - V + q2, w, wp, q);
                } else if (split) {
                  const u64 t = shoup_lazy(V, w, wp, q);
                  x[k] = U + t;
                  x[k + d] = U + V + q2 - t;
                } else if (pre1) {  // U, V < 2q, as a base conversion leaves them
                  x[k] = U + V;
                  x[k + d] = U - V + q2;
                } else if (FWD) {
                  V = shoup_lazy(V, w, wp, q);
                  x[k] = U + V;
                  x[k + d] = U - V + q2;
                } else {
                  u64 s2 = U + V;
                  if (s2 >= q2) s2 -= q2;
                  x[k] = s2;
                  x[k + d] = shoup_lazy(U - V + q2, w, wp, q);
                }
              }
            }
          }
        }
      }
    }
    if (rho == NR - 1 && DOUT) {
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        int r = rbase + (k << logu);
        u64 v = x[k];
        if (LAST && FWD) v = reduce_lazy(v, q, kb, mq);  // the inverse's last stage already reduced and scaled
        if (COLS) gbase[(long)r * stride + c] = v;
        else gbase[(c << LOGS) + r] = v;
      }
    } else {
      if (rho > 0 || !DIN) __syncthreads();  // every read of the previous layout is done
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        int r = rbase + (k << logu);
        sm[swz16<COLS>(COLS ? (r << logCPB) + c : (c << LOGS) + r)] = x[k];
      }
      __syncthreads();
    }
  }
  if (!DOUT) {
    for (int lin = tid; lin < W; lin += T) {
      u64 v = sm[swz16<COLS>(lin)];
      if (LAST && FWD) v = reduce_lazy(v, q, kb, mq);
      gbase[lin] = v;
    }
  }
}

template <bool FWD, bool COLS, bool LAST, int LOGS, bool SRC, int RING>
__global__ void __launch_bounds__(256, RING == 5 ? SS_NTT_MINB_R5 : (FWD ? SS_NTT_MINB_F : SS_NTT_MINB_I))
    k_ntt16(NttArgs A, int logCPB, int m0) {
  ntt16_tile<FWD, COLS, LAST, LOGS, SRC, RING>(A, logCPB, m0, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------- products by halves
// Transforms of N >= 8192 on primes below 2^55 (nine spare bits in a word). With
// a = h 2^32 + l, w_0 = w and w_1 = 2^32 w mod q, a w = l w_0 + h w_1 (mod q), a
// sum below 2^33 q, so its quotient by 2q is one 32-bit word and the product
// costs 26 cycles of the multiply pipe per warp (five 64-bit products at four,
// three 32-bit ones at two) where the 64-bit Shoup product costs 32, with fewer
// adds (half_mul; register-only loops, ncu pipe counters: forward butterflies
// 30.2 cycles a warp against 40.8, inverse ones 30.1 against 49, which also
// reduce every sum). A twiddle is 24 bytes (w_0, w_1, p_0, p_1).
// Bounds. Forward: the first stage lifts its upper inputs by 128q and every
// stage then subtracts products (below 6q, at most 16 stages) without an offset:
// words stay below 4q + 128q + 96q. Inverse: a round starts below 32q, sums
// double per stage (below 512q < 2^64) and differences are lifted by 32q 2^j;
// at a round's end only the words that are sums of all its stages, or of the
// last three, exceed 32q and are reduced.
// One stage of half-distance step * 2^j on sixteen words of spacing `step`;
// slot(j, blk) is the shared-memory slot of the twiddle of block blk.
template <bool FWD, class Slot>
__device__ __forceinline__ void half_stage(u64 (&x)[16], int j, int jj, const ulonglong2* tw, const uint2* tp,
                                           const HalfMod& m, bool lift, Slot slot) {
  const int d = 1 << j;
#pragma unroll
  for (int blk = 0; blk < 8; ++blk) {
    if (blk < 8 / d) {
      const int at = slot(j, blk);
      const ulonglong2 w = tw[at];
      const uint2 p = tp[at];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (i < d) {
          const int k = blk * 2 * d + i;
          u64 U = x[k];
          const u64 V = x[k + d];
          if (FWD) {
            if (lift) U += m.q << 7;
            const u64 t = half_mul(V, w.x, w.y, p.x, p.y, m.nq2);
            x[k] = U + t;
            x[k + d] = U - t;
          } else {
            x[k] = U + V;
            x[k + d] = half_mul(U - V + (m.q << (5 + jj)), w.x, w.y, p.x, p.y, m.nq2);
          }
        }
      }
    }
  }
}
// end of an inverse round of `ns` stages: back below 32q
__device__ __forceinline__ void half_settle(u64 (&x)[16], int ns, const HalfMod& m) {
#pragma unroll
  for (int k = 0; k < 16; ++k)
    if (k < (1 << (4 - ns)) || (ns == 4 && k == 1)) x[k] = reduce_half(x[k], m);
}

// Column phase: a tile is CPB = 2^CL columns (stride 2^LOG2N words) of S = 2^LOGS
// rows of one polynomial; S CPB / 16 threads. Every address in shared and global
// memory is a per-thread base plus a constant, and the phase's S twiddles are in
// shared memory (6 KiB at most; copied while the words load): with runtime tile
// shapes and twiddles from global memory the phase spent 22.4 instructions a
// warp and butterfly where the butterfly itself takes 13.
// The transform's top is node 1: of X^N + 1 (pre_w1, post_scale: PolySet), the
// m = 3N split (RING 3) or, with its children, the m = 5N/2 split (RING 5).
template <int CL>
__device__ __forceinline__ int col_swz(int lin) {
  // eight columns: rows 16 apart would share banks; odd groups of 16 rows swap row pairs
  return CL == 3 ? lin ^ (((lin >> 7) & 1) << 3) : lin;
}

template <bool FWD, int LOGS, int LOG2N, int CL, int RING>
__device__ __forceinline__ void ntt16_cols(const NttArgs& A, int tile, int poly) {
  extern __shared__ u64 sm[];
  constexpr int S = 1 << LOGS, G = S / 16, W = LOGS < 8 ? LOGS - 4 : 4;
  constexpr long STRIDE = 1L << LOG2N;
  u64* ptr;
  int pidx;
  if (!poly_of(A, poly, ptr, pidx)) return;
  const int tid = threadIdx.x;
  ulonglong2* twS = reinterpret_cast<ulonglong2*>(sm);
  uint2* tpS = reinterpret_cast<uint2*>(twS + S);
  u64* data = reinterpret_cast<u64*>(tpS + S);
  {
    const ulonglong2* gw = half_tw<FWD>(A, pidx);
    const uint4* gp = reinterpret_cast<const uint4*>(half_tp<FWD>(A, pidx));
    constexpr int T = S << CL >> 4;
#pragma unroll
    for (int i = 0; i < S; i += T)
      if (T <= S || tid < S) cp16(twS + i + tid, gw + i + tid);
#pragma unroll
    for (int i = 0; i < S / 2; i += T)
      if (T <= S / 2 || tid < S / 2) cp16(reinterpret_cast<uint4*>(tpS) + i + tid, gp + i + tid);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  const int c = tid & ((1 << CL) - 1), rest = tid >> CL;
  u64* col = ptr + ((long)tile << CL) + c;
  const HalfMod hm = half_mod(A.mods[pidx]);
  const u64 q = hm.q;
  u64 x[16];
  // wide round: rows rest + G k; narrow round: rows 16 rest + k
#pragma unroll
  for (int k = 0; k < 16; ++k) x[k] = FWD ? col[(rest + (long)G * k) * STRIDE] : col[(16 * rest + (long)k) * STRIDE];
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  auto wide_slot = [](int j, int blk) { return tw_slot((1 << (3 - j)) + blk, LOGS - 4 + j, W); };
  auto narrow_slot = [rest](int j, int blk) { return (1 << (LOGS - 1 - j)) + (blk << W) + rest; };
  const ulonglong2* spl =
      RING == 5 ? reinterpret_cast<const ulonglong2*>(A.split + (size_t)pidx * kSplitWords) : nullptr;
  if constexpr (FWD) {
    int j0 = 3;
    if (RING == 5) {
#pragma unroll
      for (int k = 0; k < 4; ++k) split4_fwd(x[k], x[k + 4], x[k + 8], x[k + 12], spl, q);
      j0 = 1;
    } else if (RING == 3) {
      const ulonglong2 w = twS[1];
      const uint2 p = tpS[1];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const u64 U = x[k] + (q << 7), V = x[k + 8];
        const u64 t = half_mul(V, w.x, w.y, p.x, p.y, hm.nq2);
        x[k] = U + t;
        x[k + 8] = U + V - t;
      }
      j0 = 2;
    } else if (A.pre_w1) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const u64 U = x[k] + (q << 7), V = x[k + 8];  // V < 4q
        x[k] = U + V;
        x[k + 8] = U - V;
      }
      j0 = 2;
    }
#pragma unroll
    for (int j = 3; j >= 0; --j)
      if (j <= j0) half_stage<true>(x, j, 0, twS, tpS, hm, RING == 5 ? j == 1 : RING == 1 && j == 3, wide_slot);
#pragma unroll
    for (int k = 0; k < 16; ++k) data[col_swz<CL>(((rest + G * k) << CL) + c)] = x[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = data[col_swz<CL>(((16 * rest + k) << CL) + c)];
#pragma unroll
    for (int j = LOGS - 5; j >= 0; --j) half_stage<true>(x, j, 0, twS, tpS, hm, false, narrow_slot);
#pragma unroll
    for (int k = 0; k < 16; ++k) col[(16 * rest + (long)k) * STRIDE] = x[k];
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) half_stage<false>(x, j, j, twS, tpS, hm, false, narrow_slot);
    half_settle(x, 4, hm);
#pragma unroll
    for (int k = 0; k < 16; ++k) data[col_swz<CL>(((16 * rest + k) << CL) + c)] = x[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = data[col_swz<CL>(((rest + G * k) << CL) + c)];
    constexpr int NS = LOGS - 4;  // stages j = 4 - NS .. 3, the last one (or two) with N^-1
    constexpr int JE = RING == 5 ? 2 : 3;
    if constexpr (4 - NS < JE) {
#pragma unroll
      for (int j = 4 - NS; j < JE; ++j) half_stage<false>(x, j, j - (4 - NS), twS, tpS, hm, false, wide_slot);
    }
    const u64* nv = A.ninv + 6 * pidx;
    const u64 off = q << (5 + NS - 1);  // no input of the last stage is above it
    if (RING == 5) {  // the split takes two stages: its inputs are below off / 2 <= 128q
#pragma unroll
      for (int k = 0; k < 4; ++k) split4_inv(x[k], x[k + 4], x[k + 8], x[k + 12], spl, q, off);
    } else if (RING == 3) {
      const u64 ni = nv[0], nip = nv[1], w = nv[2], wp = nv[3], cn = nv[4], cnp = nv[5];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const u64 sv = x[k] + x[k + 8], dv = x[k] - x[k + 8] + off;
        const u64 lo = shoup(sv, ni, nip, q), cr = shoup(dv, cn, cnp, q);
        x[k] = lo >= cr ? lo - cr : lo + q - cr;
        x[k + 8] = shoup(dv, w, wp, q);
      }
    } else if (A.post_scale) {  // N^-1 and N^-1 psi^(-N/2) left to the consumer
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const u64 U = x[k], V = x[k + 8];
        x[k] = U + V;
        x[k + 8] = U - V + off;
      }
    } else {
      const u64 ni = nv[0], nip = nv[1], w = nv[2], wp = nv[3];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const u64 U = x[k], V = x[k + 8];
        x[k] = shoup(U + V, ni, nip, q);
        x[k + 8] = shoup(U - V + off, w, wp, q);
      }
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) col[(rest + (long)G * k) * STRIDE] = x[k];
  }
}

// log2 words of a column tile: small (128 threads) or large (256 threads, twice the
// columns: 128-byte rows at 2^8 words a column, half the twiddle copies). A
// multiplication at N = 2^16, level 41, of 1, 4 and 32 ciphertexts takes 666, 2411
// and 17491 us with the small tile and 652, 2337 and 17231 with the large one (a
// tile of 2^10 words: 702, 2562, 19986), so the large one runs wherever its
// tiles fill the GPU twice; below that the small one spreads the work wider.
constexpr int kColTile = 11, kColTileBig = 12;
template <int LOGS, int CL>
constexpr size_t col_smem() {
  return ((size_t)24 << LOGS) + ((size_t)8 << (LOGS + CL));
}

template <bool FWD, int LOGS, int LOG2N, int CL, int RING>
__global__ void __launch_bounds__(1 << (LOGS + CL - 4),
                                  LOGS + CL == kColTile ? (FWD ? SS_COLS_F : SS_COLS_I) : SS_COLS_BIG)
    k_ntt16_cols(NttArgs A) {
  enter_grid();
  ntt16_cols<FWD, LOGS, LOG2N, CL, RING>(A, blockIdx.x, blockIdx.y);
}

// Chunk phase: a row is one chunk (S = 2^LOGS words) of one polynomial; S / 16 threads (16 or
// 8, within one warp) hold it, sixteen words each, so its two register rounds
// exchange words through the warp's own shared memory with warp barriers only.
// A CTA takes the same chunks of several polynomials of one limb: NP = 2^lnp of
// them times NC = rows / NP chunks. Their twiddles, 24 bytes a node, are copied
// to shared memory once per CTA (cp.async, while the first words load), where
// one polynomial's chunks per CTA read each node from L2 once per polynomial
// with its latency exposed in every stage (forward chunk phase, 328 limbs of
// 2^16 words, products by halves: 129 us, the multiply pipe 60 % busy).
// Polynomials that the set skips (a ModUp digit's own limbs) are left out of the
// groups: the v-th polynomial of a limb is the v-th that is transformed.
// word r of a row: pairs of words stay adjacent (16-byte accesses); the pairs of
// a group of 16 are permuted by the group's index, so eight threads that each
// read a pair of their own group, and sixteen that read one word each of one
// group, touch all banks once
__device__ __forceinline__ int row_swz(int r) { return r ^ (((r >> 4) & 7) << 1); }

// a thread's share of its row, in linear order of pairs (words 16 lr .. 16 lr + 15)
__device__ __forceinline__ void row_put(const u64 (&x)[16], u64* mine, int lr) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
    *reinterpret_cast<ulonglong2*>(mine + row_swz(16 * lr + 2 * i)) = make_ulonglong2(x[2 * i], x[2 * i + 1]);
}
__device__ __forceinline__ void row_get(u64 (&x)[16], const u64* mine, int lr) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(mine + row_swz(16 * lr + 2 * i));
    x[2 * i] = t.x;
    x[2 * i + 1] = t.y;
  }
}
// Both register rounds of a forward row: x holds words lr + (S/16) k on entry and
// 16 lr + k, unreduced, on return. The whole warp calls it.
template <int LOGS>
__device__ __forceinline__ void row_forward(u64 (&x)[16], u64* mine, int lr, const ulonglong2* tw, const uint2* tp,
                                            const HalfMod& hm) {
  constexpr int TPR = (1 << LOGS) / 16;
  auto wide_slot = [](int j, int blk) { return (1 << (3 - j)) + blk; };
  auto narrow_slot = [lr](int j, int blk) { return (1 << (LOGS - 1 - j)) + (blk << (LOGS - 4)) + lr; };
#pragma unroll
  for (int j = 3; j >= 0; --j) half_stage<true>(x, j, 0, tw, tp, hm, false, wide_slot);
#pragma unroll
  for (int k = 0; k < 16; ++k) mine[row_swz(lr + TPR * k)] = x[k];
  __syncwarp();
  row_get(x, mine, lr);
#pragma unroll
  for (int j = LOGS - 5; j >= 0; --j) half_stage<true>(x, j, 0, tw, tp, hm, false, narrow_slot);
}

struct RowPlan {
  int lnp, groups;  // log2 NP, groups of NP polynomials per limb (at most)
};

template <bool FWD, int LOGS, bool SRC>
__device__ __forceinline__ void ntt16_rows(const NttArgs& A, const RowPlan& R, int item, int limb) {
  extern __shared__ u64 sm[];
  constexpr int S = 1 << LOGS, TPR = S / 16, LT = LOGS - 4;
  const int tid = threadIdx.x, lane = tid & 31;
  const int lnc = (31 - __clz(blockDim.x)) - LT - R.lnp;  // log2 NC
  const int group = item % R.groups, cg = item / R.groups;
  // the limb's polynomials: all, or those whose digit is not the limb's own
  const bool own = A.skip_w > 0 && limb < A.nq && limb < A.skip_level;
  const int per = own ? A.skip_mod - 1 : A.n_outer;
  const int nv = own ? (A.n_outer / A.skip_mod) * per : A.n_outer;
  const int v0 = group << R.lnp;
  if (v0 >= nv) return;
  const int pidx = limb < A.nq ? A.q0 + limb : A.L + (limb - A.nq);
  const int n1 = A.N >> LOGS;
  // twiddles of the CTA's chunks
  ulonglong2* twS = reinterpret_cast<ulonglong2*>(sm);
  uint2* tpS = reinterpret_cast<uint2*>(twS + (S << lnc));
  u64* data = reinterpret_cast<u64*>(tpS + (S << lnc)) + (size_t)(tid >> 5) * 512;
  {
    const size_t at = (size_t)n1 + ((size_t)cg << (lnc + LOGS));
    const ulonglong2* gw = half_tw<FWD>(A, pidx) + at;
    const uint4* gp = reinterpret_cast<const uint4*>(half_tp<FWD>(A, pidx) + at);
    for (int i = tid; i < (S << lnc); i += blockDim.x) cp16(twS + i, gw + i);
    for (int i = tid; i < (S << lnc) / 2; i += blockDim.x) cp16(reinterpret_cast<uint4*>(tpS) + i, gp + i);
  }
  const int row = tid >> LT, lr = tid & (TPR - 1);
  const int v = v0 + (row & ((1 << R.lnp) - 1));
  const int chl = row >> R.lnp;
  const bool valid = v < nv;
  long off = 0, soff = 0;
  if (valid) {
    int o = v;
    if (own) {
      const int b = v / per, jj = v - b * per;
      o = b * A.skip_mod + jj + (jj >= limb / A.skip_w ? 1 : 0);
    }
    const long in_poly = (long)limb * A.N + ((long)((cg << lnc) + chl) << LOGS);
    off = (long)o * A.outer_stride + in_poly;
    soff = SRC ? (long)o * A.src_os + in_poly : off;
  }
  const u64* src = (SRC ? A.src : A.base) + soff;
  u64* dst = A.base + off;
  const HalfMod hm = half_mod(A.mods[pidx]);
  const u64 q = hm.q;
  u64* mine = data + (lane >> LT) * S;  // this thread's row in the warp's shared memory
  u64 x[16];
  // this warp's rows in linear order: lane l moves the pairs l, l + 32, ... of each
  constexpr int RPW = 32 / TPR;  // rows per warp
  if (FWD) {
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = valid ? src[lr + TPR * k] : 0;
  } else {
#pragma unroll
    for (int rw = 0; rw < RPW; ++rw) {
      const u64* rp = reinterpret_cast<const u64*>(__shfl_sync(0xffffffffu, (unsigned long long)src, rw * TPR));
      const bool ok = __shfl_sync(0xffffffffu, valid ? 1 : 0, rw * TPR) != 0;
#pragma unroll
      for (int i = 0; i < S / 64; ++i) {
        const int r = 2 * (lane + 32 * i);
        if (ok) cp16(data + rw * S + row_swz(r), rp + r);
      }
    }
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  if (!__any_sync(0xffffffffu, valid)) return;
  const ulonglong2* tw = twS + chl * S;
  const uint2* tp = tpS + chl * S;
  // the narrow round holds words 16 lr .. 16 lr + 15, the wide round words lr + TPR k
  auto wide_slot = [](int j, int blk) { return (1 << (3 - j)) + blk; };
  auto narrow_slot = [lr](int j, int blk) { return (1 << (LOGS - 1 - j)) + (blk << LT) + lr; };
  if (FWD) {
    row_forward<LOGS>(x, mine, lr, tw, tp, hm);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const u64 r = reduce_half(x[k], hm), d = r - q;  // d wraps above r when r < q
      x[k] = r < d ? r : d;
    }
    row_put(x, mine, lr);
    __syncwarp();
#pragma unroll
    for (int rw = 0; rw < RPW; ++rw) {
      u64* rp = reinterpret_cast<u64*>(__shfl_sync(0xffffffffu, (unsigned long long)dst, rw * TPR));
      const bool ok = __shfl_sync(0xffffffffu, valid ? 1 : 0, rw * TPR) != 0;
#pragma unroll
      for (int i = 0; i < S / 64; ++i) {
        const int r = 2 * (lane + 32 * i);
        if (ok)
          *reinterpret_cast<ulonglong2*>(rp + r) = *reinterpret_cast<const ulonglong2*>(data + rw * S + row_swz(r));
      }
    }
  } else {
    row_get(x, mine, lr);
#pragma unroll
    for (int j = 0; j < 4; ++j) half_stage<false>(x, j, j, tw, tp, hm, false, narrow_slot);
    half_settle(x, 4, hm);
    row_put(x, mine, lr);
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = mine[row_swz(lr + TPR * k)];
    constexpr int NS = LOGS - 4;  // stages of the wide round: half-distances 16 .. S/2
#pragma unroll
    for (int j = 4 - NS; j < 4; ++j) half_stage<false>(x, j, j - (4 - NS), tw, tp, hm, false, wide_slot);
    half_settle(x, NS, hm);
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (valid) dst[lr + TPR * k] = x[k];
  }
}

template <bool FWD, int LOGS, bool SRC>
__global__ void __launch_bounds__(128, FWD ? SS_ROWS_F : SS_ROWS_I) k_ntt16_rows(NttArgs A, RowPlan R) {
  enter_grid();
  ntt16_rows<FWD, LOGS, SRC>(A, R, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------- chunk phase with the key-switch inner product
// The last forward phase of a key switch's digits fused with their inner product
// with the key: a CTA holds one chunk of one limb for all digits of NB
// ciphertexts (rows as in ntt16_rows, the digit whose primes hold the limb read
// as it is), transforms the rows in shared memory and sums key times digit per
// word, so the transformed digits never reach memory. For the data limbs the two
// rows of the ModDown correction (its column phase done) are transformed beside
// them and the epilogue follows (k_ks_ip's types; acc_c the reduced sum):
//   type 0: acc_c[m] for the limbs the ModDown drops; with x, limb level - 1 also
//           takes P x_c;
//   type 1: out_c = (acc_c - delta_c) P^-1 (+ x_c; component 1 only if add_c1);
//   type 2: out_c = ((P x_c + acc_c) - delta_c) (q_{l-1} P)^-1.
// The separate inner product read 14 transformed limbs per limb and ciphertext
// from memory beside transforms bound by the multiply pipe; here its products (32
// pipe cycles a digit word against 112 for the phase) and the transforms share a
// kernel and the digits' write and read are gone. Each CTA reads its dn x 2 key
// rows (prefetched to L2 on entry) for NB ciphertexts; ciphertexts run fastest
// over the grid, so a chunk's key comes from DRAM once. Compiled for four CTAs of
// 256 threads per SM (64 registers): with three (80) the sums' loads were exposed
// and a multiplication at N = 2^16, level 41, took 2504 us for 4 ciphertexts
// against 2435. Query of two ciphertexts a column at N = 2^16 141.9 -> 138.3 ms,
// comparison at N = 2^15 51.6 -> 50.6, 32 ciphertexts' multiplication 18.26 -> 17.73.
constexpr int kRowsIpMax = 16;  // rows of a CTA: 256 threads at 2^8 words a row
struct RowsIp {
  const Modulus* mods;
  NttArgs tab;  // tables
  const u64 *ext, *d, *kb, *ka;
  long ext_os, d_os;
  int level, alpha, L, T, N, dn, B, m0;
  int nb, bgroups;  // ciphertexts per CTA, groups of them
  u64* acc;
  long acc_os;
  int acc_nl;
  const u64* x;
  long x_os;
  int x_cap, add_c1;
  const u64* delta;
  int nl;
  const u64 *pm, *scale;
  u64* out;
  long out_os;
  int out_cap;
};

// 128-bit sum of products of words below 2^56 and 2^55, at most 16 of them: the low
// products with their carries, the middle (below 2^62) and the high ones apart
struct MacSum {
  u32 l0 = 0, l1 = 0, c = 0, m0 = 0, m1 = 0, h0 = 0, h1 = 0;
  __device__ __forceinline__ void add(u64 x, u64 y) {
    const u32 xl = (u32)x, xh = (u32)(x >> 32), yl = (u32)y, yh = (u32)(y >> 32);
    asm("mad.lo.cc.u32 %0, %7, %9, %0;\n\tmadc.hi.cc.u32 %1, %7, %9, %1;\n\taddc.u32 %2, %2, 0;\n\t"
        "mad.lo.cc.u32 %3, %7, %10, %3;\n\tmadc.hi.u32 %4, %7, %10, %4;\n\t"
        "mad.lo.cc.u32 %3, %8, %9, %3;\n\tmadc.hi.u32 %4, %8, %9, %4;\n\t"
        "mad.lo.cc.u32 %5, %8, %10, %5;\n\tmadc.hi.u32 %6, %8, %10, %6;"
        : "+r"(l0), "+r"(l1), "+r"(c), "+r"(m0), "+r"(m1), "+r"(h0), "+r"(h1)
        : "r"(xl), "r"(xh), "r"(yl), "r"(yh));
  }
  __device__ __forceinline__ u64 reduced(u64 q, u64 qinv) const {
    const u64 l = ((u64)l1 << 32) | l0, m = ((u64)m1 << 32) | m0, h = ((u64)h1 << 32) | h0;
    const u64 lo = l + (m << 32);
    const u64 hi = h + (m >> 32) + c + (lo < l ? 1 : 0);
    return redc128(hi, lo, q, qinv);
  }
};

template <int LOGS, int TYPE>
__global__ void __launch_bounds__(256, SS_ROWS_IP) k_rows_ip(const __grid_constant__ RowsIp A) {
  extern __shared__ u64 sm[];
  constexpr int S = 1 << LOGS, TPR = S / 16;
  enter_grid();
  const int tid = threadIdx.x;
  const int bg = blockIdx.x % A.bgroups, chunk = blockIdx.x / A.bgroups;
  const int m = A.m0 + blockIdx.y, g = m < A.level ? m : A.L + (m - A.level);
  const int own = m < A.level ? m / A.alpha : A.dn;  // the digit that is not transformed (none: dn)
  const int nd = A.dn - (own < A.dn ? 1 : 0), rpc = nd + (TYPE ? 2 : 0);
  const int b0 = bg * A.nb, nb = min(A.nb, A.B - b0);
  ulonglong2* twS = reinterpret_cast<ulonglong2*>(sm);
  uint2* tpS = reinterpret_cast<uint2*>(twS + S);
  u64* data = reinterpret_cast<u64*>(tpS + S);
  const int n1 = A.N >> LOGS;
  const long pos = ((long)chunk << LOGS), limb = (long)m * A.N + pos, key = (long)g * A.N + pos;
  {
    const size_t at = (size_t)n1 + ((size_t)chunk << LOGS);
    const ulonglong2* gw = half_tw<true>(A.tab, g) + at;
    const uint4* gp = reinterpret_cast<const uint4*>(half_tp<true>(A.tab, g) + at);
    for (int i = tid; i < S; i += blockDim.x) cp16(twS + i, gw + i);
    for (int i = tid; i < S / 2; i += blockDim.x) cp16(reinterpret_cast<uint4*>(tpS) + i, gp + i);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  const int row = tid / TPR, lr = tid % TPR;
  const bool valid = row < nb * rpc;
  const HalfMod hm = half_mod(A.mods[g]);
  u64 x[16];
  if (valid) {
    const int b = row / rpc, r = row - b * rpc;
    const long digit = r + (r >= own ? 1 : 0);
    const u64* src = r < nd ? A.ext + (long)(b0 + b) * A.ext_os + digit * (A.level + A.alpha) * A.N
                            : A.delta + ((long)(b0 + b) * 2 + (r - nd)) * A.nl * A.N;
    src += limb + lr;
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = src[TPR * k];
  } else {
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = 0;
  }
  for (int i = tid; i < A.dn * (S / 8); i += blockDim.x) {  // a line of each 128 bytes of the key rows
    const int j = i / (S / 8), w = i - j * (S / 8);
    const u64* p = (w < S / 16 ? A.kb : A.ka) + (size_t)j * A.T * A.N + key + (w % (S / 16)) * 16;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  u64* mine = data + (size_t)row * S;
  if (__any_sync(0xffffffffu, valid)) {
    row_forward<LOGS>(x, mine, lr, twS, tpS, hm);
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = reduce_half(x[k], hm);  // below 2q
    row_put(x, mine, lr);
  }
  __syncthreads();
  const u64 q = hm.q, qinv = A.mods[g].qinv;
  const size_t kstride = (size_t)A.T * A.N;
  for (int p = tid; p < nb << LOGS; p += blockDim.x) {
    const int b = p >> LOGS, n = p & (S - 1);
    const long o = b0 + b;
    const u64* kbp = A.kb + key + n;
    const u64* kap = A.ka + key + n;
    const u64* rows = data + b * rpc * S + row_swz(n);
    MacSum s0, s1;
    auto digits = [&](int r0, int r1) {
#pragma unroll 4
      for (int r = r0; r < r1; ++r) {
        const u64 v = *rows, kv = *kbp, av = *kap;
        s0.add(v, kv);
        s1.add(v, av);
        rows += S;
        kbp += kstride;
        kap += kstride;
      }
    };
    digits(0, min(own, nd));
    if (own < A.dn) {
      const u64 v = A.d[o * A.d_os + limb + n], kv = *kbp, av = *kap;
      s0.add(v, kv);
      s1.add(v, av);
      kbp += kstride;
      kap += kstride;
      digits(own, nd);
    }
    u64 a[2] = {s0.reduced(q, qinv), s1.reduced(q, qinv)};
    if (TYPE == 0) {
      if (A.x != nullptr && m == A.level - 1) {
        const u64 pw = __ldg(A.pm + 2 * m), pwp = __ldg(A.pm + 2 * m + 1);
#pragma unroll
        for (int c = 0; c < 2; ++c)
          a[c] = add_mod(a[c], shoup(A.x[o * A.x_os + (long)c * A.x_cap * A.N + limb + n], pw, pwp, q), q);
      }
      u64* out = A.acc + o * A.acc_os + (long)(m - A.m0) * A.N + pos + n;
      out[0] = a[0];
      out[(long)A.acc_nl * A.N] = a[1];
    } else {
      const u64 sc = __ldg(A.scale + 2 * m), scp = __ldg(A.scale + 2 * m + 1);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const u64 dl = rows[c * S];  // the rows after the digits', below 2q
        const bool has_x = A.x != nullptr && (TYPE == 2 || c == 0 || A.add_c1);
        const u64 xv = has_x ? A.x[o * A.x_os + (long)c * A.x_cap * A.N + limb + n] : 0;
        u64 r;
        if (TYPE == 2) {
          const u64 px = shoup(xv, __ldg(A.pm + 2 * m), __ldg(A.pm + 2 * m + 1), q);
          r = shoup(px + a[c] + 2 * q - dl, sc, scp, q);
        } else {
          r = shoup(a[c] + 2 * q - dl, sc, scp, q);
          if (has_x) r = add_mod(r, xv, q);
        }
        A.out[o * A.out_os + (long)c * A.out_cap * A.N + limb + n] = r;
      }
    }
  }
}

// ---------------------------------------------------------------- persistent multi-transform phase
// One phase of up to kMaxNttJobs transforms of any ring dimensions N >= 8192
// (each job: one polynomial set of one context, with its own moduli and
// twiddles) in one launch: the tiles of all jobs form one work list, job j
// owning tiles [start_j, start_j + polys_j * tiles_j); every CTA of a grid
// sized to the resident CTAs of the device walks the list with stride
// gridDim.x. All jobs share the tile size (blockDim = tile / 16), so tiles
// of different N run side by side; the sub-transform length of a job's phase
// (2^logS, 5 <= logS <= 8) selects the instantiation per tile.
constexpr int kMaxNttJobs = 24;
struct NttJob {
  NttArgs A;
  int logS, log2n, tiles, start;  // log2 column and chunk length; tiles per polynomial (columns) or limb (chunks)
  RowPlan rows;  // chunk phase
  int ring;  // the context's m_odd: 3 (m = 3N) or 5 (m = 5N/2) give the column phase its split; 1 none
};
struct NttMulti {
  int njobs, total;
  NttJob j[kMaxNttJobs];
};

// a separate function per instantiation, so each keeps its own register allocation
template <bool FWD, int LOGS, int LOG2N, int RING>
__device__ __noinline__ void ntt16_cols_fn(const NttArgs& A, int tile, int poly) {
  ntt16_cols<FWD, LOGS, LOG2N, kColTile - LOGS, RING>(A, tile, poly);
}
template <bool FWD, int LOGS, bool SRC>
__device__ __noinline__ void ntt16_rows_fn(const NttArgs& A, const RowPlan& R, int item, int limb) {
  ntt16_rows<FWD, LOGS, SRC>(A, R, item, limb);
}

template <bool FWD, bool COLS, bool SRC>
__global__ void __launch_bounds__(128, 6) k_ntt16_multi(const __grid_constant__ NttMulti M) {
  for (int t = blockIdx.x; t < M.total; t += gridDim.x) {
    int j = 0;
    while (j + 1 < M.njobs && t >= M.j[j + 1].start) ++j;
    const NttJob& J = M.j[j];
    const int local = t - J.start;
    const int poly = local / J.tiles, tile = local - poly * J.tiles;
    if constexpr (COLS) {
      switch (J.ring * 16 + J.logS) {
        case 16 + 5: ntt16_cols_fn<FWD, 5, 8, 1>(J.A, tile, poly); break;
        case 16 + 6: ntt16_cols_fn<FWD, 6, 8, 1>(J.A, tile, poly); break;
        case 16 + 7: ntt16_cols_fn<FWD, 7, 8, 1>(J.A, tile, poly); break;
        case 16 + 8: ntt16_cols_fn<FWD, 8, 8, 1>(J.A, tile, poly); break;
        case 48 + 5: ntt16_cols_fn<FWD, 5, 8, 3>(J.A, tile, poly); break;
        case 48 + 6: ntt16_cols_fn<FWD, 6, 8, 3>(J.A, tile, poly); break;
        case 48 + 7: ntt16_cols_fn<FWD, 7, 8, 3>(J.A, tile, poly); break;
        case 48 + 8: ntt16_cols_fn<FWD, 8, 8, 3>(J.A, tile, poly); break;
        case 80 + 6:
          if (J.log2n == 7) ntt16_cols_fn<FWD, 6, 7, 5>(J.A, tile, poly);
          else ntt16_cols_fn<FWD, 6, 8, 5>(J.A, tile, poly);
          break;
        case 80 + 7: ntt16_cols_fn<FWD, 7, 8, 5>(J.A, tile, poly); break;
        default: ntt16_cols_fn<FWD, 8, 8, 5>(J.A, tile, poly); break;
      }
    } else if (J.log2n == 7) {
      ntt16_rows_fn<FWD, 7, SRC>(J.A, J.rows, tile, poly);  // poly counts limbs here
    } else {
      ntt16_rows_fn<FWD, 8, SRC>(J.A, J.rows, tile, poly);
    }
    __syncthreads();  // the next tile reuses the shared memory
  }
}

// column phase of one transform by halves
template <bool FWD, int LOGS, int LOG2N, int RING>
void launch_cols_as(int sms, int npoly, cudaStream_t st, const NttArgs& A) {
  constexpr int CL = kColTile - LOGS, CLB = kColTileBig - LOGS;
  if (((long)npoly << (LOGS + LOG2N - kColTileBig)) >= 2L * SS_COLS_BIG * sms)
    launch_early(k_ntt16_cols<FWD, LOGS, LOG2N, CLB, RING>, dim3(1 << (LOG2N - CLB), npoly), 256,
                 col_smem<LOGS, CLB>(), st, A);
  else
    launch_early(k_ntt16_cols<FWD, LOGS, LOG2N, CL, RING>, dim3(1 << (LOG2N - CL), npoly), 128,
                 col_smem<LOGS, CL>(), st, A);
}
template <bool FWD>
void launch_cols(const Context& C, int logS, int log2n, int npoly, cudaStream_t st, const NttArgs& A) {
  switch (C.m_odd * 16 + logS) {
    case 16 + 5: launch_cols_as<FWD, 5, 8, 1>(C.sms, npoly, st, A); break;
    case 16 + 6: launch_cols_as<FWD, 6, 8, 1>(C.sms, npoly, st, A); break;
    case 16 + 7: launch_cols_as<FWD, 7, 8, 1>(C.sms, npoly, st, A); break;
    case 16 + 8: launch_cols_as<FWD, 8, 8, 1>(C.sms, npoly, st, A); break;
    case 48 + 5: launch_cols_as<FWD, 5, 8, 3>(C.sms, npoly, st, A); break;
    case 48 + 6: launch_cols_as<FWD, 6, 8, 3>(C.sms, npoly, st, A); break;
    case 48 + 7: launch_cols_as<FWD, 7, 8, 3>(C.sms, npoly, st, A); break;
    case 48 + 8: launch_cols_as<FWD, 8, 8, 3>(C.sms, npoly, st, A); break;
    case 80 + 6:
      if (log2n == 7) launch_cols_as<FWD, 6, 7, 5>(C.sms, npoly, st, A);
      else launch_cols_as<FWD, 6, 8, 5>(C.sms, npoly, st, A);
      break;
    case 80 + 7: launch_cols_as<FWD, 7, 8, 5>(C.sms, npoly, st, A); break;
    default: launch_cols_as<FWD, 8, 8, 5>(C.sms, npoly, st, A); break;
  }
}

// one phase of a transform in the Shoup form
template <bool FWD, bool COLS, bool LAST, bool SRC = false, int RING = 1>
void launch16(int logS, dim3 g, int thr, size_t smem, cudaStream_t st, const NttArgs& A, int logc, int m0) {
  if constexpr (COLS) {
    switch (logS) {
      case 5: k_ntt16<FWD, COLS, LAST, 5, SRC, RING><<<g, thr, smem, st>>>(A, logc, m0); return;
      case 6: k_ntt16<FWD, COLS, LAST, 6, SRC, RING><<<g, thr, smem, st>>>(A, logc, m0); return;
      default: break;
    }
  }
  if (logS == 7) k_ntt16<FWD, COLS, LAST, 7, SRC, RING><<<g, thr, smem, st>>>(A, logc, m0);
  else k_ntt16<FWD, COLS, LAST, 8, SRC, RING><<<g, thr, smem, st>>>(A, logc, m0);
}

// How one launch of the chunk phase covers a set: the polynomials of a limb in
// groups of up to a CTA's rows (fewer when the limb has fewer), and the shared
// memory a CTA needs.
RowPlan row_plan(const PolySet& s, int rows) {
  RowPlan R;
  R.lnp = 0;
  while ((1 << R.lnp) < rows && (1 << R.lnp) < s.n_outer) ++R.lnp;
  R.groups = (s.n_outer + (1 << R.lnp) - 1) >> R.lnp;
  return R;
}
size_t row_smem(int logS, int thr, int lnp) {
  const int rows = thr >> (logS - 4);
  return ((size_t)(rows >> lnp) << logS) * 24 + (size_t)rows * 8 * (1 << logS);
}

template <bool FWD, bool SRC>
void launch_rows(int logS, const PolySet& s, cudaStream_t st, const NttArgs& A) {
  int thr = 128;
  RowPlan R = row_plan(s, thr >> (logS - 4));
  while (row_smem(logS, thr, R.lnp) > 48 * 1024) {  // few polynomials: fewer rows, not more than the default limit
    thr /= 2;
    R = row_plan(s, thr >> (logS - 4));
  }
  const dim3 g(((A.N >> logS) / ((thr >> (logS - 4)) >> R.lnp)) * R.groups, s.nl);
  const size_t smem = row_smem(logS, thr, R.lnp);
  if (logS == 7) launch_early(k_ntt16_rows<FWD, 7, SRC>, g, thr, smem, st, A, R);
  else launch_early(k_ntt16_rows<FWD, 8, SRC>, g, thr, smem, st, A, R);
}

// log2 of the chunk length N2 of the two-phase split: 256, except that the
// m = 5N/2 ring needs at least 64 column words (its inverse split takes the
// column phase's last two stages in one register round)
int chunk_log(const Context& C) { return C.m_odd == 5 && C.logN - 8 < 6 ? C.logN - 6 : 8; }

NttArgs make_args(Context& C, const PolySet& s) {
  NttArgs A;
  A.base = s.base;
  A.outer_stride = s.outer_stride;
  A.n_outer = s.n_outer;
  A.nl = s.nl;
  A.q0 = s.q0;
  A.nq = s.nq;
  A.L = C.L;
  A.N = C.N;
  A.skip_w = s.skip_w;
  A.skip_mod = s.skip_mod;
  A.skip_level = s.skip_level;
  A.mods = reinterpret_cast<const Modulus*>(C.d_mod);
  A.tw = C.d_tw;
  A.tp = C.d_tp;
  A.tws = C.d_tp ? ntt_tw_slots(C) : 0;
  A.ninv = C.d_ninv;
  A.split = C.d_split;
  A.src = nullptr;
  A.src_os = 0;
  if (s.pre_w1 && C.m_odd != 1) throw Error(SS_ERR_PARAM, "node-1 twiddle folding is for the ring X^N + 1");
  if (s.post_scale && (C.m_odd != 1 || C.N <= TILE))
    throw Error(SS_ERR_PARAM, "deferred inverse scaling is for two-phase transforms on the ring X^N + 1");
  A.pre_w1 = s.pre_w1 ? 1 : 0;
  A.post_scale = s.post_scale ? 1 : 0;
  return A;
}

double active_polys(const PolySet& s);

// Shoup products of one transform of the set: N/2 per stage and polynomial,
// less node 1's when folded (pre_w1), plus the inverse's N^-1: on the sums of
// the last stage (two-phase transforms, N/2) or on every word (single-phase,
// N), none when the last stage is deferred (post_scale: no products there)
double ntt_products(const Context& C, const PolySet& s, bool fwd) {
  const double half = C.N / 2.0;
  const int inv_extra = s.post_scale ? -1 : (C.N <= TILE ? 2 : 1);
  return active_polys(s) * half * (C.logN + (fwd ? (s.pre_w1 ? -1 : 0) : inv_extra));
}

// polynomials a transform actually touches (ModUp outputs skip the digit's own limbs)
double active_polys(const PolySet& s) {
  double n = (double)s.n_outer * s.nl;
  if (s.skip_w > 0)
    for (int o = 0; o < s.n_outer; ++o) {
      int lo = (o % s.skip_mod) * s.skip_w, hi = std::min(lo + s.skip_w, s.skip_level);
      if (hi > lo) n -= hi - lo;
    }
  return n;
}

}  // namespace

NttMerger*& ntt_merger() {
  static thread_local NttMerger* m = nullptr;
  return m;
}

// Products by halves: slot of node k in one prime's and direction's table of
// N + N1 slots (see half_tw).
int ntt_tw_slots(const Context& C) { return C.N + (C.N >> chunk_log(C)); }
int ntt_tw_slot(const Context& C, int k) {
  const int l2 = chunk_log(C), l1 = C.logN - l2;
  int depth = 0;
  while ((2 << depth) <= k) ++depth;
  if (depth < l1) return tw_slot(k, l1 - 1 - depth, l1 < 8 ? l1 - 4 : 4);  // the column phase's stages come first
  const int s = depth - l1, chunk = (k >> s) - (1 << l1), local = (1 << s) + (k & ((1 << s) - 1));
  return (1 << l1) + (chunk << l2) + tw_slot(local, l2 - 1 - s, l2 - 4);
}

// src: optional out-of-place source read by the first phase (inverse only)
static void launch(Context& C, const PolySet& s, bool fwd, cudaStream_t st, const u64* src = nullptr,
                   long src_os = 0) {
  int npoly = s.n_outer * s.nl;
  if (npoly == 0) return;
  if (ntt_merger() && C.N > TILE && C.d_tp && !is_dry(C)) {
    ntt_merger()->submit(NttReq{&C, s, src, src_os}, fwd, st);
    return;
  }
  if (npoly > 65535) throw Error(SS_ERR_SHAPE, "too many polynomials in one transform");
  NttArgs A = make_args(C, s);
  const int N = C.N, logN = C.logN;
  auto smem = [](int words) { return (size_t)(words + words / 8) * 8; };
  if (N <= TILE) {
    if (src)  // one in-place phase: copy first
      SS_CUDA(cudaMemcpy2DAsync(s.base, (size_t)s.outer_stride * 8, src, (size_t)src_os * 8, (size_t)s.nl * N * 8,
                                s.n_outer, cudaMemcpyDeviceToDevice, st));
    int kr = kt_begin(C, st);
    dim3 g(1, npoly);
    int thr = N / 8;
    if (C.m_odd == 5) {  // the split, then the four factors as chunks of N/4 (nodes 4..7 and below)
      if (fwd) k_ntt<true, false, true, 5><<<g, thr, smem(N), st>>>(A, logN - 2, 2, 4);
      else k_ntt<false, false, true, 5><<<g, thr, smem(N), st>>>(A, logN - 2, 2, 4);
    } else if (C.m_odd == 3) {
      if (fwd) k_ntt<true, false, true, 3><<<g, thr, smem(N), st>>>(A, logN, 0, 1);
      else k_ntt<false, false, true, 3><<<g, thr, smem(N), st>>>(A, logN, 0, 1);
    } else {
      if (fwd) k_ntt<true, false, true><<<g, thr, smem(N), st>>>(A, logN, 0, 1);
      else k_ntt<false, false, true><<<g, thr, smem(N), st>>>(A, logN, 0, 1);
    }
    ++C.launches;
    if (kr >= 0) C.kt.ntt_products += ntt_products(C, s, fwd);
    kt_end(C, kr, KC_NTT, 16.0 * N * active_polys(s), st);
  } else {
    int kr = kt_begin(C, st);
    const int log2n = chunk_log(C), log1 = logN - log2n;  // N = N1 * N2, N2 = 2^log2n
    const int tl = C.ntt_tile_log == 11 ? 11 : 12, tile = 1 << tl;
    const int logc1 = tl - log1, logc2 = tl - log2n;
    dim3 g1(1 << (log2n - logc1), npoly), g2(1 << (log1 - logc2), npoly);
    const int thr = tile / 16;
    if (A.tp) {
      NttArgs A1 = A;
      if (src) {
        A1.src = src;
        A1.src_os = src_os;
      }
      if (fwd) {
        launch_cols<true>(C, log1, log2n, npoly, st, A);
        launch_rows<true, false>(log2n, s, st, A);
      } else {
        if (src) launch_rows<false, true>(log2n, s, st, A1);
        else launch_rows<false, false>(log2n, s, st, A);
        launch_cols<false>(C, log1, log2n, npoly, st, A);
      }
    } else if (fwd) {
      if (C.m_odd == 3) launch16<true, true, false, false, 3>(log1, g1, thr, smem(tile), st, A, logc1, 1);
      else if (C.m_odd == 5) launch16<true, true, false, false, 5>(log1, g1, thr, smem(tile), st, A, logc1, 1);
      else launch16<true, true, false>(log1, g1, thr, smem(tile), st, A, logc1, 1);
      launch16<true, false, true>(log2n, g2, thr, smem(tile), st, A, logc2, 1 << log1);
    } else {
      if (src) {
        NttArgs A1 = A;
        A1.src = src;
        A1.src_os = src_os;
        launch16<false, false, false, true>(log2n, g2, thr, smem(tile), st, A1, logc2, 1 << log1);
      } else {
        launch16<false, false, false>(log2n, g2, thr, smem(tile), st, A, logc2, 1 << log1);
      }
      if (C.m_odd == 3) launch16<false, true, true, false, 3>(log1, g1, thr, smem(tile), st, A, logc1, 1);
      else if (C.m_odd == 5) launch16<false, true, true, false, 5>(log1, g1, thr, smem(tile), st, A, logc1, 1);
      else launch16<false, true, true>(log1, g1, thr, smem(tile), st, A, logc1, 1);
    }
    C.launches += 2;
    if (kr >= 0) C.kt.ntt_products += ntt_products(C, s, fwd);
    kt_end(C, kr, KC_NTT, 16.0 * N * active_polys(s), st);
  }
  SS_CUDA(cudaGetLastError());
}

static int resident_ctas() {
  static std::atomic<int> n{0};
  int v = n.load();
  if (!v) {
    int dev = 0, sms = 0;
    SS_CUDA(cudaGetDevice(&dev));
    SS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    v = sms * 6;
    n.store(v);
  }
  return v;
}

template <bool FWD, bool COLS, bool SRC>
static void launch_multi(const NttMulti& M, int thr, size_t smem, cudaStream_t st) {
  if (M.total == 0) return;
  const int grid = std::min(M.total, resident_ctas());
  if (smem > 48 * 1024) {  // many chunks of few polynomials: opt in once per kernel and device
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    SS_CUDA(cudaGetDevice(&dev));
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(done.load() & bit)) {
      SS_CUDA(cudaFuncSetAttribute(k_ntt16_multi<FWD, COLS, SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   128 * 1024));
      done.fetch_or(bit);
    }
  }
  k_ntt16_multi<FWD, COLS, SRC><<<grid, thr, smem, st>>>(M);
  SS_CUDA(cudaGetLastError());
}

void ntt_multi(const std::vector<NttReq>& reqs, bool fwd, cudaStream_t st) {
  const int thr = 128;
  const size_t smem_cols = col_smem<8, kColTile - 8>();  // the longest columns' twiddles and a tile
  for (size_t b0 = 0; b0 < reqs.size(); b0 += kMaxNttJobs) {
    const size_t b1 = std::min(reqs.size(), b0 + kMaxNttJobs);
    // phase 1 (columns forward, chunks inverse) and phase 2 of every job
    NttMulti P1, P2;
    P1.njobs = P2.njobs = 0;
    P1.total = P2.total = 0;
    double bytes = 0, prods = 0;
    size_t smem_rows = 0;
    for (size_t r = b0; r < b1; ++r) {
      const NttReq& q = reqs[r];
      Context& C = *q.C;
      if (C.N < 8192 || !C.d_tp) throw Error(SS_ERR_PARAM, "merged transforms need N >= 8192 and primes below 2^55");
      const int npoly = q.s.n_outer * q.s.nl;
      if (npoly == 0) continue;
      NttArgs A = make_args(C, q.s);
      const int l2 = chunk_log(C), log1 = C.logN - l2;
      const RowPlan R = row_plan(q.s, thr >> (l2 - 4));
      const int rows = thr >> (l2 - 4);
      NttJob cols{A, log1, l2, 1 << (l2 - (kColTile - log1)), 0, R, C.m_odd};
      NttJob chunks{A, log1, l2, ((1 << log1) / (rows >> R.lnp)) * R.groups, 0, R, 1};
      smem_rows = std::max(smem_rows, row_smem(l2, thr, R.lnp));
      if (!fwd) {  // the chunk phase reads the source (the polynomials themselves when in place)
        chunks.A.src = q.src ? q.src : q.s.base;
        chunks.A.src_os = q.src ? q.src_os : q.s.outer_stride;
      }
      NttJob& j1 = P1.j[P1.njobs++];
      NttJob& j2 = P2.j[P2.njobs++];
      j1 = fwd ? cols : chunks;
      j2 = fwd ? chunks : cols;
      j1.start = P1.total;
      j2.start = P2.total;
      P1.total += (fwd ? npoly : q.s.nl) * j1.tiles;
      P2.total += (fwd ? q.s.nl : npoly) * j2.tiles;
      bytes += 16.0 * C.N * active_polys(q.s);
      prods += ntt_products(C, q.s, fwd);
    }
    if (P1.njobs == 0) continue;
    Context& C0 = *reqs[b0].C;
    int kr = kt_begin(C0, st);
    if (fwd) {
      launch_multi<true, true, false>(P1, 128, smem_cols, st);
      launch_multi<true, false, false>(P2, thr, smem_rows, st);
    } else {
      launch_multi<false, false, true>(P1, thr, smem_rows, st);
      launch_multi<false, true, false>(P2, 128, smem_cols, st);
    }
    C0.launches += 2;
    if (kr >= 0) C0.kt.ntt_products += prods;
    kt_end(C0, kr, KC_NTT, bytes, st);
  }
}

void ntt_forward(Context& C, const PolySet& s, cudaStream_t st) { launch(C, s, true, st); }

bool rows_ip_fits(const Context& C, int level) {
  return C.d_tp && !ntt_merger() && !ks_merger() && (level + C.alpha - 1) / C.alpha + 1 <= kRowsIpMax;
}

void ntt_forward_cols(Context& C, const PolySet& s, cudaStream_t st) {
  const int npoly = s.n_outer * s.nl, l2 = chunk_log(C);
  if (npoly == 0) return;
  if (npoly > 65535) throw Error(SS_ERR_SHAPE, "too many polynomials in one transform");
  int kr = kt_begin(C, st);
  launch_cols<true>(C, C.logN - l2, l2, npoly, st, make_args(C, s));
  ++C.launches;
  if (kr >= 0) C.kt.ntt_products += ntt_products(C, s, true);
  kt_end(C, kr, KC_NTT, 16.0 * C.N * active_polys(s), st);
}

void rows_ip(Context& C, const RowsIpReq& R, cudaStream_t st) {
  const int l2 = chunk_log(C), tpr = (1 << l2) / 16;
  RowsIp A{};
  PolySet none{nullptr, 0, 1, 1, 0, 1};
  A.tab = make_args(C, none);
  A.mods = A.tab.mods;
  A.ext = R.ext;
  A.d = R.d;
  A.kb = R.K->b;
  A.ka = R.K->a;
  A.level = R.level;
  A.alpha = C.alpha;
  A.L = C.L;
  A.T = C.ntot;
  A.N = C.N;
  A.dn = (R.level + C.alpha - 1) / C.alpha;
  A.ext_os = (long)A.dn * (R.level + C.alpha) * C.N;
  A.d_os = R.d_os;
  A.B = R.B;
  A.m0 = R.m0;
  A.acc = R.acc;
  A.acc_os = 2L * R.nlimbs * C.N;
  A.acc_nl = R.nlimbs;
  A.x = R.x ? R.x->data : nullptr;
  A.x_os = R.x ? (long)R.x->ncomp * R.x->cap * C.N : 0;
  A.x_cap = R.x ? R.x->cap : 0;
  A.add_c1 = R.add_c1 ? 1 : 0;
  A.delta = R.delta;
  A.nl = R.nlimbs;
  A.pm = R.pm;
  A.scale = R.scale;
  if (R.out) {
    A.out = R.out->data;
    A.out_os = (long)R.out->ncomp * R.out->cap * C.N;
    A.out_cap = R.out->cap;
  }
  // rows of one ciphertext: every digit but a data limb's own, and the two of the correction
  const int rpc = R.type == 0 ? A.dn : A.dn + 1;
  A.nb = std::max(1, std::min(R.B, kRowsIpMax / rpc));
  A.bgroups = (R.B + A.nb - 1) / A.nb;
  const dim3 g((C.N >> l2) * A.bgroups, R.nlimbs);
  // the rows' threads; a grid that leaves room gets 256 a CTA for the sums, whose
  // loads are then one round deep (rotations near the chain's end: 815 -> 610 us)
  int thr = (A.nb * rpc * tpr + 31) / 32 * 32;
  if ((long)g.x * g.y <= (long)SS_ROWS_IP * C.sms) thr = 256;
  const size_t smem = ((size_t)24 << l2) + (size_t)(thr / tpr) * 8 * (1 << l2);
  const double words = (double)A.dn * R.nlimbs * (R.B + 2.0) +
                       (R.type == 0 ? 2.0 : 4.0 + (R.x ? 2.0 : 0.0)) * R.nlimbs * R.B;
  int kr = kt_begin(C, st);
  if (l2 == 7) {
    if (R.type == 0) launch_early(k_rows_ip<7, 0>, g, thr, smem, st, A);
    else if (R.type == 1) launch_early(k_rows_ip<7, 1>, g, thr, smem, st, A);
    else launch_early(k_rows_ip<7, 2>, g, thr, smem, st, A);
  } else {
    if (R.type == 0) launch_early(k_rows_ip<8, 0>, g, thr, smem, st, A);
    else if (R.type == 1) launch_early(k_rows_ip<8, 1>, g, thr, smem, st, A);
    else launch_early(k_rows_ip<8, 2>, g, thr, smem, st, A);
  }
  ++C.launches;
  kt_end(C, kr, KC_KSIP, words * C.N * 8.0, st);
}

void ntt_inverse(Context& C, const PolySet& s, cudaStream_t st) { launch(C, s, false, st); }

void ntt_inverse_from(Context& C, const PolySet& s, const u64* src, long src_os, cudaStream_t st) {
  launch(C, s, false, st, src, src_os);
}

}  // namespace ss
