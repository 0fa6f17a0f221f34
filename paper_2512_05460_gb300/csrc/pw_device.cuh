// Device-side building blocks of the ProbeWalk walk kernel (sm_103a).
//
//  * Philox4x32-10 (Salmon et al., SC'11), written from its published round
//    and key-schedule definition.
//  * The stateless Paired-Sign Probe of Section 3.3: a cycle-walking Feistel
//    permutation pi_k on [n], zero set U = {v : pi_k(v) >= n - r}, pair id
//    floor(pi_k(v)/2), 2-universal sign hash h_k(u) = ((a_k u + b_k) mod p) mod 2
//    with p = 2^31 - 1, and z_v = (-1)^(h_k(pair) + pi_k(v)).
//  * Graph records: every CSR entry e of row v holds the neighbour u = col[e] as
//    {u, row_start(u), deg(u), bits of the FP32 reciprocal 1/deg(u)}, so one
//    16-byte gather per step yields everything the next step and the
//    accumulation need (Algorithm 1, inner loop).
#pragma once
#include <stdint.h>

namespace pw {

constexpr uint32_t kPhiloxM0 = 0xD2511F53u;
constexpr uint32_t kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u;
constexpr uint32_t kPhiloxW1 = 0xBB67AE85u;

// Counter word 3 tags of the independent streams.
constexpr uint32_t kTagWalk = 1u, kTagWalkPilot = 2u, kTagProbe = 3u, kTagProbePilot = 4u, kTagSeed = 0x5EEDu;
constexpr uint64_t kHashPrime = 2147483647ull;  // p = 2^31 - 1

struct Philox4 {
  uint32_t x, y, z, w;
};

__host__ __device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * (uint64_t)b) >> 32);
#endif
}

// Ten rounds; round r uses key + r * (W0, W1).
__host__ __device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                           uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = mulhi32(kPhiloxM0, c0), lo0 = kPhiloxM0 * c0;
    const uint32_t hi1 = mulhi32(kPhiloxM1, c2), lo1 = kPhiloxM1 * c2;
    c0 = hi1 ^ c1 ^ k0;
    c1 = lo1;
    c2 = hi0 ^ c3 ^ k1;
    c3 = lo0;
    k0 += kPhiloxW0;
    k1 += kPhiloxW1;
  }
  return Philox4{c0, c1, c2, c3};
}

// Round keys of one query key, hoisted out of the walk loop (the key schedule
// is the same for every counter of the query).
struct PhiloxKeys {
  uint32_t k0[10], k1[10];
};

__host__ __device__ __forceinline__ PhiloxKeys philox_keys(uint64_t seed) {
  PhiloxKeys K;
  uint32_t a = (uint32_t)seed, b = (uint32_t)(seed >> 32);
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    K.k0[r] = a;
    K.k1[r] = b;
    a += kPhiloxW0;
    b += kPhiloxW1;
  }
  return K;
}

__host__ __device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                           const PhiloxKeys& K) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = mulhi32(kPhiloxM0, c0), lo0 = kPhiloxM0 * c0;
    const uint32_t hi1 = mulhi32(kPhiloxM1, c2), lo1 = kPhiloxM1 * c2;
    c0 = hi1 ^ c1 ^ K.k0[r];
    c1 = lo1;
    c2 = hi0 ^ c3 ^ K.k1[r];
    c3 = lo0;
  }
  return Philox4{c0, c1, c2, c3};
}

__host__ __device__ __forceinline__ Philox4 philox_seeded(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2,
                                                           uint32_t c3) {
  return philox4x32_10(c0, c1, c2, c3, (uint32_t)seed, (uint32_t)(seed >> 32));
}

__host__ __device__ __forceinline__ uint64_t default_seed(uint64_t global_seed, int64_t s, int64_t t, double eps,
                                                          int32_t L) {
  uint64_t eb;
#ifdef __CUDA_ARCH__
  eb = (uint64_t)__double_as_longlong(eps);
#else
  __builtin_memcpy(&eb, &eps, sizeof eb);
#endif
  const Philox4 o = philox_seeded(global_seed ^ eb, (uint32_t)s, (uint32_t)t, (uint32_t)L, kTagSeed);
  return (uint64_t)o.x | ((uint64_t)o.y << 32);
}

// Seed of truncation level L of a stabilized query: the first two words of the
// Philox block keyed by the query seed with counter (L, 0, 0, 0x57AB).
constexpr uint32_t kTagLevel = 0x57ABu;
__host__ __device__ __forceinline__ uint64_t level_seed(uint64_t seed, int32_t L) {
  const Philox4 o = philox_seeded(seed, (uint32_t)L, 0u, 0u, kTagLevel);
  return (uint64_t)o.x | ((uint64_t)o.y << 32);
}

// ---- Paired-Sign Probe -------------------------------------------------------

struct Probe {
  uint32_t n;         // nodes
  uint32_t n_active;  // n - r
  uint32_t lo;        // Feistel halves hi and lo: domain 2^(hi + lo) >= n, hi = lo or lo + 1
  uint32_t sh_hi, sh_lo;  // 32 - hi, 32 - lo
  uint32_t pow_lo, mask_lo;  // 2^lo, 2^lo - 1
  uint32_t rounds;    // 8, or 12 when hi + lo <= 4
  uint32_t a, b;      // hash parameters, a in [1, p-1], b in [0, p-1]
  uint32_t key[12];   // round keys 0 and 1, then key i XOR key i - 2 (feistel_pass)
  uint32_t out1, out2;  // the last two round keys: out2 of the last round, out1 of the one before
};

// Domain bits: the smallest b >= 2 with 2^b >= n, with b = 3 raised to 4 (the
// 2+1-bit network on [8] pairs visibly non-uniformly for n = 5, 6).  Odd b
// splits into a left half one bit wider than the right half.
__host__ __device__ __forceinline__ void feistel_bits(uint32_t n, uint32_t& hi, uint32_t& lo) {
  uint32_t b = 2;
  while (b < 31 && (1ull << b) < (uint64_t)n) ++b;
  if (b == 3) b = 4;
  hi = (b + 1) / 2;
  lo = b / 2;
}

// Probe k of the query keyed by `seed` on stream tag `tag`:
//   words of (k,0,0,tag): a = 1 + (w0|w1<<32) mod (p-1), b = (w2|w3<<32) mod p;
//   words of (k,1,j,tag), j = 0,1,2: round keys 4j..4j+3;
//   word 0 of (k,2,0,tag): parity coin r = 2 (bit 0) for even n, r = 1 for odd n.
__host__ __device__ __forceinline__ Probe probe_from_words(uint32_t n, const Philox4& ab, const Philox4& k0,
                                                           const Philox4& k1, const Philox4& k2, uint32_t coin) {
  Probe P;
  P.n = n;
  uint32_t hi;
  feistel_bits(n, hi, P.lo);
  P.sh_hi = 32u - hi;
  P.sh_lo = 32u - P.lo;
  P.pow_lo = 1u << P.lo;
  P.mask_lo = P.pow_lo - 1u;
  P.rounds = (hi + P.lo <= 4) ? 12u : 8u;
  const uint64_t wa = (uint64_t)ab.x | ((uint64_t)ab.y << 32);
  const uint64_t wb = (uint64_t)ab.z | ((uint64_t)ab.w << 32);
  P.a = (uint32_t)(1 + wa % (kHashPrime - 1));
  P.b = (uint32_t)(wb % kHashPrime);
  const uint32_t key[12] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w, k2.x, k2.y, k2.z, k2.w};
  P.key[0] = key[0];
  P.key[1] = key[1];
#pragma unroll
  for (int i = 2; i < 12; ++i) P.key[i] = key[i] ^ key[i - 2];
  P.out1 = P.rounds == 8u ? key[6] : key[10];
  P.out2 = P.rounds == 8u ? key[7] : key[11];
  P.n_active = n - ((n & 1u) ? 1u : 2u * (coin & 1u));
  return P;
}

__host__ __device__ __forceinline__ Probe make_probe(uint32_t n, uint64_t seed, uint32_t k, uint32_t tag) {
  return probe_from_words(n, philox_seeded(seed, k, 0u, 0u, tag), philox_seeded(seed, k, 1u, 0u, tag),
                          philox_seeded(seed, k, 1u, 1u, tag), philox_seeded(seed, k, 1u, 2u, tag),
                          philox_seeded(seed, k, 2u, 0u, tag).x);
}

#ifdef __CUDACC__
// The same by a whole warp with the same arguments: lanes 0 to 4 evaluate one
// of the five Philox blocks each and the words go round by shuffles, a quarter
// of the instructions of five blocks in every lane.
__device__ __forceinline__ Probe make_probe_warp(uint32_t n, uint64_t seed, uint32_t k, uint32_t tag) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t c1 = lane == 0u ? 0u : (lane <= 3u ? 1u : 2u), c2 = lane == 2u ? 1u : (lane == 3u ? 2u : 0u);
  const Philox4 own = philox_seeded(seed, k, c1, c2, tag);
  Philox4 w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    w[j].x = __shfl_sync(0xffffffffu, own.x, j);
    w[j].y = __shfl_sync(0xffffffffu, own.y, j);
    w[j].z = __shfl_sync(0xffffffffu, own.z, j);
    w[j].w = __shfl_sync(0xffffffffu, own.w, j);
  }
  return probe_from_words(n, w[0], w[1], w[2], w[3], __shfl_sync(0xffffffffu, own.x, 4));
}
#endif

// Round function of u = x ^ key: top 32 - shift bits of (u * C1, xor-folded by
// 16, * C2).  (The last shift as a high-word product, to move it off the
// shift-and-logic pipe, was slower: 64 shifts but 32 high words per SM and clock.)
__host__ __device__ __forceinline__ uint32_t feistel_f(uint32_t u, uint32_t shift) {
  uint32_t y = u * 0x9E3779B1u;
  y ^= y >> 16;
  y *= 0x85EBCA6Bu;
  return y >> shift;
}

// One pass of the Feistel network on [2^hi] x [2^lo] (the generalised
// construction for such domains, Black and Rogaway 2002): a round maps
// (left, right) to (right, left ^ F(right)) with F as wide as the left half,
// so the halves trade widths every round; after the even round count the left
// half has hi bits again.  With x_0 = left, x_1 = right and x_{i+1} = x_{i-1} ^
// F(x_i ^ key), the pass carries u_i = x_i ^ key(i-1): then u_{i+1} = u_{i-1} ^
// F ^ (key(i-2) ^ key(i)) is one three-input operation a round, where x and x ^
// key took three.
template <int ROUNDS>
__host__ __device__ __forceinline__ uint32_t feistel_pass(const Probe& P, uint32_t x) {
  const uint32_t left = x >> P.lo, right = x & P.mask_lo;
  uint32_t u0 = right ^ P.key[0];                                   // u_1
  uint32_t u1 = left ^ feistel_f(u0, P.sh_hi) ^ P.key[1];          // u_2
#pragma unroll
  for (int i = 2; i < ROUNDS; ++i) {
    const uint32_t u2 = u0 ^ feistel_f(u1, (i & 1) ? P.sh_hi : P.sh_lo) ^ P.key[i];
    u0 = u1;
    u1 = u2;
  }
  // the halves do not overlap: a product and a sum join them off the shift-and-logic pipe
  return (u1 ^ P.out2) * P.pow_lo + (u0 ^ feistel_f(u1, P.sh_lo) ^ P.out1);
}

__host__ __device__ __forceinline__ uint32_t feistel_once(const Probe& P, uint32_t x) {
  return P.rounds == 8u ? feistel_pass<8>(P, x) : feistel_pass<12>(P, x);
}

// pi_k(v) by cycle-walking the permutation of [2^(hi + lo)] back into [n].
__host__ __device__ __forceinline__ uint32_t probe_pi(const Probe& P, uint32_t v) {
  uint32_t x = v;
  do {
    x = feistel_once(P, x);
  } while (x >= P.n);
  return x;
}

// Sign of a node outside the zero set (pi < n - r), in bit 31: set (z = -1) when
// h(pi / 2) + pi is odd, h the parity of (a u + b) mod p, p = 2^31 - 1, for
// a, b < p and u < 2^30.  One Mersenne fold m = (t mod 2^31) + floor(t / 2^31) <
// 2p stays in 32 bits; p is odd, so subtracting it when m >= p, that is when
// m + 1 has bit 31 set, flips the parity.  The other bits are not meaningful.
__host__ __device__ __forceinline__ uint32_t probe_sign(const Probe& P, uint32_t pi) {
  const uint64_t t = (uint64_t)P.a * (uint64_t)(pi >> 1) + (uint64_t)P.b;
  const uint32_t lo = (uint32_t)t, hi = (uint32_t)(t >> 32);
#ifdef __CUDA_ARCH__
  const uint32_t m = (lo & 0x7FFFFFFFu) + __funnelshift_l(lo, hi, 1);
#else
  const uint32_t m = (lo & 0x7FFFFFFFu) + ((hi << 1) | (lo >> 31));
#endif
  return ((m ^ pi) * 0x80000000u) ^ (m + 1u);
}

__host__ __device__ __forceinline__ int probe_z(const Probe& P, uint32_t v) {
  const uint32_t pi = probe_pi(P, v);
  return pi >= P.n_active ? 0 : ((probe_sign(P, pi) >> 31) ? -1 : 1);
}

// sum + z/d in FP32 from the stored correctly rounded reciprocal: +-1/d is the
// IEEE quotient of +-1 by d, and 0/d = +0 leaves the sum (never -0: it starts at
// +0).  `sign`: bit 31 set for z = -1; its other bits are ignored.
__device__ __forceinline__ float add_term(float sum, bool zero, uint32_t sign, uint32_t inv_bits) {
  const float next = __fadd_rn(sum, __uint_as_float(inv_bits ^ (sign & 0x80000000u)));
  return zero ? sum : next;
}

}  // namespace pw
