// Walk building blocks shared by the batch kernels and the server kernel:
// Algorithm 1's inner loop for the replicas of one probe, with probe entries
// evaluated at each visit (a warp's pool of visits) or read from a per-probe
// table in shared memory.
#pragma once
#include <stdint.h>

#include "pw_device.cuh"

namespace pw {

// The graph as a walk reads it.  A node record is {v, row_start(v), deg(v),
// bits of the FP32 reciprocal 1/deg(v)}; a step from record `cur` with random
// word w moves to neighbour floor(w deg / 2^32) of the row (Algorithm 1's
// uniform neighbour) and yields that neighbour's record.
//   FusedRecords: rec[e] is the record of col[e]; one 16-byte gather per step.
//     For graphs whose 16 B per entry sit comfortably in L2.
//   SplitRecords: a 4-byte col[e] gather, then the neighbour's record from the
//     n-entry node array; two dependent gathers into arrays 4x and nnz/n times
//     smaller.  For graphs whose fused records would spill out of L2.
//   RankedRecords: the split layout, packed and ordered by degree (below).
struct FusedRecords {
  const int4* __restrict__ rec;
  const int4* __restrict__ node;
  __device__ __forceinline__ int4 start(int32_t v) const { return __ldg(node + v); }
  __device__ __forceinline__ int4 next(const int4& cur, uint32_t w) const {
    return __ldg(rec + ((uint32_t)cur.y + __umulhi(w, (uint32_t)cur.z)));
  }
};

struct SplitRecords {
  const int32_t* __restrict__ col;
  const int4* __restrict__ node;
  __device__ __forceinline__ int4 start(int32_t v) const { return __ldg(node + v); }
  __device__ __forceinline__ int4 next(const int4& cur, uint32_t w) const {
    const int32_t u = __ldg(col + ((uint32_t)cur.y + __umulhi(w, (uint32_t)cur.z)));
    return __ldg(node + u);
  }
};

// The split layout with its nodes ranked by degree: three 21-bit ranks to a
// 64-bit word, 2.67 B an entry, and the node records in rank order, so that the
// hubs, which a walk visits in proportion to their degree, share few lines.  For
// graphs of at most 2^21 nodes whose two arrays do not fit what L2 holds at full
// rate (64 MB: gathers fall from 0.94 per SM and clock to 0.56 at 96 MB and 0.41
// at 126 MB).  R-MAT 2^20, against SplitRecords: 9.3 ps a visit evaluating the
// probe and 4.5 with the table, 10.2 and 5.9 before; ranking is 1.5 % of it.
struct RankedRecords {
  const uint64_t* __restrict__ col;
  const int4* __restrict__ node;    // by node id
  const int4* __restrict__ ranked;  // by rank
  static constexpr uint32_t kBits = 21;
  __device__ __forceinline__ int4 start(int32_t v) const { return __ldg(node + v); }
  __device__ __forceinline__ int4 next(const int4& cur, uint32_t w) const {
    const uint32_t e = (uint32_t)cur.y + __umulhi(w, (uint32_t)cur.z);
    const uint32_t i = e / 3u;
    const uint64_t three = __ldg((const unsigned long long*)col + i);
    return __ldg(ranked + ((uint32_t)(three >> (kBits * (e - 3u * i))) & ((1u << kBits) - 1u)));
  }
};

// Probe entries read from the block's table of z^(k) (built once per probe):
// one sign bit per node (set = negative; node v in bit 31 - v mod 32 of its
// word) plus the ids of the r <= 2 nodes of the zero set, which the bits cannot
// express.
struct ZTable {
  const uint32_t* tab;
  uint32_t zero0, zero1;  // zero-set nodes, 0xFFFFFFFF when absent
  __device__ __forceinline__ uint32_t word(uint32_t v) const { return tab[v >> 5]; }
  // sum + z/d of node v from its table word: rotating left by v mod 32 puts the
  // node's bit in the sign position
  __device__ __forceinline__ float add(float sum, uint32_t word, uint32_t v, uint32_t inv) const {
    return add_term(sum, v == zero0 || v == zero1, __funnelshift_l(word, word, v), inv);
  }
};

// Visits per side that a warp walks ahead before it evaluates their probe
// entries, and the shared memory of one warp's pool (the nodes, then pi, of
// 2 x 32 walks).  Kept small: what shared memory takes of the SM's 256 KB is
// not there for the graph and for the lines of gathers in flight (128 B each,
// 1,500 walks and more per SM): at 50 KB a block the server's walks ran at half
// speed, and with twice the steps a 2000^2 grid took 6.3 ps a visit, not 5.3.
constexpr uint32_t kPoolSteps = 4;  // one Philox block of each walk
struct VisitPool {
  uint32_t node[2 * kPoolSteps * 32];
  Probe probe;  // kept here, not in registers, while the warp walks
};

// pi of every node in pool.node[0..total), in place, by the whole warp.  A
// lane runs one Feistel pass per iteration and takes the pool's next node when
// its pass lands in [n], so that the lanes stay busy whatever their
// cycle-walks' lengths.
template <int ROUNDS>
__device__ __forceinline__ void pool_permute(VisitPool& pool, uint32_t total, uint32_t lane) {
  const Probe pr = pool.probe;
  const uint32_t below = (1u << lane) - 1u;
  // byte offsets into pool.node: of this lane's node, of the next one to take
  const uint32_t end = 4u * total;
  uint32_t at = 4u * lane, next = 128u;
  auto node = [&](uint32_t offset) -> uint32_t& { return *(uint32_t*)((char*)pool.node + offset); };
  uint32_t limit = at < end ? pr.n : 0u;  // no pass of a lane without a node is done
  uint32_t x = at < end ? node(at) : 0u;
  while (next < end + 128u) {  // until as many were done as there are
    x = feistel_pass<ROUNDS>(pr, x);
    const bool done = x < limit;
    const uint32_t who = __ballot_sync(0xffffffffu, done);
    if (done) {
      node(at) = x;
      at = next + 4u * (uint32_t)__popc(who & below);
      if (at < end)
        x = node(at);
      else
        limit = 0u;
    }
    next += 4u * (uint32_t)__popc(who);
  }
}

// One replica per lane (lanes below m <= 32 of one warp; all lanes call) of the
// probe in pool.probe: U_p
// from the walks of pair `pair` from s and t, a and b summed in FP32 in step
// order (Eq. hatphi-def).  The warp walks both sides kPoolSteps visits ahead
// into its pool, evaluates the pool's probe entries together, then adds the
// terms in order.
//
// Bound by the shift-and-logic pipe: a visit costs 2^b / n passes of 26 such
// operations and 16 products, a quarter of a Philox block, and about 20 more.
// Evaluating each step's two nodes in their lane, the warp waited for the
// longest of 32 pairs of cycle-walks: 7.3 passes a step against 3.3 on average
// at n = 0.62 2^b, 3.1 against 2.1 at 0.95 2^b.  Per visit, before and with the
// pool: 10.9 -> 5.8 ps (n = 10^5 in L2), 16.5 -> 10.2 (R-MAT 2^20), 7.4 -> 5.3
// (2000^2 grid).
template <bool DEBUG, class GR>
__device__ __forceinline__ float walk_pair_visit(const GR& gr, uint32_t* visits, uint32_t walk_tag, VisitPool& pool,
                                                 int32_t s, int32_t t, int32_t L, uint64_t seed, uint64_t pair,
                                                 uint32_t m, uint32_t lane) {
  const bool active = lane < m;
  int4 xs = gr.start(s), xt = gr.start(t);
  float a = 0.0f, b = 0.0f;
  const uint64_t ws = 2 * pair;
  uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  const uint32_t count = (uint32_t)L + 1u;
  for (uint32_t v0 = 0; v0 < count; v0 += kPoolSteps) {
    const uint32_t steps = count - v0 < kPoolSteps ? count - v0 : kPoolSteps;
    uint32_t inv_s[kPoolSteps], inv_t[kPoolSteps];
    if (active) {
      asm volatile("" : "+r"(k0), "+r"(k1));  // keeps the 20 round keys from being held over the pool's phase
      // ws is even, so the walks share the high word, and with it the second round's first product
      const Philox4 rs = philox4x32_10((uint32_t)ws, (uint32_t)(ws >> 32), v0 >> 2, walk_tag, k0, k1);
      const Philox4 rt = philox4x32_10((uint32_t)ws + 1u, (uint32_t)(ws >> 32), v0 >> 2, walk_tag, k0, k1);
#pragma unroll
      for (uint32_t j = 0; j < kPoolSteps; ++j) {
        if (j < steps) {
          if (j != 0 || v0 != 0) {
            xs = gr.next(xs, j == 0u ? rs.x : (j == 1u ? rs.y : (j == 2u ? rs.z : rs.w)));
            xt = gr.next(xt, j == 0u ? rt.x : (j == 1u ? rt.y : (j == 2u ? rt.z : rt.w)));
          }
          pool.node[2u * j * m + lane] = (uint32_t)xs.x;
          pool.node[(2u * j + 1u) * m + lane] = (uint32_t)xt.x;
          inv_s[j] = (uint32_t)xs.w;
          inv_t[j] = (uint32_t)xt.w;
          if (DEBUG) {
            atomicAdd(visits + xs.x, 1u);
            atomicAdd(visits + xt.x, 1u);
          }
        }
      }
    }
    __syncwarp();
    if (pool.probe.rounds == 8u)
      pool_permute<8>(pool, 2u * steps * m, lane);
    else
      pool_permute<12>(pool, 2u * steps * m, lane);
    __syncwarp();
    if (active) {
      const Probe pr = pool.probe;
#pragma unroll
      for (uint32_t j = 0; j < kPoolSteps; ++j) {
        if (j < steps) {
          const uint32_t ps = pool.node[2u * j * m + lane], pt = pool.node[(2u * j + 1u) * m + lane];
          a = add_term(a, ps >= pr.n_active, probe_sign(pr, ps), inv_s[j]);
          b = add_term(b, pt >= pr.n_active, probe_sign(pr, pt), inv_t[j]);
        }
      }
    }
  }
  return __fsub_rn(a, b);
}

// Words of the per-probe table: one sign bit per node, then two words for
// the zero set.
__host__ __device__ __forceinline__ uint32_t table_words(uint32_t n) { return (n + 31u) / 32u + 2u; }

// One replica with probe entries from the shared-memory table, software
// pipelined: at step i the gather of X_{i+1} and the table read of X_i are
// issued, and the term of X_{i-1} (whose table word was read one step
// earlier) is added.  The additions keep step order, so the result equals
// walk_pair_visit's bit for bit.
template <bool DEBUG, class GR>
__device__ __forceinline__ float walk_pair_table(const GR& gr, uint32_t* visits, uint32_t walk_tag, const ZTable& zt,
                                                 int32_t s, int32_t t, int32_t L, uint64_t seed, uint64_t pair) {
  const int4 xs = gr.start(s), xt = gr.start(t);
  float a = zt.add(0.0f, zt.word((uint32_t)xs.x), (uint32_t)xs.x, (uint32_t)xs.w);
  float b = zt.add(0.0f, zt.word((uint32_t)xt.x), (uint32_t)xt.x, (uint32_t)xt.w);
  if (DEBUG) {
    atomicAdd(visits + xs.x, 1u);
    atomicAdd(visits + xt.x, 1u);
  }
  if (L == 0) return __fsub_rn(a, b);
  const uint64_t ws = 2 * pair;  // even: both walks have its high word
  const PhiloxKeys keys = philox_keys(seed);
  Philox4 rs = philox4x32_10((uint32_t)ws, (uint32_t)(ws >> 32), 0u, walk_tag, keys);
  Philox4 rt = philox4x32_10((uint32_t)ws + 1u, (uint32_t)(ws >> 32), 0u, walk_tag, keys);
  int4 ns = gr.next(xs, rs.y);
  int4 nt = gr.next(xt, rt.y);
  // pending term: table word, node and reciprocal of the previous step's nodes
  uint32_t ps_word = 0, pt_word = 0, ps_v = 0xFFFFFFFFu, pt_v = 0xFFFFFFFFu, ps_inv = 0, pt_inv = 0;
  bool pending = false;
  for (uint32_t blk = 0;; ++blk) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      if (w == 0 && blk == 0) continue;
      const uint32_t i = blk * 4u + (uint32_t)w;  // ns, nt hold X_i
      const bool more = i < (uint32_t)L;
      int4 ns2 = ns, nt2 = nt;
      if (more) {
        uint32_t wsw, wtw;
        if (w == 3) {
          rs = philox4x32_10((uint32_t)ws, (uint32_t)(ws >> 32), blk + 1u, walk_tag, keys);
          rt = philox4x32_10((uint32_t)ws + 1u, (uint32_t)(ws >> 32), blk + 1u, walk_tag, keys);
          wsw = rs.x;
          wtw = rt.x;
        } else {
          wsw = (w == 0) ? rs.y : (w == 1) ? rs.z : rs.w;
          wtw = (w == 0) ? rt.y : (w == 1) ? rt.z : rt.w;
        }
        ns2 = gr.next(ns, wsw);
        nt2 = gr.next(nt, wtw);
      }
      const uint32_t cs_word = zt.word((uint32_t)ns.x), ct_word = zt.word((uint32_t)nt.x);
      if (pending) {
        a = zt.add(a, ps_word, ps_v, ps_inv);
        b = zt.add(b, pt_word, pt_v, pt_inv);
      }
      if (DEBUG) {
        atomicAdd(visits + ns.x, 1u);
        atomicAdd(visits + nt.x, 1u);
      }
      ps_word = cs_word;
      pt_word = ct_word;
      ps_v = (uint32_t)ns.x;
      pt_v = (uint32_t)nt.x;
      ps_inv = (uint32_t)ns.w;
      pt_inv = (uint32_t)nt.w;
      pending = true;
      if (!more) {
        a = zt.add(a, ps_word, ps_v, ps_inv);
        b = zt.add(b, pt_word, pt_v, pt_inv);
        return __fsub_rn(a, b);
      }
      ns = ns2;
      nt = nt2;
    }
  }
}

// z^(k) of every node into the shared-memory table: one Feistel cycle-walk
// per node, by `threads` threads, of which this is number `tid`.  Each thread
// owns whole 32-node words and runs a flat queue (one
// Feistel pass per iteration; it moves to its next node when a pass lands in
// [n]), so lanes stay busy even though cycle-walk lengths vary.  Nodes of the
// zero set (pi >= n - r) are listed in the two words after the bits.
// The caller sets the two zero-set words to 0xFFFFFFFF beforehand.
__device__ __forceinline__ void build_probe_table(const Probe& pr, uint32_t* tab, uint32_t n, uint32_t tid,
                                                  uint32_t threads) {
  const uint32_t nwords = (n + 31u) / 32u;
  uint32_t* zero = tab + nwords;
  uint32_t w = tid, v = w * 32u, x = v, acc = 0;
  uint32_t stop = n - v < 32u ? n : v + 32u;  // end of the word's nodes
  while (w < nwords) {
    x = feistel_once(pr, x);
    if (x < n) {
      if (x >= pr.n_active) zero[x - pr.n_active] = v;  // its bit is not read
      acc = __funnelshift_l(probe_sign(pr, x), acc, 1);
      if (++v == stop) {
        tab[w] = acc << ((w + 1u) * 32u - stop);  // a last word may hold fewer nodes
        w += threads;
        v = w * 32u;
        stop = n - v < 32u ? n : v + 32u;
      }
      x = v;
    }
  }
}

// The same for a graph of few nodes by `warps` warps, of which this is number
// `warp`, each taking its share, up to 256 nodes at a time, through its pool.
__device__ __forceinline__ void build_probe_table_team(VisitPool& pool, uint32_t* tab, uint32_t n, uint32_t warp,
                                                       uint32_t warps, uint32_t lane) {
  constexpr uint32_t kMost = 2u * kPoolSteps * 32u;
  const uint32_t n_active = pool.probe.n_active;
  const uint32_t share = (n / warps + 32u) & ~31u;  // whole words
  const uint32_t batch = share < kMost ? share : kMost;
  for (uint32_t base = warp * batch; base < n; base += warps * batch) {
    const uint32_t count = n - base < batch ? n - base : batch;
    for (uint32_t i = lane; i < count; i += 32u) pool.node[i] = base + i;
    __syncwarp();
    if (pool.probe.rounds == 8u)
      pool_permute<8>(pool, count, lane);
    else
      pool_permute<12>(pool, count, lane);
    __syncwarp();
    for (uint32_t i = lane; i - lane < count; i += 32u) {
      const uint32_t pi = i < count ? pool.node[i] : 0u;
      if (i < count && pi >= n_active) tab[(n + 31u) / 32u + pi - n_active] = base + i;
      const uint32_t word = __ballot_sync(0xffffffffu, (int32_t)probe_sign(pool.probe, pi) < 0);
      if (lane == 0) tab[(base + i) >> 5] = __brev(word);
    }
    __syncwarp();
  }
}

__device__ __forceinline__ ZTable table_reader(const uint32_t* tab, uint32_t n) {
  const uint32_t nwords = (n + 31u) / 32u;
  return ZTable{tab, tab[nwords], tab[nwords + 1]};
}

}  // namespace pw
