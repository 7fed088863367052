// Matching schedule of k-way refinement (Section 5, "K-Way Refinement:
// Matching Schedule").  The quotient graph Q has the blocks as vertices and
// an edge {i, j} when some hyperedge has pins in both V_i and V_j.  Block
// pairs are scheduled in rounds, each a maximal matching in the quotient
// edges not scheduled yet, the blocks of high remaining degree first, so
// that every block takes part in at most one two-way refinement at a time.
//
// k_quotient builds Q as k rows of KWP bit words from the edge bitmasks
// Lambda(e) (for every block i of Lambda(e), row i |= Lambda(e)), aggregated
// per thread block in shared memory.  k_schedule runs the rounds in one
// thread block: per round the blocks are ordered by (remaining degree at the
// round's start desc, id asc); each one still unmatched in its turn takes its
// unmatched remaining neighbour of the largest such degree (ties to the
// smaller id).
#include "jet_gain.cuh"
#include "jet_internal.cuh"

namespace jet {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// One row of KWP words from shared memory (rows are KWP-word aligned), read whole.
template <int KWP>
__device__ __forceinline__ void lds_row(const uint32_t *row, uint32_t (&R)[KWP]) {
  if constexpr (KWP == 1) {
    R[0] = *row;
  } else if constexpr (KWP == 2) {
    const uint2 x = *reinterpret_cast<const uint2 *>(row);
    R[0] = x.x; R[1] = x.y;
  } else {
#pragma unroll
    for (int h = 0; h < KWP / 4; ++h) {
      const uint4 x = reinterpret_cast<const uint4 *>(row)[h];
      R[4 * h] = x.x; R[4 * h + 1] = x.y; R[4 * h + 2] = x.z; R[4 * h + 3] = x.w;
    }
  }
}

// Bound by the reads of Lambda(e) (KWP of the 2 KWP words of every row, whose
// sectors come whole).  Most bits are set early on, so a block's row is read
// and compared first and the atomics are few.  The mask width is a template
// parameter: with a run-time width the row sat in local memory and the kernel
// took 133 us for 1.1 M edges at k = 128 (35 MB of rows).
template <int KWP>
__global__ void __launch_bounds__(256) k_quotient(const uint32_t *mask, int32_t m, int32_t k, uint32_t *q) {
  __shared__ __align__(16) uint32_t s_q[kMaxK * KWP];
  for (int x = threadIdx.x; x < k * KWP; x += blockDim.x) s_q[x] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  auto add_row = [&](int i, const uint32_t (&L)[KWP]) {  // row i |= L
    uint32_t *row = s_q + i * KWP;
    uint32_t R[KWP];
    lds_row<KWP>(row, R);
#pragma unroll
    for (int u = 0; u < KWP; ++u)
      if (L[u] & ~R[u]) atomicOr(&row[u], L[u]);
  };
  for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); e0 < m;
       e0 += (int64_t)gridDim.x * blockDim.x) {  // a warp's lanes go together
    const int64_t e = e0 + lane;
    uint32_t L[KWP], L2[KWP];
#pragma unroll
    for (int w = 0; w < KWP; ++w) L[w] = 0;
    if (e < m) load_rows<KWP>(mask + e * 2 * KWP, L, L2);
    int bits = 0;
#pragma unroll
    for (int w = 0; w < KWP; ++w) bits += __popc(L[w]);
    // a hyperedge inside one block links no pair; rows of many blocks (hubs) are left to the whole warp
    const bool wide = bits > 8;
    if (bits >= 2 && !wide) {
#pragma unroll
      for (int w = 0; w < KWP; ++w)
        for (uint32_t x = L[w]; x; x &= x - 1) add_row(w * 32 + __ffs(x) - 1, L);
    }
    for (unsigned bal = __ballot_sync(kFull, wide); bal; bal &= bal - 1) {
      uint32_t W[KWP];
#pragma unroll
      for (int w = 0; w < KWP; ++w) W[w] = __shfl_sync(kFull, L[w], __ffs(bal) - 1);
#pragma unroll
      for (int w = 0; w < KWP; ++w)
        if ((W[w] >> lane) & 1u) add_row(w * 32 + lane, W);
    }
  }
  __syncthreads();
  for (int x = threadIdx.x; x < k * KWP; x += blockDim.x)
    if (s_q[x]) atomicOr(&q[x], s_q[x]);
}

// The schedule by one thread block.  A round has k turns that depend on each
// other, so a turn has to be short; everything that does not depend on the
// turns runs beside them in parallel:
//   1. degrees; the rank of each block in the turn order (k comparisons per
//      block, kRankLanes lanes share a block);
//   2. the remaining graph with both ends renamed to ranks: row x of s_perm
//      holds the neighbours of the block of rank x, so "the unmatched
//      neighbour of largest degree, smallest id" is the lowest set bit of
//      row & unmatched;
//   3. the turns, by one warp, in registers: rows do not depend on the turns,
//      so their loads run ahead, and a turn is some eight dependent integer
//      instructions with no memory access, vote or branch on its path (the
//      partner leaves the unmatched set by its one-bit word; its index is
//      found beside the chain);
//   4. the matched pairs, in turn order, by all threads.
constexpr int kSchedThreads = 512;

template <int KWP>
__global__ void __launch_bounds__(kSchedThreads) k_schedule(const uint32_t *q, int32_t k, int32_t *pairs,
                                                            int32_t *round_of, int32_t *out_counts) {
  constexpr int kRankLanes = kSchedThreads / (32 * KWP) < 16 ? kSchedThreads / (32 * KWP) : 16;  // lanes per block
  constexpr int K = 32 * KWP;  // ranks; those of k.. and of blocks with no edge left have empty rows
  __shared__ __align__(16) uint32_t s_rem[K * KWP];
  __shared__ __align__(16) uint32_t s_perm[K * KWP];
  __shared__ int s_key[K];       // (K - degree) << 8 | id: ascending = turn order
  __shared__ int s_order[K];     // block of each rank
  __shared__ int s_pick[K];      // rank of the partner taken in turn x, or -1
  __shared__ int s_part[K / 32]; // pairs per 32 turns
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  for (int x = t; x < K * KWP; x += kSchedThreads) {
    const int j = x / KWP, w = x % KWP;
    uint32_t r = j < k ? q[x] : 0u;
    if (w == (j >> 5)) r &= ~(1u << (j & 31));  // no self pairs
    s_rem[x] = r;
  }
  __syncthreads();
  int np = 0, round = 0;
  for (;; ++round) {
    int deg = 0;
    if (t < K) {
#pragma unroll
      for (int w = 0; w < KWP; ++w) deg += __popc(s_rem[t * KWP + w]);
      s_key[t] = ((K - deg) << 8) | t;
    }
    const int live = __syncthreads_count(deg > 0);  // blocks with an edge left: the first `live` ranks
    if (live == 0) break;
    {
      const int j = t / kRankLanes, part = t % kRankLanes;
      int rank = 0, key = 0;
      if (j < K) {
        key = s_key[j];
#pragma unroll 8
        for (int i = part; i < K; i += kRankLanes) rank += s_key[i] < key;
      }
#pragma unroll
      for (int o = 1; o < kRankLanes; o <<= 1) rank += __shfl_xor_sync(kFull, rank, o);
      if (j < K && part == 0) s_order[rank] = j;
    }
    __syncthreads();
    {
      int ord[KWP];
#pragma unroll
      for (int w = 0; w < KWP; ++w) ord[w] = s_order[w * 32 + lane];
      for (int x = wid; x < live; x += kSchedThreads / 32) {
        const uint32_t *row = s_rem + s_order[x] * KWP;
        uint32_t mine = 0;
#pragma unroll
        for (int w = 0; w < KWP; ++w) {
          const uint32_t bal = __ballot_sync(kFull, (row[ord[w] >> 5] >> (ord[w] & 31)) & 1u);
          if (lane == w) mine = bal;
        }
        if (lane < KWP) s_perm[x * KWP + lane] = mine;
      }
    }
    __syncthreads();
    if (wid == 0) {
      uint32_t U[KWP];  // unmatched ranks
#pragma unroll
      for (int w = 0; w < KWP; ++w) U[w] = ~0u;
#pragma unroll
      for (int w0 = 0; w0 < KWP; ++w0) {
        if (w0 * 32 < live) {
#pragma unroll 8
          for (int i = 0; i < 32; ++i) {
            const int x = w0 * 32 + i;
            uint32_t R[KWP];
            lds_row<KWP>(s_perm + x * KWP, R);  // rows from `live` on are stale: masked below
            // the lowest set bit of row & unmatched, word by word: its own word's lowest bit, if the words below
            // have none
            const uint32_t turn = x < live ? 0u - ((U[w0] >> i) & 1u) : 0u;
            uint32_t take[KWP], low = 0;
#pragma unroll
            for (int w = 0; w < KWP; ++w) {
              const uint32_t c = R[w] & U[w];
              take[w] = low == 0 ? c & (0u - c) : 0u;
              low |= c;
            }
#pragma unroll
            for (int w = 0; w < KWP; ++w) {
              take[w] &= turn;
              U[w] ^= take[w];
            }
            U[w0] &= ~(1u << i);  // no later turn finds it: a neighbour still unmatched would have been taken
            int pick = -1;
#pragma unroll
            for (int w = 0; w < KWP; ++w)
              if (take[w]) pick = w * 32 + 31 - __clz(take[w]);
            if (lane == 0) s_pick[x] = pick;
          }
        } else {
          s_pick[w0 * 32 + lane] = -1;
        }
      }
    }
    __syncthreads();
    const int pick = t < K ? s_pick[t] : -1;
    const unsigned bal = __ballot_sync(kFull, pick >= 0);
    if (lane == 0 && t < K) s_part[wid] = __popc(bal);
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < K / 32; ++w) {
      before += w < wid ? s_part[w] : 0;
      total += s_part[w];
    }
    if (pick >= 0) {
      const int i = s_order[t], p = s_order[pick], at = np + before + __popc(bal & ((1u << lane) - 1));
      pairs[2 * at] = i;
      pairs[2 * at + 1] = p;
      round_of[at] = round;
      s_rem[i * KWP + (p >> 5)] &= ~(1u << (p & 31));  // a block is in one pair: its row has one writer
      s_rem[p * KWP + (i >> 5)] &= ~(1u << (i & 31));
    }
    np += total;
    __syncthreads();
  }
  if (t == 0) {
    out_counts[0] = np;
    out_counts[1] = round;
  }
}

template <int KWP>
void launch_schedule_kwp(jet_ctx *c, uint32_t *qbits, int32_t *pairs, int32_t *round_of, int32_t *counts) {
  if (c->m > 0) {
    k_quotient<KWP><<<grid_for(c->m, 256, c->launch_sms, 4), 256, 0, c->stream>>>(c->mask, c->m, c->k, qbits);
    ++c->kernel_launches;
  }
  k_schedule<KWP><<<1, kSchedThreads, 0, c->stream>>>(qbits, c->k, pairs, round_of, counts);
  ++c->kernel_launches;
}

}  // namespace

cudaError_t launch_quotient_schedule(jet_ctx *c, uint32_t *qbits, int32_t *pairs, int32_t *round_of,
                                     int32_t *counts) {
  cudaError_t e = cudaMemsetAsync(qbits, 0, sizeof(uint32_t) * c->k * c->kwp, c->stream);
  if (e != cudaSuccess) return e;
  switch (c->kwp) {
    case 1: launch_schedule_kwp<1>(c, qbits, pairs, round_of, counts); break;
    case 2: launch_schedule_kwp<2>(c, qbits, pairs, round_of, counts); break;
    case 4: launch_schedule_kwp<4>(c, qbits, pairs, round_of, counts); break;
    default: launch_schedule_kwp<8>(c, qbits, pairs, round_of, counts); break;
  }
  return cudaGetLastError();
}

}  // namespace jet
