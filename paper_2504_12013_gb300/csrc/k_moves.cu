// ApplyMoves (Algorithm 1), deterministic rebalancing rounds (Section 4.3),
// statistics and rollback moves.
//
// All updates are integer atomics whose final values do not depend on their
// order: phi row entries +-1, block weights and counts aggregated per thread
// block, and XOR toggles of the edge bitmasks at the phi crossings.
#include <algorithm>

#include "jet_internal.cuh"

namespace jet {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ void add_i64(long long *p, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long *>(p), static_cast<unsigned long long>(v));
}

struct MoveArgs {
  const int64_t *vptr;
  const int32_t *inc, *vwgt;
  int32_t *part, *phi;
  int64_t *bw;
  uint32_t *mask;
  const int32_t *mv_v;
  const uint32_t *mv_st;
  int32_t k, kwp;
  int graph;  // graph path: phi and the bitmasks are not kept, a move changes Pi and c(V_i) only
  int weights;  // c(V_i) and |V_i| are kept here (0: the kernel that made the list has done it)
  unsigned long long rebuild_min;  // from this many moves on, phi is counted anew (launch_apply_jet)
  Counters *cnt;
};

// A group of kMoveLanes lanes per move, the lanes striding over I(v): more
// loads and atomics in flight than one thread per move when the move list is
// short (rebalancing rounds).
constexpr int kMoveLanes = 8;

// The phi and bitmask updates of one move s -> t over the incidences j,
// j + kMoveLanes, ... below j1 (one lane's share of I(v)).  kMoveIlp
// incidences are loaded first and their atomics issued together, so that
// several atomics with return are in flight per lane before the first result
// is needed.
constexpr int kMoveIlp = 4;
// Grids of the apply kernels: this many waves of resident blocks.  The moves
// are dealt to blocks round-robin but their costs differ (degree, hub rows
// shared with other moves), and blocks that finish early take the next wave.
// A block with no move (or record) to take returns at once, so short move
// lists (late rebalancing rounds) do not pay for the large grid.
constexpr int kMoveWaves = 4;
constexpr int kRbMoveWaves = 4;  // the same for the rebalancing apply

__device__ __forceinline__ void move_incidences(const MoveArgs &a, int64_t j, int64_t j1, int s, int t) {
  const uint32_t sbit = 1u << (s & 31), tbit = 1u << (t & 31);
  for (; j < j1; j += kMoveIlp * kMoveLanes) {
    int64_t e[kMoveIlp];
#pragma unroll
    for (int q = 0; q < kMoveIlp; ++q) {
      const int64_t jj = j + q * kMoveLanes;
      e[q] = jj < j1 ? a.inc[jj] : -1;
    }
    int os[kMoveIlp], ot[kMoveIlp];
#pragma unroll
    for (int q = 0; q < kMoveIlp; ++q) {
      os[q] = 0;  // no crossing for an absent incidence
      ot[q] = 2;
      if (e[q] >= 0) {
        os[q] = atomicSub(&a.phi[e[q] * a.k + s], 1);  // os -> os - 1
        ot[q] = atomicAdd(&a.phi[e[q] * a.k + t], 1);  // ot -> ot + 1
      }
    }
#pragma unroll
    for (int q = 0; q < kMoveIlp; ++q) {
      if (e[q] < 0) continue;
      uint32_t *row = a.mask + e[q] * 2 * a.kwp;
      if (os[q] == 1) atomicXor(&row[s >> 5], sbit);           // 1 -> 0
      if (os[q] == 2) atomicXor(&row[a.kwp + (s >> 5)], sbit);  // 2 -> 1
      if (ot[q] == 0) atomicXor(&row[t >> 5], tbit);           // 0 -> 1
      if (ot[q] == 1) atomicXor(&row[a.kwp + (t >> 5)], tbit);  // 1 -> 2
    }
  }
}

// ---------------------------------------------------------------- rebalancing
// Selection of the minimal prefix per overloaded block (Section 4.3) as a
// radix select over all records at once.  Every vertex v of an overloaded
// block with a valid target has a record with the key
// K(v) = hi(v) << vb | v  (priority descending, then id ascending, as one
// ascending number of hb + vb bits; 64-bit when it fits, else 128-bit).
// Per level (rb_digit <= kRbMaxDigit = 11 bits, from the top, so a pick scans
// at most 2048 bins per block; three levels cover keys of up to 33 bits) a
// grid-wide pass adds c(v) of every record that matches its
// block's fixed prefix into the (block, digit) histogram -- for the first
// level the target kernels do this while they write the records -- and one
// small kernel per overloaded block picks the digit at which the cumulative
// weight reaches the excess.  After the last level the prefix is the
// threshold key, and every record up to it moves.
typedef unsigned __int128 u128;
constexpr int kPickThreads = 256;

struct RbArgs {
  const int64_t *bw;
  RbBlock *rbb;
  const RbRec *rec;              // segmented records
  int32_t *cur;                  // records of each block (kCurStride apart)
  const uint64_t *rb_hi;
  const int32_t *rb_v, *rb_ct;  // record: vertex; c << 16 | block << 8 | target
  unsigned long long *hist;
  int32_t *mv_v;
  uint32_t *mv_st;
  int32_t n, k;
  int segments;
  int vbits, tbits;
  int digit, bins;               // radix-select digit width and bins per block row
  long long Lmax, dz_min;
  int32_t max_rounds;
  Counters *cnt;
};

// Exclusive prefix sum of x over the kMaxK threads of the block (every thread calls it).
__device__ __forceinline__ int segment_base(int x) {
  __shared__ int s_w[kMaxK / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_w[wid] = incl;
  __syncthreads();
  int before = 0;
#pragma unroll
  for (int w = 0; w < kMaxK / 32; ++w) before += w < wid ? s_w[w] : 0;
  return before + incl - x;
}

// Per-block state of the next round: overloaded flag, excess, target
// capacity (deadzone and L_max), cleared selection state and counters.  One
// block of kMaxK threads, thread b for block b.
__device__ __forceinline__ void rb_prep_blocks(const RbArgs &a) {
  const int b = threadIdx.x;
  const long long bwb = b < a.k ? __ldcg(&a.bw[b]) : 0;
  const int room = bwb > a.Lmax ? __ldcg(&a.cnt->vcount[b]) : 0;
  const int base = segment_base(room);
  if (b < a.k) {
    RbBlock r;
    r.bw = bwb;
    r.over = bwb > a.Lmax ? 1 : 0;
    r.excess = r.over ? bwb - a.Lmax : 0;
    r.cap = (r.over || bwb >= a.dz_min) ? -1 : a.Lmax - bwb;
    r.before = 0;
    r.pre_hi = 0;
    r.pre_lo = 0;
    r.all = 0;
    r.room = room;
    r.base = base;
    a.rbb[b] = r;
    a.cur[b * kCurStride] = 0;
  }
  if (b == 0) {
    // segmented: an apply that reads the count may be running beside this; the target kernels reset it
    if (!a.segments) a.cnt->n_moves = 0;
    a.cnt->n_rec = 0;
  }
}

// Any block above L_max?  If so, the state of the first round.  In a CUDA
// graph (use_cond) it also sets the condition of the rebalancing WHILE node.
__device__ __forceinline__ void rb_check(const RbArgs &a, cudaGraphConditionalHandle cond, int use_cond) {
  const int b = threadIdx.x;
  const bool over = b < a.k && __ldcg(&a.bw[b]) > a.Lmax;
  const int any = __syncthreads_or(over);
  if (b == 0) {
    a.cnt->rb_any = any;
    a.cnt->rb_done = !any;
    if (use_cond) cudaGraphSetConditional(cond, (any && a.max_rounds > 0) ? 1u : 0u);
  }
  if (any) rb_prep_blocks(a);
}

__global__ void k_rb_check(RbArgs a, cudaGraphConditionalHandle cond, int use_cond) { rb_check(a, cond, use_cond); }

// End of a round: count it, and stop if nothing moved, nothing is overloaded
// any more, or the round cap is reached; otherwise the state of the next round.
__device__ __forceinline__ void rb_post(const RbArgs &a, cudaGraphConditionalHandle cond, int use_cond) {
  __shared__ int s_done;
  const int b = threadIdx.x;
  const bool over = b < a.k && __ldcg(&a.bw[b]) > a.Lmax;
  const int any = __syncthreads_or(over);
  if (b == 0) {
    const long long moved = (long long)__ldcg(&a.cnt->n_moves);
    a.cnt->rb_rounds += 1;
    a.cnt->rb_moves += moved;
    a.cnt->rb_any = any;
    const int done = (moved == 0) || !any || (a.cnt->rb_rounds >= a.max_rounds);
    a.cnt->rb_done = done;
    s_done = done;
    if (use_cond) cudaGraphSetConditional(cond, done ? 0u : 1u);
  }
  __syncthreads();
  if (!s_done) rb_prep_blocks(a);
}

__global__ void k_rb_post(RbArgs a, cudaGraphConditionalHandle cond, int use_cond) { rb_post(a, cond, use_cond); }

// Pi(v) <- t and phi_e[s]--, phi_e[t]++ for every e in I(v); c(V_s), c(V_t)
// and |V_s|, |V_t| through shared-memory partial sums; and both bitmasks of
// every touched edge, exactly, without a second pass: the atomic updates of
// one phi entry are serialized in some order, so its 0 <-> 1 crossings (and
// 1 <-> 2 crossings) alternate, and the final bit is the initial bit XOR the
// parity of the crossings.  Each thread whose own atomic crosses toggles the
// bit with atomicXor; XOR commutes, so the order of the toggles is irrelevant.
__global__ void __launch_bounds__(256) k_apply(MoveArgs a) {
  __shared__ long long s_dw[kMaxK];
  __shared__ int s_dc[kMaxK];
  const long long nm = (long long)a.cnt->n_moves;
  if ((long long)blockIdx.x * (blockDim.x / kMoveLanes) >= nm) return;  // no move for this block
  if ((unsigned long long)nm >= a.rebuild_min) return;                  // k_apply_part's
  for (int b = threadIdx.x; b < a.k; b += blockDim.x) { s_dw[b] = 0; s_dc[b] = 0; }
  __syncthreads();
  unsigned long long pins = 0;  // incidences moved by this thread's moves (work count)
  const int sub = threadIdx.x % kMoveLanes;
  const long long g0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kMoveLanes;
  const long long ng = ((long long)gridDim.x * blockDim.x) / kMoveLanes;
  for (long long i = g0; i < nm; i += ng) {
    const int v = a.mv_v[i];
    const uint32_t st = a.mv_st[i];
    const int s = st & 0xffff, t = st >> 16;
    if (sub == 0) {
      a.part[v] = t;
      if (a.weights) {
        const int c = a.vwgt[v];
        atomicAdd(reinterpret_cast<unsigned long long *>(&s_dw[s]), (unsigned long long)(-(long long)c));
        atomicAdd(reinterpret_cast<unsigned long long *>(&s_dw[t]), (unsigned long long)c);
        atomicSub(&s_dc[s], 1);
        atomicAdd(&s_dc[t], 1);
      }
    }
    const int64_t j1 = a.vptr[v + 1];
    if (sub == 0) pins += (unsigned long long)(j1 - a.vptr[v]);
    move_incidences(a, a.vptr[v] + sub, j1, s, t);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pins += __shfl_xor_sync(kFull, pins, o);
  __shared__ unsigned long long s_pins;
  if (threadIdx.x == 0) s_pins = 0;
  __syncthreads();
  if ((threadIdx.x & 31) == 0 && pins) atomicAdd(&s_pins, pins);
  __syncthreads();
  if (threadIdx.x == 0 && s_pins) atomicAdd(&a.cnt->w_apply_pins, s_pins);
  for (int b = threadIdx.x; b < a.k; b += blockDim.x) {
    if (s_dw[b]) add_i64(reinterpret_cast<long long *>(&a.bw[b]), s_dw[b]);
    if (s_dc[b]) atomicAdd(&a.cnt->vcount[b], s_dc[b]);
  }
}

// The moves' share of the partition and the block weights only, a thread per
// move: on the graph path, and where phi is counted anew afterwards
// (rebuild_min moves or more).  k_apply's eight lanes per move left seven idle
// here: 119 us for the 1.7 M moves of a graph's first iteration.
__global__ void __launch_bounds__(256) k_apply_part(MoveArgs a) {
  __shared__ long long s_dw[kMaxK];
  __shared__ int s_dc[kMaxK];
  __shared__ unsigned long long s_pins;
  const long long nm = (long long)a.cnt->n_moves;
  if ((long long)blockIdx.x * blockDim.x >= nm || (unsigned long long)nm < a.rebuild_min) return;
  for (int b = threadIdx.x; b < a.k; b += blockDim.x) { s_dw[b] = 0; s_dc[b] = 0; }
  if (threadIdx.x == 0) s_pins = 0;
  __syncthreads();
  unsigned long long pins = 0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < nm; i0 += 2 * stride) {
    int v[2], c[2];
    uint32_t st[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      v[q] = i0 + q * stride < nm ? a.mv_v[i0 + q * stride] : -1;
      st[q] = i0 + q * stride < nm ? a.mv_st[i0 + q * stride] : 0;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      c[q] = 0;
      if (v[q] < 0) continue;
      if (a.weights) c[q] = a.vwgt[v[q]];
      pins += (unsigned long long)(a.vptr[v[q] + 1] - a.vptr[v[q]]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (v[q] < 0) continue;
      const int s = st[q] & 0xffff, t = st[q] >> 16;
      a.part[v[q]] = t;
      if (!a.weights) continue;
      atomicAdd(reinterpret_cast<unsigned long long *>(&s_dw[s]), (unsigned long long)(-(long long)c[q]));
      atomicAdd(reinterpret_cast<unsigned long long *>(&s_dw[t]), (unsigned long long)c[q]);
      atomicSub(&s_dc[s], 1);
      atomicAdd(&s_dc[t], 1);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pins += __shfl_xor_sync(kFull, pins, o);
  if ((threadIdx.x & 31) == 0 && pins) atomicAdd(&s_pins, pins);
  __syncthreads();
  if (threadIdx.x == 0 && s_pins) atomicAdd(&a.cnt->w_apply_pins, s_pins);
  for (int b = threadIdx.x; b < a.k; b += blockDim.x) {
    if (s_dw[b]) add_i64(reinterpret_cast<long long *>(&a.bw[b]), s_dw[b]);
    if (s_dc[b]) atomicAdd(&a.cnt->vcount[b], s_dc[b]);
  }
}

template <class KT>
__device__ __forceinline__ KT rb_full_key(uint64_t hi, int v, int vbits) {
  return ((KT)hi << vbits) | (KT)(uint32_t)v;
}

template <class KT>
__device__ __forceinline__ KT rb_prefix(const RbBlock &r) {
  if constexpr (sizeof(KT) > 8) return ((KT)r.pre_hi << 64) | (KT)r.pre_lo;
  else return (KT)r.pre_lo;
}

// One level: digit = bits [lo, lo + w) of K(v) for the records whose higher bits
// equal their block's prefix; one atomic per matching record.
template <class KT>
__global__ void __launch_bounds__(256) k_rb_level(RbArgs a, int lo, int w) {
  const int up = lo + w;
  const KT dmask = ((KT)1 << w) - 1;
  const long long nrec = (long long)a.cnt->n_rec;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < nrec; base += (long long)gridDim.x * blockDim.x) {
    const long long i = base + threadIdx.x;
    bool m = false;
    int b = 0, d = 0;
    unsigned c = 0;
    if (i < nrec) {
      const int32_t ct = a.rb_ct[i];
      b = (ct >> 8) & 255;
      const RbBlock &r = a.rbb[b];
      if (!r.all) {
        const KT K = rb_full_key<KT>(a.rb_hi[i], a.rb_v[i], a.vbits);
        m = up >= a.tbits || (K >> up) == (rb_prefix<KT>(r) >> up);
        d = (int)((K >> lo) & dmask);
        c = (unsigned)(ct >> 16);
      }
    }
    if (m) atomicAdd(&a.hist[(int64_t)b * a.bins + d], (unsigned long long)c);
  }
}

// Per overloaded block: the digit at which the cumulative weight first reaches
// the excess; at the first level a total below the excess selects everything.
// Warp w owns a contiguous segment of bins and reads it 32 bins at a time
// (coalesced); the warp whose segment holds the threshold walks it again.
// Leaves the histogram row zeroed.  Bound by latency: eight bins per lane in
// flight at 256 threads and 11-bit digits, and short chains behind the barrier.
// 1,024 threads with two bins each took 8.53 against 8.46 ms for eight
// iterations of a graph of 4 M vertices at k = 64, 7.89 against 7.80 on 2 M VLSI
// vertices.
__global__ void __launch_bounds__(kPickThreads) k_rb_pick(RbArgs a, int lo, int first) {
  constexpr int kWarps = kPickThreads / 32;
  const int b = blockIdx.x;
  RbBlock *r = &a.rbb[b];
  if (!r->over || r->all) return;
  __shared__ long long s_warp[kWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int seg = (a.bins + kWarps - 1) / kWarps;
  const int x0 = wid * seg < a.bins ? wid * seg : a.bins;
  const int x1 = x0 + seg < a.bins ? x0 + seg : a.bins;
  unsigned long long *row = a.hist + (int64_t)b * a.bins;
  long long part = 0;
#pragma unroll 8
  for (int x = x0 + lane; x < x1; x += 32) part += (long long)row[x];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(kFull, part, o);
  if (lane == 0) s_warp[wid] = part;
  // read before the barrier: the threshold warp rewrites r->before below
  const long long before = r->before, need = r->excess;
  __syncthreads();
  long long excl = 0, total = 0;
  for (int i = 0; i < kWarps; ++i) {
    if (i < wid) excl += s_warp[i];
    total += s_warp[i];
  }
  if (first && total < need) {
    if (threadIdx.x == 0) r->all = 1;
  } else if (before + excl < need && before + excl + part >= need) {  // warp-uniform
    long long run = before + excl;
    for (int x = x0; x < x1; x += 32) {
      const long long w = x + lane < x1 ? (long long)row[x + lane] : 0;
      long long incl = w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      const unsigned hit = __ballot_sync(kFull, run + incl >= need);
      if (hit) {
        const int l = __ffs(hit) - 1;
        const long long prev = __shfl_sync(kFull, incl - w, l);
        if (lane == 0) {
          r->before = run + prev;
          const u128 pre = (((u128)r->pre_hi << 64) | r->pre_lo) | ((u128)(unsigned)(x + l) << lo);
          r->pre_hi = (unsigned long long)(pre >> 64);
          r->pre_lo = (unsigned long long)pre;
        }
        break;
      }
      run += __shfl_sync(kFull, incl, 31);
    }
  }
  __syncthreads();  // the threshold walk above reads the row
  for (int x = x0 + lane; x < x1; x += 32) row[x] = 0ull;
}

// Segmented form: one thread block per overloaded block of the partition does
// the whole selection of a round in one launch.  The target kernels have put
// the block's records into a segment of their own; each thread holds kSelHeld
// of them in registers (any beyond are read again per level).  Per 8-bit
// digit the block histograms its records in shared memory and every warp
// picks the digit by itself, so a level has two barriers; after the last digit
// the records up to the threshold go to the move list, which k_apply works
// through.  Bound by the latency of the loads and levels.  A round's selection
// was 2 x levels - 1 dependent launches whatever the number of records, and
// the apply kernel looked at every record again: 1.03 -> 0.31 ms for the 26
// rounds of 300k vertices at k = 200.  (Moving the selected records here, and
// not through the list, saves a launch and leaves most of the GPU idle: the
// four iterations of that case took 3.08 against 2.58 ms.)  The line (kSegVertices, on average):
// beyond a segment that fits the registers of one block, the grid-wide passes
// are as fast.  Measured per round on 31k vertices per block: they take 34 us
// at k = 128; clusters of 4 to 16 blocks per segment that sum their histograms
// over distributed shared memory took 33 to 61, and the target kernels lose
// more to the segments' cursors than that gives.
constexpr int kSelThreads = 512;
constexpr int kSelHeld = 8;  // records per thread held in registers
constexpr int kSelBins = 1 << kSelBits;
static_assert(kSelThreads * kSelHeld == kSegVertices, "a segment of average size fits the registers");

template <class T>
__device__ __forceinline__ T warp_incl(T x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// A record in registers; the priority part of a 64-bit key is compact (below 2^32).
template <class KT>
struct SelRec {
  uint32_t hi = 0;
  int32_t v = 0, ct = 0;
  SelRec() = default;
  __device__ __forceinline__ explicit SelRec(const RbRec &r) : hi((uint32_t)r.hi), v(r.v), ct(r.ct) {}
};
template <>
struct SelRec<u128> {
  unsigned long long hi = 0;
  int32_t v = 0, ct = 0;
  SelRec() = default;
  __device__ __forceinline__ explicit SelRec(const RbRec &r) : hi(r.hi), v(r.v), ct(r.ct) {}
};

// Segments of more than kSelLarge records go to a cluster of kSelCluster thread
// blocks, each with its share of the records and a histogram of its own; the
// sums over the cluster go through distributed shared memory.  A partition may
// have a block of nearly all vertices (a seed partition, or the round after
// many small blocks moved to one).  Bound by the reads of the records, once
// per level beyond those in registers: jet_rebalance with every vertex in one
// block, 32 rounds, took 49.1 ms by one thread block at n = 100,003, k = 37
// (most of it 64-bit shared-memory atomics on the one target's weight) and
// 54.9 ms at n = 1,000,000, k = 256; so 1.93 and 16.5 ms (grid-wide passes:
// 2.52 and 20.7).  The line: up to it one block reads the records beyond its
// registers in about the time of the grid-wide passes (20,000 vertices in one
// block, k = 8: 0.38 against 0.47 ms), and clusters lose to them where every
// block of the partition is that large (above).
constexpr int kSelCluster = 8;
constexpr int kSelLarge = 16384;
constexpr int kSelGroups = 8;  // clusters for large segments, at most

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// *p of the cluster's block `rank`.
template <class T>
__device__ __forceinline__ T ld_cluster(const T *p, int rank) {
  uint32_t at = (uint32_t)__cvta_generic_to_shared(p);
  asm("mapa.shared::cluster.u32 %0, %0, %1;\n" : "+r"(at) : "r"(rank));
  T x;
  if constexpr (sizeof(T) == 4) asm volatile("ld.shared::cluster.u32 %0, [%1];\n" : "=r"(x) : "r"(at) : "memory");
  else asm volatile("ld.shared::cluster.u64 %0, [%1];\n" : "=l"(x) : "r"(at) : "memory");
  return x;
}

// The selection of block b's segment by one thread block, or (CLUSTER) by all of a cluster.
// WT: unsigned when c(V) < 2^32 (no sum of weights leaves it), else unsigned long long.
template <class KT, class WT, bool CLUSTER>
__device__ __forceinline__ void select_segment(const RbArgs &a, int64_t *bw, int b, int rank) {
  typedef SelRec<KT> Rec;
  constexpr int kPer = kSelBins / 32;  // bins per lane
  constexpr int T = kSelThreads * (CLUSTER ? kSelCluster : 1);
  __shared__ __align__(16) WT s_hist[2][kSelBins];
  __shared__ __align__(16) WT s_sum[CLUSTER ? kSelBins : 1];
  // weight and vertices that move to each block.  64-bit shared-memory atomics are retried until they win, and many
  // records may go to one block; where block weights are kept here (at most kEarlyVertices), c(V) < 2^32
  __shared__ WT s_dw[kMaxK];
  __shared__ int s_dc[kMaxK];
  const int t = threadIdx.x, lane = t & 31, tc = rank * kSelThreads + t;  // tc: thread of the cluster
  const RbBlock &blk = a.rbb[b];
  const int room = blk.room, count = a.cur[b * kCurStride];
  const WT excess = (WT)blk.excess;
  const RbRec *rec = a.rec + blk.base;
  const int cnt = min(count, room);
  Rec held[kSelHeld];  // weight 0: no record
#pragma unroll
  for (int q = 0; q < kSelHeld; ++q) held[q] = tc + q * T < cnt ? Rec(rec[tc + q * T]) : Rec();
  if (t < kSelBins) s_hist[0][t] = s_hist[1][t] = 0;
  if (t < kMaxK) {
    s_dw[t] = 0;
    s_dc[t] = 0;
  }
  __syncthreads();
  KT pre = 0;  // the fixed digits of the threshold key
  WT before = 0;
  bool all = false;
  int buf = 0;
  for (int up = a.tbits; up > 0; buf ^= 1) {
    const int lo = up > kSelBits ? up - kSelBits : 0;
    const unsigned dmask = (1u << (up - lo)) - 1;
    auto add = [&](const Rec &r) {
      const KT K = rb_full_key<KT>(r.hi, r.v, a.vbits);
      const WT c = (WT)(unsigned)(r.ct >> 16);
      if (c && (up >= a.tbits || (K >> up) == (pre >> up))) atomicAdd(&s_hist[buf][(unsigned)(K >> lo) & dmask], c);
    };
#pragma unroll
    for (int q = 0; q < kSelHeld; ++q)
      if (q * T < cnt) add(held[q]);
    for (int i = tc + kSelHeld * T; i < cnt; i += 4 * T) {
      Rec r[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) r[q] = i + q * T < cnt ? Rec(rec[i + q * T]) : Rec();
#pragma unroll
      for (int q = 0; q < 4; ++q) add(r[q]);
    }
    if constexpr (CLUSTER) {
      cluster_sync();
      if (t < kSelBins) {
        WT x = 0;
#pragma unroll
        for (int r = 0; r < kSelCluster; ++r) x += ld_cluster(&s_hist[buf][t], r);
        s_sum[t] = x;
      }
    }
    if (!CLUSTER) __syncthreads();
    if (t < kSelBins) s_hist[buf ^ 1][t] = 0;  // read a level ago (by the cluster: before the barrier)
    if (CLUSTER) __syncthreads();
    const WT *sum = (CLUSTER ? s_sum : s_hist[buf]) + lane * kPer;
    WT w[kPer], mine = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      w[q] = sum[q];
      mine += w[q];
    }
    const WT incl = warp_incl(mine);
    if (up >= a.tbits && __shfl_sync(kFull, incl, 31) < excess) {  // every record moves
      all = true;
      break;
    }
    // the lane whose bins reach the excess, and the bin
    WT run = before + incl - mine;
    const unsigned hit = __ballot_sync(kFull, run < excess && run + mine >= excess);
    int digit = lane * kPer;
    bool more = true;
#pragma unroll
    for (int q = 0; q < kPer - 1; ++q) {
      more = more && run + w[q] < excess;
      if (more) {
        run += w[q];
        ++digit;
      }
    }
    const int src = hit ? __ffs(hit) - 1 : 0;
    before = __shfl_sync(kFull, run, src);
    pre |= (KT)(unsigned)__shfl_sync(kFull, digit, src) << lo;
    up = lo;
    if (up > 0 && !CLUSTER) __syncthreads();  // the cleared buffer is added to next
  }
  // the records up to the threshold: one atomic per warp (and batch) on the move list
  auto emit = [&](const Rec *r, int n) {
    unsigned bal[kSelHeld], tot = 0;
#pragma unroll
    for (int q = 0; q < kSelHeld; ++q) {
      bal[q] = 0;
      if (q < n) {
        const bool sel = (r[q].ct >> 16) && (all || rb_full_key<KT>(r[q].hi, r[q].v, a.vbits) <= pre);
        bal[q] = __ballot_sync(kFull, sel);
        tot += __popc(bal[q]);
      }
    }
    if (!tot) return;
    unsigned long long at = 0;
    if (lane == 0) at = atomicAdd(&a.cnt->n_moves, (unsigned long long)tot);
    at = __shfl_sync(kFull, at, 0);
#pragma unroll
    for (int q = 0; q < kSelHeld; ++q) {
      if (q < n) {
        if ((bal[q] >> lane) & 1u) {
          const unsigned long long x = at + __popc(bal[q] & ((1u << lane) - 1));
          const int to = r[q].ct & 255;
          a.mv_v[x] = r[q].v;
          a.mv_st[x] = (uint32_t)b | ((uint32_t)to << 16);
          if (bw) {
            atomicAdd(&s_dw[to], (WT)(unsigned)(r[q].ct >> 16));
            atomicAdd(&s_dc[to], 1);
          }
        }
        at += __popc(bal[q]);
      }
    }
  };
  emit(held, kSelHeld);
  // the warp's lanes go together, from its first record
  for (int i = tc + kSelHeld * T, iw = i - lane; iw < cnt; i += 4 * T, iw += 4 * T) {
    Rec r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) r[q] = i + q * T < cnt ? Rec(rec[i + q * T]) : Rec();
    emit(r, 4);
  }
  if (bw) {
    __syncthreads();
    // the block weights already, so that the end of the round need not wait for the apply
    if (t < kMaxK) {
      long long dw = (long long)s_dw[t];
      int dc = s_dc[t];
      if (dc) {
        add_i64(reinterpret_cast<long long *>(&bw[t]), dw);
        atomicAdd(&a.cnt->vcount[t], dc);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dw += __shfl_xor_sync(kFull, dw, o);
      dc = __reduce_add_sync(kFull, dc);
      if (lane == 0 && dc) {
        add_i64(reinterpret_cast<long long *>(&bw[b]), -dw);
        atomicSub(&a.cnt->vcount[b], dc);
      }
    }
  }
  if (CLUSTER) cluster_sync();  // no block leaves or clears a histogram that another still reads
}

// A thread block per block of the partition; LARGE (a segment may be large): the blocks from `first` on are clusters
// that take the large segments in turn.
template <class KT, class WT, bool LARGE>
__global__ void __launch_bounds__(kSelThreads, 2) k_rb_select(RbArgs a, int64_t *bw, int first, int groups) {
  const int b = blockIdx.x;
  if (!LARGE || b < first) {
    if (b < a.k && a.rbb[b].over && (!LARGE || a.rbb[b].room <= kSelLarge))
      select_segment<KT, WT, false>(a, bw, b, 0);
    return;
  }
  if constexpr (LARGE) {
    __shared__ int s_list[kMaxK / 32], s_which;
    const int t = threadIdx.x, lane = t & 31;
    const bool large = t < a.k && a.rbb[t].over && a.rbb[t].room > kSelLarge;
    const unsigned bal = __ballot_sync(kFull, large);
    if (lane == 0 && t < kMaxK) s_list[t >> 5] = bal;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kMaxK / 32; ++w) {
      before += w < (t >> 5) ? __popc(s_list[w]) : 0;
      total += __popc(s_list[w]);
    }
    before += __popc(bal & ((1u << lane) - 1));
    const int group = (b - first) / kSelCluster, rank = (b - first) % kSelCluster;
    for (int i = group; i < total; i += groups) {  // the same in every block of the cluster
      if (large && before == i) s_which = t;
      __syncthreads();
      select_segment<KT, WT, true>(a, bw, s_which, rank);
    }
  }
}

__global__ void __launch_bounds__(256) k_count_blocks(const int32_t *part, int32_t n, int32_t k, Counters *cnt) {
  __shared__ int s_c[kMaxK];
  s_c[threadIdx.x] = 0;  // kMaxK = blockDim.x
  __syncthreads();
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int b = part[v];
    if ((unsigned)b < (unsigned)k) atomicAdd(&s_c[b], 1);
  }
  __syncthreads();
  if (s_c[threadIdx.x]) atomicAdd(&cnt->vcount[threadIdx.x], s_c[threadIdx.x]);
}

// Apply the selection: every record with K(v) <= its block's threshold (or of
// an `all` block) moves v to its target.  A warp tests 32 records (one per
// lane) and then applies the selected ones four at a time, kMoveLanes lanes
// per move striding over I(v) as k_apply does; the moves are counted for the
// round's statistics.
template <class KT>
__global__ void __launch_bounds__(256) k_rb_apply(RbArgs r, MoveArgs a) {
  __shared__ long long s_dw[kMaxK];
  __shared__ int s_dc[kMaxK];
  __shared__ unsigned long long s_moves, s_pins;
  const long long nrec = (long long)r.cnt->n_rec;
  if ((long long)blockIdx.x * blockDim.x >= nrec) return;  // no record for this block
  for (int b = threadIdx.x; b < a.k; b += blockDim.x) { s_dw[b] = 0; s_dc[b] = 0; }
  if (threadIdx.x == 0) { s_moves = 0; s_pins = 0; }
  __syncthreads();
  unsigned long long moves = 0, pins = 0;
  const int lane = threadIdx.x & 31, grp = lane / kMoveLanes, sub = lane % kMoveLanes;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long base = w0 * 32; base < nrec; base += nw * 32) {
    const long long i = base + lane;
    bool sel = false;
    int v = 0;
    int32_t ct = 0;
    if (i < nrec) {
      ct = r.rb_ct[i];
      v = r.rb_v[i];
      const RbBlock &rb = r.rbb[(ct >> 8) & 255];
      KT pre;
      if constexpr (sizeof(KT) > 8) pre = ((KT)rb.pre_hi << 64) | (KT)rb.pre_lo;
      else pre = (KT)rb.pre_lo;
      sel = rb.all || rb_full_key<KT>(r.rb_hi[i], v, r.vbits) <= pre;
    }
    unsigned bal = __ballot_sync(kFull, sel);
    while (bal) {
      const int nsel = __popc(bal);
      const int src = grp < nsel ? (int)__fns(bal, 0, grp + 1) : -1;  // this group's record lane
      const int mv = __shfl_sync(kFull, v, src < 0 ? 0 : src);
      const int32_t mct = __shfl_sync(kFull, ct, src < 0 ? 0 : src);
      if (src >= 0) {
        const int s = (mct >> 8) & 255, t = mct & 255;
        const int64_t j0 = a.vptr[mv], j1 = a.vptr[mv + 1];
        if (sub == 0) {
          a.part[mv] = t;
          const int c = (mct >> 16) & 0xffff;
          atomicAdd(reinterpret_cast<unsigned long long *>(&s_dw[s]), (unsigned long long)(-(long long)c));
          atomicAdd(reinterpret_cast<unsigned long long *>(&s_dw[t]), (unsigned long long)c);
          atomicSub(&s_dc[s], 1);
          atomicAdd(&s_dc[t], 1);
          ++moves;
          pins += (unsigned long long)(j1 - j0);
        }
        if (!a.graph) move_incidences(a, j0 + sub, j1, s, t);
      }
      // drop the (up to) 32 / kMoveLanes records just applied
      for (int q = 0; q < 32 / kMoveLanes && bal; ++q) bal &= bal - 1;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    moves += __shfl_xor_sync(kFull, moves, o);
    pins += __shfl_xor_sync(kFull, pins, o);
  }
  if (lane == 0) {
    if (moves) atomicAdd(&s_moves, moves);
    if (pins) atomicAdd(&s_pins, pins);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_moves) atomicAdd(&r.cnt->n_moves, s_moves);
    if (s_pins) atomicAdd(&r.cnt->w_apply_pins, s_pins);
  }
  for (int b = threadIdx.x; b < a.k; b += blockDim.x) {
    if (s_dw[b]) add_i64(reinterpret_cast<long long *>(&a.bw[b]), s_dw[b]);
    if (s_dc[b]) atomicAdd(&a.cnt->vcount[b], s_dc[b]);
  }
}

// Moves that take part back to best (rollback at the end of a phase).
__global__ void __launch_bounds__(256) k_rollback_moves(const int32_t *part, const int32_t *best, int32_t n,
                                                        int32_t *mv_v, uint32_t *mv_st, Counters *cnt,
                                                        const int *enable) {
  __shared__ unsigned s_wc[8];
  __shared__ unsigned long long s_base;
  if (enable && !*enable) return;  // uniform: no snapshot to roll back to
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = base + threadIdx.x;
    int s = 0, t = 0;
    bool mv = false;
    if (v < n) {
      s = part[v];
      t = best[v];
      mv = s != t && (unsigned)s < kMaxK && (unsigned)t < kMaxK;
    }
    const unsigned long long pos = block_append(mv, &cnt->n_moves, s_wc, &s_base);
    if (mv) {
      mv_v[pos] = (int32_t)v;
      mv_st[pos] = (uint32_t)s | ((uint32_t)t << 16);
    }
  }
}

MoveArgs move_args(jet_ctx *c, int32_t *part, int32_t *phi, int64_t *block_w) {
  MoveArgs a{};
  a.vptr = c->vptr;
  a.inc = c->inc;
  a.vwgt = c->vwgt;
  a.part = part;
  a.phi = phi;
  a.bw = block_w;
  a.mask = c->mask;
  a.graph = c->graph_path;
  a.rebuild_min = c->graph_path ? 0 : ~0ull;
  a.weights = 1;
  a.mv_v = c->mv_v;
  a.mv_st = c->mv_st;
  a.k = c->k;
  a.kwp = c->kwp;
  a.cnt = c->cnt;
  return a;
}

RbArgs rb_args(jet_ctx *c, const int64_t *block_w) {
  RbArgs a{};
  a.bw = block_w;
  a.rbb = c->rbb;
  a.segments = c->rb_segments;
  a.rec = c->rb_rec;
  a.cur = c->rb_cur;
  a.rb_hi = c->rb_hi;
  a.rb_v = c->rb_v;
  a.rb_ct = c->rb_ct;
  a.hist = c->rb_hist;
  a.mv_v = c->mv_v;
  a.mv_st = c->mv_st;
  a.n = c->n;
  a.k = c->k;
  a.vbits = c->rb_vbits;
  a.tbits = c->rb_hbits + c->rb_vbits;
  a.digit = c->rb_digit;
  a.bins = 1 << c->rb_digit;
  a.Lmax = c->Lmax;
  a.dz_min = c->dz_min;
  a.max_rounds = c->params.max_rebalance_rounds;
  a.cnt = c->cnt;
  return a;
}

}  // namespace

cudaError_t prepare_move_kernels(jet_ctx *c) {
  c->rb_segments = c->n / c->k <= kSegVertices ? 1 : 0;
  c->rb_early = c->rb_segments && c->n <= kEarlyVertices ? 1 : 0;
  cudaError_t e = resident_blocks(k_apply, 256, 0, &c->move_bps[0]);
  if (e == cudaSuccess) e = resident_blocks(k_rb_apply<unsigned long long>, 256, 0, &c->move_bps[1]);
  if (e == cudaSuccess) e = resident_blocks(k_rb_apply<u128>, 256, 0, &c->move_bps[2]);
  return e;
}

static cudaError_t apply_phi(jet_ctx *c, const MoveArgs &a) {
  k_apply<<<grid_for((int64_t)c->n * kMoveLanes, 256, c->launch_sms, kMoveWaves * c->move_bps[0]), 256, 0,
            c->stream>>>(a);
  ++c->kernel_launches;
  return cudaGetLastError();
}

static cudaError_t apply_part(jet_ctx *c, const MoveArgs &a) {
  k_apply_part<<<grid_for(c->n, 512, c->launch_sms), 256, 0, c->stream>>>(a);
  ++c->kernel_launches;
  return cudaGetLastError();
}

// The Jet moves of an iteration.  An apply pays two atomics with return on random sectors of phi per moved incidence
// (0.06 to 0.09 ns each on tables beyond L2, whatever their number), a count of phi from the partition streams the
// table once (at 4.2 TB/s or so: 0.65 ms for the 2 GB of the row-net workload).  So from
// rebuild_min = bytes / (4.2 TB/s * 0.075 ns * P/n) moves on, only the partition and the block weights move and phi
// and the bitmasks are counted anew.  Both forms are launched and the move count decides on the device; below 256 MB
// of phi, where the atomics stay in L2, only the first.  The first iterations of a refinement are of the second kind:
// eight iterations of rownet_4m took 42.6 ms with the apply alone and 39.1 so (vlsi_2m 7.99 and 7.94).
cudaError_t launch_apply_jet(jet_ctx *c, int32_t *part, int32_t *phi, int64_t *block_w) {
  const double phi_bytes = 4.0 * c->m * c->k;
  if (c->n == 0) return cudaSuccess;
  if (c->graph_path || phi_bytes < 256e6) {
    MoveArgs a = move_args(c, part, phi, block_w);
    a.weights = !c->rb_early;  // else launch_approve has done it
    return c->graph_path ? apply_part(c, a) : apply_phi(c, a);
  }
  const double bytes = phi_bytes + 8.0 * c->m * c->kwp + 8.0 * c->m + 8.0 * c->P;
  MoveArgs a = move_args(c, part, phi, block_w);
  a.weights = !c->rb_early;
  a.rebuild_min = (unsigned long long)(bytes / (4.2e3 * 0.075) * c->n / std::max<int64_t>(c->P, 1)) + 1;
  cudaError_t e = apply_phi(c, a);
  if (e == cudaSuccess) e = apply_part(c, a);
  if (e == cudaSuccess) e = launch_recount(c, part, phi, &c->cnt->n_moves, a.rebuild_min);
  return e;
}

cudaError_t launch_apply(jet_ctx *c, int32_t *part, int32_t *phi, int64_t *block_w) {
  if (c->n == 0) return cudaSuccess;
  const MoveArgs a = move_args(c, part, phi, block_w);
  return c->graph_path ? apply_part(c, a) : apply_phi(c, a);
}

cudaError_t launch_rb_check(jet_ctx *c, const int64_t *block_w, cudaGraphConditionalHandle cond, int use_cond) {
  k_rb_check<<<1, kMaxK, 0, c->stream>>>(rb_args(c, block_w), cond, use_cond);
  ++c->kernel_launches;
  return cudaGetLastError();
}

template <class KT>
void rb_select_levels(jet_ctx *c, const RbArgs &a) {
  const int g = grid_for(c->n, 256, c->launch_sms);
  int first = 1;
  for (int hi = a.tbits; hi > 0; first = 0) {
    const int lo = hi - a.digit > 0 ? hi - a.digit : 0;
    if (!first) {  // the first level's histogram comes from the target kernels
      k_rb_level<KT><<<g, 256, 0, c->stream>>>(a, lo, hi - lo);
      ++c->kernel_launches;
    }
    k_rb_pick<<<c->k, kPickThreads, 0, c->stream>>>(a, lo, first);
    ++c->kernel_launches;
    hi = lo;
  }
}

template <class KT, class WT>
cudaError_t select_segments(jet_ctx *c, const RbArgs &a, int64_t *bw) {
  ++c->kernel_launches;
  if (c->n <= kSelLarge) {  // no segment can be large
    k_rb_select<KT, WT, false><<<c->k, kSelThreads, 0, c->stream>>>(a, bw, 0, 0);
    return cudaGetLastError();
  }
  const int first = (c->k + kSelCluster - 1) / kSelCluster * kSelCluster;
  const int groups = std::min(c->n / kSelLarge, kSelGroups);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(first + groups * kSelCluster);
  cfg.blockDim = dim3(kSelThreads);
  cfg.stream = c->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kSelCluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_rb_select<KT, WT, true>, a, bw, first, groups);
}

cudaError_t launch_count_blocks(jet_ctx *c, const int32_t *part) {
  if (c->n == 0 || !c->rb_segments) return cudaSuccess;
  k_count_blocks<<<grid_for(c->n, 1024, c->launch_sms, 4), kMaxK, 0, c->stream>>>(part, c->n, c->k, c->cnt);
  ++c->kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_rb_select(jet_ctx *c, int64_t *block_w) {
  if (c->n == 0) return cudaSuccess;
  const RbArgs a = rb_args(c, nullptr);
  if (c->rb_segments) {
    int64_t *bw = c->rb_early ? block_w : nullptr;
    if (c->W < (1ll << 32))
      return a.tbits <= 64 ? select_segments<unsigned long long, unsigned>(c, a, bw)
                           : select_segments<u128, unsigned>(c, a, bw);
    return a.tbits <= 64 ? select_segments<unsigned long long, unsigned long long>(c, a, bw)
                         : select_segments<u128, unsigned long long>(c, a, bw);
  }
  if (a.tbits <= 64) rb_select_levels<unsigned long long>(c, a);
  else rb_select_levels<u128>(c, a);
  return cudaGetLastError();
}

cudaError_t launch_rb_apply(jet_ctx *c, int32_t *part, int32_t *phi, int64_t *block_w) {
  if (c->n == 0) return cudaSuccess;
  if (c->rb_segments) {  // the selection is a move list
    MoveArgs a = move_args(c, part, phi, block_w);
    a.weights = !c->rb_early;
    return c->graph_path ? apply_part(c, a) : apply_phi(c, a);
  }
  const RbArgs r = rb_args(c, block_w);
  const MoveArgs a = move_args(c, part, phi, block_w);
  if (r.tbits <= 64)
    k_rb_apply<unsigned long long><<<grid_for(c->n, 256, c->launch_sms, kRbMoveWaves * c->move_bps[1]), 256, 0,
                                     c->stream>>>(r, a);
  else
    k_rb_apply<u128><<<grid_for(c->n, 256, c->launch_sms, kRbMoveWaves * c->move_bps[2]), 256, 0, c->stream>>>(r, a);
  ++c->kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_rb_post(jet_ctx *c, const int64_t *block_w, cudaGraphConditionalHandle cond, int use_cond) {
  k_rb_post<<<1, kMaxK, 0, c->stream>>>(rb_args(c, block_w), cond, use_cond);
  ++c->kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_rollback_moves(jet_ctx *c, const int32_t *part, const int32_t *best, const int *enable) {
  cudaError_t e = cudaMemsetAsync(&c->cnt->n_moves, 0, sizeof(unsigned long long), c->stream);
  if (e != cudaSuccess || c->n == 0) return e;
  k_rollback_moves<<<grid_for(c->n, 256, c->launch_sms), 256, 0, c->stream>>>(part, best, c->n, c->mv_v, c->mv_st,
                                                                         c->cnt, enable);
  ++c->kernel_launches;
  return cudaGetLastError();
}

}  // namespace jet
