// State kernels: input validation, size classes, pin counts phi_e[i] with
// their connectivity bitmasks, block weights, and the connectivity metric
// (lambda-1) of Section 2.
#include <cstddef>
#include <type_traits>
#include <vector>

#include "jet_internal.cuh"

namespace jet {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ void add_i64(long long *p, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long *>(p), static_cast<unsigned long long>(v));
}

// Sum of a long long over the block, returned on thread 0.
__device__ long long block_sum_ll(long long x) {
  __shared__ long long s_part[32];
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(kFull, x, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) s_part[w] = x;
  __syncthreads();
  long long tot = 0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += s_part[i];
  __syncthreads();
  return tot;
}

// ---------------------------------------------------------------- validation
// Phase 1: offsets monotone and in range, weights positive and bounded.
__global__ void k_validate_offsets(const int64_t *eptr, const int64_t *vptr, const int32_t *vwgt,
                                   const int32_t *ewgt, int32_t n, int32_t m, int64_t P, Counters *cnt) {
  int err = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (int64_t)m + n + 2;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i <= m) {  // eptr[i]
      int64_t a = eptr[i];
      if (a < 0 || a > P) err |= kErrOffsets;
      if (i == 0 && a != 0) err |= kErrOffsets;
      if (i == m && a != P) err |= kErrOffsets;
      if (i < m && eptr[i + 1] < a) err |= kErrOffsets;
      if (i < m && ewgt[i] < 1) err |= kErrWeight;
    } else {
      int64_t v = i - m - 1;  // vptr[v], v in [0, n]
      int64_t a = vptr[v];
      if (a < 0 || a > P) err |= kErrOffsets;
      if (v == 0 && a != 0) err |= kErrOffsets;
      if (v == n && a != P) err |= kErrOffsets;
      if (v < n && vptr[v + 1] < a) err |= kErrOffsets;
      if (v < n && vwgt[v] < 1) err |= kErrWeight;
    }
  }
  if (err) atomicOr(&cnt->err, err);
}

// Phase 2: pin and incidence ids in range; occurrences of every vertex among the pins.
__global__ void k_validate_ids(const int32_t *pins, const int32_t *inc, int32_t n, int32_t m, int64_t P,
                               int32_t *degcount, Counters *cnt) {
  int err = 0;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < P; p += (int64_t)gridDim.x * blockDim.x) {
    int32_t v = pins[p];
    if (v < 0 || v >= n) err |= kErrPinRange;
    else atomicAdd(&degcount[v], 1);
    int32_t e = inc[p];
    if (e < 0 || e >= m) err |= kErrIncRange;
  }
  if (err) atomicOr(&cnt->err, err);
}

// Phase 3: degree of the transpose, weighted degree sum of omega over I(v), c(V), max c(v).
// scal[0] = c(V), scal[1] = max weighted degree, scal[2] = max c(v),
// scal[3] = max omega(e) over edges with at least one pin.
__global__ void k_validate_degrees(const int64_t *vptr, const int32_t *inc, const int32_t *vwgt,
                                   const int32_t *ewgt, int32_t n, const int32_t *degcount, int64_t *wdeg,
                                   unsigned long long *scal, Counters *cnt) {
  int err = 0;
  long long wsum = 0;
  unsigned long long wmax = 0, cm = 0, om = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    int64_t j0 = vptr[v], j1 = vptr[v + 1];
    if (j1 - j0 != degcount[v]) err |= kErrTranspose;
    long long d = 0;
    for (int64_t j = j0; j < j1; ++j) {
      const int32_t w = ewgt[inc[j]];
      d += w;
      om = (unsigned long long)w > om ? (unsigned long long)w : om;
    }
    wdeg[v] = d;
    wmax = d > (long long)wmax ? (unsigned long long)d : wmax;
    int32_t c = vwgt[v];
    wsum += c;
    cm = (unsigned long long)c > cm ? (unsigned long long)c : cm;
  }
  long long tot = block_sum_ll(wsum);
  if (threadIdx.x == 0) atomicAdd(&scal[0], (unsigned long long)tot);
  // one atomic per warp and maximum: from every thread they serialised on three addresses and the kernel
  // took 633 us for 1 M vertices
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    wmax = max(wmax, __shfl_xor_sync(kFull, wmax, o));
    cm = max(cm, __shfl_xor_sync(kFull, cm, o));
    om = max(om, __shfl_xor_sync(kFull, om, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&scal[1], wmax);
    atomicMax(&scal[2], cm);
    atomicMax(&scal[3], om);
  }
  if (err) atomicOr(&cnt->err, err);
}

// ---------------------------------------------------------------- classes
// Stable partition of ids [0, count) by class code (0 .. kClasses-1).
constexpr int kClasses = 24;
static_assert(kClasses < 32, "class codes and the no-class code fit match_bits<5>");

__global__ void k_class_count(const uint8_t *code, int32_t count, int32_t *blk_counts) {
  __shared__ int s_c[kClasses];
  if (threadIdx.x < kClasses) s_c[threadIdx.x] = 0;
  __syncthreads();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int c = i < count ? code[i] : kClasses;
  const unsigned grp = match_bits<5>((unsigned)c);  // c <= kClasses < 32
  if (c < kClasses && (threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(&s_c[c], __popc(grp));
  __syncthreads();
  if (threadIdx.x < kClasses) blk_counts[blockIdx.x * kClasses + threadIdx.x] = s_c[threadIdx.x];
}

__global__ void k_class_scatter(const uint8_t *code, int32_t count, const int32_t *blk_off, int32_t *out) {
  __shared__ int s_w[32][kClasses];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int x = threadIdx.x; x < 32 * kClasses; x += blockDim.x) s_w[x / kClasses][x % kClasses] = 0;
  __syncthreads();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int c = i < count ? code[i] : kClasses;
  const unsigned grp = match_bits<5>((unsigned)c);  // c <= kClasses < 32
  const unsigned rank = __popc(grp & ((1u << lane) - 1));
  if (c < kClasses && lane == __ffs(grp) - 1) s_w[w][c] = __popc(grp);
  __syncthreads();
  if (c < kClasses) {
    int base = blk_off[blockIdx.x * kClasses + c];
    for (int ww = 0; ww < w; ++ww) base += s_w[ww][c];
    out[base + rank] = (int32_t)i;
  }
}

__global__ void k_vertex_codes(const int64_t *wdeg, int32_t n, uint8_t *code) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    code[v] = wdeg[v] < (1ll << kLightPlanes) ? 0 : 1;
}

// Edge classes: code = |e| for |e| <= kTinyEdge (so the tiny list comes out
// ordered by size and a warp's edges tend to share one size); then the warp
// class split into edges of at most kHalfMidEdge and of at most
// kSmallMidEdge pins (one code each) and larger ones by size bucket, largest
// first, so the warps that get the longest edges start first; then the block
// class.
__global__ void k_edge_codes(const int64_t *eptr, int32_t m, uint8_t *code) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t sz = eptr[e + 1] - eptr[e];
    int c;
    if (sz <= kTinyEdge) c = (int)sz;
    else if (sz <= kHalfMidEdge) c = kTinyEdge + 1;
    else if (sz <= kSmallMidEdge) c = kTinyEdge + 2;
    else if (sz <= kWarpEdge) c = sz > 64 ? kTinyEdge + 3 : kTinyEdge + 4;  // 65..128 first, then 33..64
    else c = kTinyEdge + 5;
    code[e] = (uint8_t)c;
  }
}

// ---------------------------------------------------------------- pin counts
// A count that the device may call off: it runs if *value >= min (always without a value).
struct Gate {
  const unsigned long long *value;
  unsigned long long min;
  __device__ __forceinline__ bool closed() const { return value && *value < min; }
};

// A group of G lanes per edge of at most kWarpEdge pins: the pins' blocks are
// counted in the group's row in shared memory, which then goes out whole,
// four counts per lane, with its two mask words.  Bound by the writes of phi
// (4 k bytes an edge), so the loads must not stand in their way: the offsets
// of the edge three steps ahead, the pins of the one two ahead and the blocks
// of the next are in flight while an edge is counted (a warp per edge with
// nothing in flight took 364 us for 1.1 M edges at k = 128, 563 MB of phi).
// G = 8 lanes at k <= 64, else 16: the row goes out in two steps at most (four
// at k > 128), and most edges are that short.  Longer edges are counted by
// k_pincounts_seg; the rows of those longer than one segment are cleared here.
template <int KWP>
constexpr int kPinLanes = KWP <= 2 ? 8 : 16;
constexpr int kPinRegs = 2;  // pins per lane in flight

template <int KWP, bool VEC>  // VEC: rows are 16-byte aligned (k a multiple of 4, phi aligned)
__global__ void __launch_bounds__(256) k_pincounts(const int64_t *eptr, const int32_t *pins, const int32_t *part,
                                                   int32_t m, int32_t k, int32_t *phi, uint32_t *mask,
                                                   Counters *cnt, Gate gate) {
  if (gate.closed()) return;
  constexpr int G = kPinLanes<KWP>, K = 32 * KWP, Q = K / (4 * G), R = kPinRegs;
  __shared__ __align__(16) int s_h[256 / G][K];
  const int li = threadIdx.x % G;
  int *h = s_h[threadIdx.x / G];
  int4 *h4 = reinterpret_cast<int4 *>(h);
#pragma unroll
  for (int q = 0; q < Q; ++q) h4[li + q * G] = make_int4(0, 0, 0, 0);
  __syncwarp();
  const int64_t nw = (int64_t)gridDim.x * blockDim.x / G;
  int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  // the groups of a warp run in lockstep up to the warp's first group; one past the end has no pins
  int64_t iw = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / G;
  int err = 0;
  // stages, named by how many edges ahead they are; sz = 0 and pin = -1 past the end of an edge or the list
  auto offsets = [&](int64_t e, int64_t &p, int &sz) {
    p = e < m ? eptr[e] : 0;
    sz = e < m ? (int)min(eptr[e + 1] - p, (int64_t)kSegPins + 1) : 0;
  };
  auto load_pins = [&](int64_t p, int sz, int (&v)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = li + r * G < sz && sz <= kWarpEdge ? pins[p + li + r * G] : -1;
  };
  auto load_blocks = [&](const int (&v)[R], int (&b)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) b[r] = v[r] >= 0 ? part[v[r]] : 0;
  };
  int64_t p0, p1, p2, p3;
  int sz0, sz1, sz2, sz3, v0[R], v1[R], v2[R], b0[R], b1[R];
  offsets(i, p0, sz0);
  offsets(i + nw, p1, sz1);
  offsets(i + 2 * nw, p2, sz2);
  load_pins(p0, sz0, v0);
  load_pins(p1, sz1, v1);
  load_blocks(v0, b0);
  for (; iw < m; i += nw, iw += nw) {
    offsets(i + 3 * nw, p3, sz3);
    load_pins(p2, sz2, v2);
    load_blocks(v1, b1);
    const bool store = i < m && sz0 <= kWarpEdge;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (v0[r] < 0) continue;
      if ((unsigned)b0[r] < (unsigned)k) atomicAdd(&h[b0[r]], 1);
      else err |= kErrPartRange;
    }
    if (store) {
#pragma unroll 4
      for (int j = R * G + li; j < sz0; j += G) {
        const int b = part[pins[p0 + j]];
        if ((unsigned)b < (unsigned)k) atomicAdd(&h[b], 1);
        else err |= kErrPartRange;
      }
    }
    __syncwarp();
    int32_t *row = phi + i * k;
    if (i < m && sz0 > kSegPins)
      for (int b = li; b < k; b += G) row[b] = 0;
    if (!VEC && store)
      for (int b = li; b < k; b += G) row[b] = h[b];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int4 x = h4[li + q * G];
      if (VEC && store && 4 * (li + q * G) < k) reinterpret_cast<int4 *>(row)[li + q * G] = x;
      const int sh = 4 * (li & 7);
      uint32_t one = ((x.x > 0 ? 1u : 0u) | (x.y > 0 ? 2u : 0u) | (x.z > 0 ? 4u : 0u) | (x.w > 0 ? 8u : 0u)) << sh;
      uint32_t two = ((x.x > 1 ? 1u : 0u) | (x.y > 1 ? 2u : 0u) | (x.z > 1 ? 4u : 0u) | (x.w > 1 ? 8u : 0u)) << sh;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {  // the eight lanes of one mask word
        one |= __shfl_xor_sync(kFull, one, o);
        two |= __shfl_xor_sync(kFull, two, o);
      }
      if (store && (li & 7) == 0) {
        const int w = (li + q * G) >> 3;
        mask[i * 2 * KWP + w] = one;        // Lambda(e)
        mask[i * 2 * KWP + KWP + w] = two;  // blocks holding >= 2 pins of e
      }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < Q; ++q) h4[li + q * G] = make_int4(0, 0, 0, 0);
    __syncwarp();
    p0 = p1; sz0 = sz1;
    p1 = p2; sz1 = sz2;
    p2 = p3; sz2 = sz3;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v0[r] = v1[r];
      b0[r] = b1[r];
      v1[r] = v2[r];
    }
  }
  if (err) atomicOr(&cnt->err, err);
}

// The edges of more than kWarpEdge pins, by the segments of at most kSegPins
// pins that the afterburner's list holds (largest first): the blocks of a
// segment's pins are counted in shared memory, by a thread block
// (k_pincounts_seg) or a warp (k_pincounts_warp).  An edge of one segment
// (slot < 0) gets its row and mask words from there; the segments of a longer
// edge add their counts into the row, cleared by k_pincounts (one atomic per
// block of the partition that the segment touches), and k_masks_from_phi
// completes it.  Bound by the chain segment -> offset -> pins -> blocks ->
// counts where the segments are few, by the gathers of the blocks where they
// are many.  So a thread block has the shorter time for one segment and waits
// out three barriers per segment, and warps are the better form of segments of
// up to kSegWarp pins when there are many (n_seg_block, prepare_afterburner).
// 80,000 edges of 150 pins, k = 128: 116 us by thread blocks, 85 by warps;
// 20,000 of them, k = 256: 46.7 and 45; 20,000 of 600 pins 74 and 70, 8,000 of
// 1,500 pins 65 and 80; 20 of 1,000 pins beside 100,000 small ones 27.5 and
// 32 us.  Four pins per lane in flight: with eight and the registers for them
// (40) 92 us in the first of these.
__device__ __forceinline__ void store_counts(const int4 &sg, int b, int val, int32_t k, int32_t kwp, int32_t *phi,
                                             uint32_t *mask) {  // by whole warps, blocks b, b + 1, ... in its lanes
  int32_t *row = phi + (int64_t)sg.x * k;
  if (sg.w >= 0) {
    if (b < k && val) atomicAdd(&row[b], val);
    return;
  }
  if (b < k) row[b] = val;
  const unsigned one = __ballot_sync(kFull, val > 0), two = __ballot_sync(kFull, val > 1);
  if ((b & 31) == 0 && (b >> 5) < kwp) {
    mask[(int64_t)sg.x * 2 * kwp + (b >> 5)] = one;
    mask[(int64_t)sg.x * 2 * kwp + kwp + (b >> 5)] = two;
  }
}

__global__ void __launch_bounds__(256) k_pincounts_seg(const int64_t *eptr, const int32_t *pins, const int32_t *part,
                                                       const int4 *seg, int32_t nseg, int32_t k, int32_t kwp,
                                                       int32_t *phi, uint32_t *mask, Counters *cnt, Gate gate) {
  if (gate.closed()) return;
  __shared__ int s_h[kMaxK];
  int err = 0;
  for (int i = blockIdx.x; i < nseg; i += gridDim.x) {
    const int4 sg = seg[i];  // edge, first pin (offset in the edge), pins, slot
    s_h[threadIdx.x] = 0;    // kMaxK = blockDim.x
    __syncthreads();
    const int64_t p0 = eptr[sg.x] + sg.y;
#pragma unroll 4
    for (int j = threadIdx.x; j < sg.z; j += blockDim.x) {
      const int b = part[pins[p0 + j]];
      if ((unsigned)b < (unsigned)k) atomicAdd(&s_h[b], 1);
      else err |= kErrPartRange;
    }
    __syncthreads();
    store_counts(sg, threadIdx.x, s_h[threadIdx.x], k, kwp, phi, mask);
    __syncthreads();
  }
  if (err) atomicOr(&cnt->err, err);
}

template <int KWP>
__global__ void __launch_bounds__(256, 6) k_pincounts_warp(const int64_t *eptr, const int32_t *pins,
                                                           const int32_t *part, const int4 *seg, int32_t nseg,
                                                           int32_t k, int32_t *phi, uint32_t *mask, Counters *cnt,
                                                           Gate gate) {
  if (gate.closed()) return;
  constexpr int R = 4;  // pins per lane in flight
  __shared__ int s_h[256 / 32][32 * KWP];
  const int lane = threadIdx.x & 31, nw = gridDim.x * (256 / 32);
  int *h = s_h[threadIdx.x >> 5];
#pragma unroll
  for (int w = 0; w < KWP; ++w) h[32 * w + lane] = 0;
  __syncwarp();
  int err = 0;
  int i = blockIdx.x * (256 / 32) + (threadIdx.x >> 5);
  int4 next = i < nseg ? seg[i] : make_int4(0, 0, 0, -1);
  int64_t pn = i < nseg ? eptr[next.x] : 0;
  for (; i < nseg; i += nw) {
    const int4 sg = next;
    const int64_t p0 = pn + sg.y;
    if (i + nw < nseg) {  // used in the next turn
      next = seg[i + nw];
      pn = eptr[next.x];
    }
    for (int j0 = 0; j0 < sg.z; j0 += 32 * R) {
      int v[R];
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = j0 + 32 * q + lane < sg.z ? pins[p0 + j0 + 32 * q + lane] : -1;
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (j0 + 32 * q < sg.z) v[q] = v[q] >= 0 ? part[v[q]] : -2;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        if (j0 + 32 * q >= sg.z) break;  // the warp's lanes together
        if ((unsigned)v[q] < (unsigned)k) atomicAdd(&h[v[q]], 1);
        else if (v[q] != -2) err |= kErrPartRange;
      }
    }
    __syncwarp();
    int c[KWP];
#pragma unroll
    for (int w = 0; w < KWP; ++w) {
      c[w] = h[32 * w + lane];
      h[32 * w + lane] = 0;
    }
    __syncwarp();
#pragma unroll
    for (int w = 0; w < KWP; ++w) store_counts(sg, 32 * w + lane, c[w], k, KWP, phi, mask);
  }
  if (err) atomicOr(&cnt->err, err);
}

// c(V_i), aggregated per thread block in shared memory.  Bound by the
// shared-memory atomics on k addresses, so their width counts: W = unsigned
// when a block's share of the weights cannot leave 32 bits (the launcher
// checks it against max c(v)).  Four vertices in flight per thread.
template <class W>
__global__ void __launch_bounds__(256) k_block_weights(const int32_t *part, const int32_t *vwgt, int32_t n, int32_t k,
                                                       int64_t *bw, Counters *cnt) {
  __shared__ W s_bw[kMaxK];
  for (int b = threadIdx.x; b < k; b += blockDim.x) s_bw[b] = 0;
  __syncthreads();
  int err = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v0 < n; v0 += 4 * stride) {
    int b[4], c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t v = v0 + q * stride;
      b[q] = v < n ? part[v] : -2;
      c[q] = v < n ? vwgt[v] : 0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if ((unsigned)b[q] < (unsigned)k) atomicAdd(&s_bw[b[q]], (W)c[q]);
      else if (v0 + q * stride < n) err |= kErrPartRange;
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < k; b += blockDim.x)
    if (s_bw[b]) add_i64(reinterpret_cast<long long *>(&bw[b]), (long long)s_bw[b]);
  if (err) atomicOr(&cnt->err, err);
}

// Bitmasks of Lambda(e) and of the blocks with >= 2 pins from a dense phi
// (warp per edge): of every edge, or of the m edges listed in `list`.
__global__ void __launch_bounds__(256) k_masks_from_phi(const int32_t *phi, int32_t m, int32_t k, int32_t kwp,
                                                        uint32_t *mask, const int32_t *list, Gate gate) {
  if (gate.closed()) return;
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = gw; i < m; i += nw) {
    const int64_t e = list ? list[i] : i;
    const int32_t *row = phi + e * k;
    for (int q = 0; q < kwp; ++q) {
      int b = q * 32 + lane;
      const int val = b < k ? row[b] : 0;
      const unsigned one = __ballot_sync(kFull, val > 0), two = __ballot_sync(kFull, val > 1);
      if (lane == 0) {
        mask[e * 2 * kwp + q] = one;
        mask[e * 2 * kwp + kwp + q] = two;
      }
    }
  }
}

// (lambda-1) from a dense phi of 16-byte aligned rows, read once: a group of G
// lanes per row (four entries per lane and load), eight rows in flight per
// group.  A lane adds omega(e) per nonzero entry it sees and the group's first
// lane takes one omega(e) off if the row has any, so no sum crosses lanes
// until the end.  Bound by the read of phi (a warp per row, one load at a
// time: 300 us for 563 MB at k = 128).
template <int G>
__global__ void __launch_bounds__(256) k_connectivity_dense(const int32_t *phi, const int32_t *ewgt, int32_t m,
                                                            int32_t k, long long *out) {
  constexpr int kRows = 8;
  const int lane = threadIdx.x & 31, li = lane % G;
  const unsigned group = (G == 32 ? kFull : ((1u << (G % 32)) - 1) << (lane - li));
  const int64_t ng = (int64_t)gridDim.x * blockDim.x / G;
  const int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const int64_t gfirst = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / G;  // the warp's first group
  long long acc = 0;
  for (int64_t d = 0; gfirst + d < m; d += kRows * ng) {
    int c[kRows], w[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int64_t e = g + d + r * ng;
      c[r] = 0;
      w[r] = 0;
      if (e < m) {
        w[r] = ewgt[e];
        const int4 *row4 = reinterpret_cast<const int4 *>(phi + e * k);
#pragma unroll 2
        for (int x = li; 4 * x < k; x += G) {
          const int4 y = __ldcs(row4 + x);
          c[r] += (y.x > 0) + (y.y > 0) + (y.z > 0) + (y.w > 0);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const bool any = (__ballot_sync(kFull, c[r] > 0) & group) != 0;
      acc += (long long)(c[r] - (any && li == 0 ? 1 : 0)) * w[r];
    }
  }
  long long tot = block_sum_ll(acc);
  if (threadIdx.x == 0 && tot) add_i64(out, tot);
}

// The same for rows off the 16-byte boundary: one entry per lane and load, so
// a row takes Q loads per lane, all issued before the first is used.  Such
// rows share lines with their neighbours, so the loads go through L1, and rows
// in flight beyond what L1 holds cost more than they hide: 1 M rows at k = 255
// took 432 us with a loop over the loads of each of eight rows, 600 with four
// rows of eight loads in flight per warp and 32 warps, 243 with two and 48,
// and 190 with the grid in one wave.  At k = 61 eight rows and 32 warps take
// 127 us (177 by the loop), against 144 with 48 warps.
template <int Q>
constexpr int kRowsBlocks = Q <= 2 ? 4 : 6;  // resident blocks per SM
template <int G, int Q>
__global__ void __launch_bounds__(256, kRowsBlocks<Q>) k_connectivity_rows(const int32_t *phi, const int32_t *ewgt,
                                                                           int32_t m, int32_t k, long long *out) {
  constexpr int kRows = Q <= 2 ? 8 : Q <= 4 ? 4 : 2;
  const int lane = threadIdx.x & 31, li = lane % G;
  const unsigned group = (G == 32 ? kFull : ((1u << (G % 32)) - 1) << (lane - li));
  const int64_t ng = (int64_t)gridDim.x * blockDim.x / G;
  const int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const int64_t gfirst = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / G;  // the warp's first group
  long long acc = 0;
  for (int64_t d = 0; gfirst + d < m; d += kRows * ng) {
    int c[kRows], w[kRows], y[kRows][Q];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int64_t e = g + d + r * ng;
      const int32_t *row = phi + (e < m ? e : 0) * k;
      w[r] = e < m ? ewgt[e] : 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) y[r][q] = e < m && li + q * G < k ? row[li + q * G] : 0;
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      c[r] = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) c[r] += y[r][q] > 0;
      const bool any = (__ballot_sync(kFull, c[r] > 0) & group) != 0;
      acc += (long long)(c[r] - (any && li == 0 ? 1 : 0)) * w[r];
    }
  }
  long long tot = block_sum_ll(acc);
  if (threadIdx.x == 0 && tot) add_i64(out, tot);
}

// What follows the objective, done by the last of its blocks (a launch each
// took 1.3 to 2 us of an iteration of some 30 launches): the statistics and,
// in Algorithm 1's loop (rs), its control: a balanced, strictly smaller
// (lambda-1) resets the iteration counter and asks for a snapshot; the next
// iteration starts from cleared counters.
struct ObjEnd {
  const int64_t *bw;
  int32_t k;
  long long Lmax;
  jet_round_stats *out;
  int rebalance_only;
  RefineState *rs;
  int32_t limit;
  cudaGraphConditionalHandle loop;
};

__device__ void iteration_end(const ObjEnd &o, Counters *cnt, long long objective) {
  __shared__ long long s_mx[kMaxK / 32];
  const int t = threadIdx.x;  // kMaxK threads
  long long mx = t < o.k ? __ldcg(&o.bw[t]) : 0;
#pragma unroll
  for (int q = 16; q > 0; q >>= 1) mx = max(mx, __shfl_xor_sync(kFull, mx, q));
  if ((t & 31) == 0) s_mx[t >> 5] = mx;
  __syncthreads();
  if (t == 0) {
    for (int w = 0; w < kMaxK / 32; ++w) mx = max(mx, s_mx[w]);
    jet_round_stats st;
    st.candidates = o.rebalance_only ? 0 : (long long)cnt->n_cand;
    st.approved = o.rebalance_only ? 0 : (long long)cnt->approved;
    st.rebalance_rounds = cnt->rb_rounds;
    st.rebalance_moves = cnt->rb_moves;
    st.objective = objective;
    st.max_block_weight = mx;
    st.imbalanced = mx > o.Lmax ? 1 : 0;
    st.reserved = 0;
    *o.out = st;
    if (o.rs) {
      RefineState *rs = o.rs;
      rs->res.iterations += 1;
      rs->in_phase += 1;
      rs->it += 1;
      int snap = 0;
      if (!st.imbalanced && (!rs->have_best || st.objective < rs->best)) {
        rs->have_best = 1;
        rs->best = st.objective;
        rs->it = 0;
        snap = 1;
      }
      rs->snap = snap;
      cudaGraphSetConditional(o.loop, rs->it < o.limit ? 1u : 0u);
    }
  }
  if (o.rs) {
    __syncthreads();  // the counters have been read
    for (int x = t; x < (int)(offsetof(Counters, err) / 4); x += blockDim.x) reinterpret_cast<int *>(cnt)[x] = 0;
  }
}

// Adds the block's share of the objective; the last block to do so ends the call.
__device__ __forceinline__ void objective_add(long long acc, const ObjEnd &o, Counters *cnt) {
  __shared__ int s_last;
  const long long tot = block_sum_ll(acc);
  if (threadIdx.x == 0) {
    if (tot) add_i64(&cnt->objective, tot);
    __threadfence();
    s_last = atomicAdd(&cnt->ob_done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) iteration_end(o, cnt, __ldcg(&cnt->objective));  // every block has added before it counted itself
}

// (lambda-1) from the bitmasks: thread per edge, four rows in flight.
template <int KWP>
__global__ void __launch_bounds__(256) k_objective_masks(const uint32_t *mask, const int32_t *ewgt, int32_t m,
                                                         Counters *cnt, ObjEnd o) {
  long long acc = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e0 < m; e0 += 4 * stride) {
    int lam[4], w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int64_t e = e0 + r * stride;
      lam[r] = 0;
      w[r] = 0;
      if (e < m) {
        const uint32_t *row = mask + e * 2 * KWP;
        w[r] = ewgt[e];
        if constexpr (KWP == 1) {
          lam[r] = __popc(row[0]);
        } else if constexpr (KWP == 2) {
          const uint2 x = *reinterpret_cast<const uint2 *>(row);
          lam[r] = __popc(x.x) + __popc(x.y);
        } else {
#pragma unroll
          for (int h = 0; h < KWP / 4; ++h) {
            const uint4 x = reinterpret_cast<const uint4 *>(row)[h];
            lam[r] += __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (lam[r] > 0) acc += (long long)(lam[r] - 1) * w[r];
  }
  objective_add(acc, o, cnt);
}

// (lambda-1) of a graph (every edge two pins, so edge e's pins are pins[2e], pins[2e+1]): the weighted
// edge cut.  `pairs` is pins read as 8-byte pairs (NULL when pins is not 8-byte aligned); unit: all omega = 1.
// Bound by the gathers of the blocks: four edges in flight.
__global__ void __launch_bounds__(256) k_objective_cut(const int32_t *pins, const int2 *pairs, const int32_t *part,
                                                       const int32_t *ewgt, int32_t m, int unit, Counters *cnt,
                                                       ObjEnd o) {
  long long acc = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e0 < m; e0 += 4 * stride) {
    int2 p[4];
    int a[4], b[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int64_t e = e0 + r * stride;
      p[r] = e >= m ? make_int2(-1, -1) : pairs ? __ldcs(pairs + e) : make_int2(pins[2 * e], pins[2 * e + 1]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      a[r] = p[r].x >= 0 ? part[p[r].x] : 0;
      b[r] = p[r].x >= 0 ? part[p[r].y] : 0;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (a[r] != b[r]) acc += unit ? 1 : ewgt[e0 + r * stride];
  }
  objective_add(acc, o, cnt);
}

// The end of a call on a hypergraph without edges.
__global__ void __launch_bounds__(kMaxK) k_objective_none(Counters *cnt, ObjEnd o) { iteration_end(o, cnt, 0); }

// Edges that are not two distinct pins (the graph path needs none).
__global__ void k_count_non_pairs(const int64_t *eptr, const int32_t *pins, int32_t m, int32_t *bad) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = eptr[e];
    if (eptr[e + 1] - p != 2 || pins[p] == pins[p + 1]) atomicAdd(bad, 1);
  }
}

// adj[j] = the other pin of edge inc[j], for every incidence j of every vertex.
__global__ void k_build_adj(const int64_t *vptr, const int32_t *inc, const int64_t *eptr, const int32_t *pins,
                            int32_t n, int32_t *adj) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    for (int64_t j = vptr[v]; j < vptr[v + 1]; ++j) {
      const int64_t p = eptr[inc[j]];
      adj[j] = pins[p] == (int32_t)v ? pins[p + 1] : pins[p];
    }
  }
}

}  // namespace

cudaError_t launch_validate(jet_ctx *c, int64_t *wdeg_tmp, int32_t *degcount_tmp, unsigned long long *scal) {
  // phases 1..3; the caller synchronizes and checks cnt->err between phases
  cudaStream_t s = c->stream;
  int g = grid_for((int64_t)c->m + c->n + 2, 256, c->launch_sms);
  k_validate_offsets<<<g, 256, 0, s>>>(c->eptr, c->vptr, c->vwgt, c->ewgt, c->n, c->m, c->P, c->cnt);
  ++c->kernel_launches;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(c->cnt_host, c->cnt, sizeof(Counters), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
  if (c->cnt_host->err) return cudaSuccess;  // offsets unusable: stop before indexing with them
  if (c->P > 0) {
    k_validate_ids<<<grid_for(c->P, 256, c->launch_sms), 256, 0, s>>>(c->pins, c->inc, c->n, c->m, c->P, degcount_tmp,
                                                                    c->cnt);
    ++c->kernel_launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  e = cudaMemcpyAsync(c->cnt_host, c->cnt, sizeof(Counters), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
  if (c->cnt_host->err) return cudaSuccess;
  if (c->n > 0) {
    k_validate_degrees<<<grid_for(c->n, 256, c->launch_sms), 256, 0, s>>>(c->vptr, c->inc, c->vwgt, c->ewgt, c->n,
                                                                        degcount_tmp, wdeg_tmp, scal, c->cnt);
    ++c->kernel_launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Builds the class lists into one id array per kind (vertex: light, heavy;
// edge: tiny, mid, big).  Synchronizes.
static cudaError_t stable_partition(jet_ctx *c, const uint8_t *code, int32_t count, int32_t *out,
                                    int32_t totals[kClasses]) {
  for (int cl = 0; cl < kClasses; ++cl) totals[cl] = 0;
  if (count == 0) return cudaSuccess;
  const int bs = 1024;
  const int nb = (int)((count + bs - 1) / bs);
  int32_t *d_cnt = nullptr, *d_off = nullptr;
  cudaError_t e = jet::pool_alloc(&d_cnt, sizeof(int32_t) * kClasses * nb, c->stream);
  if (e != cudaSuccess) return e;
  e = jet::pool_alloc(&d_off, sizeof(int32_t) * kClasses * nb, c->stream);
  if (e != cudaSuccess) { cudaFreeAsync(d_cnt, c->stream); return e; }
  std::vector<int32_t> h((size_t)kClasses * nb);
  k_class_count<<<nb, bs, 0, c->stream>>>(code, count, d_cnt);
  e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h.data(), d_cnt, sizeof(int32_t) * kClasses * nb, cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e == cudaSuccess) {
    int64_t tot[kClasses] = {0}, run[kClasses];
    for (int b = 0; b < nb; ++b)
      for (int cl = 0; cl < kClasses; ++cl) tot[cl] += h[(size_t)kClasses * b + cl];
    int64_t acc = 0;
    for (int cl = 0; cl < kClasses; ++cl) { run[cl] = acc; acc += tot[cl]; }
    for (int b = 0; b < nb; ++b)
      for (int cl = 0; cl < kClasses; ++cl) {
        const int32_t x = h[(size_t)kClasses * b + cl];
        h[(size_t)kClasses * b + cl] = (int32_t)run[cl];
        run[cl] += x;
      }
    for (int cl = 0; cl < kClasses; ++cl) totals[cl] = (int32_t)tot[cl];
    e = cudaMemcpyAsync(d_off, h.data(), sizeof(int32_t) * kClasses * nb, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) {
      k_class_scatter<<<nb, bs, 0, c->stream>>>(code, count, d_off, out);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  }
  cudaFreeAsync(d_cnt, c->stream);
  cudaFreeAsync(d_off, c->stream);
  return e;
}

cudaError_t launch_classify(jet_ctx *c, const int64_t *wdeg) {
  // vertex lists live in one array: [light | heavy]; edge lists in one array
  // of m + (mid count) entries: [tiny | mid | big | room for deferred mid edges]
  int64_t mx = c->n > c->m ? c->n : c->m;
  uint8_t *code = nullptr;
  cudaError_t e = jet::pool_alloc(&code, mx > 0 ? mx : 1, c->stream);
  if (e != cudaSuccess) return e;
  int32_t t[kClasses];
  if (c->n > 0) {
    k_vertex_codes<<<grid_for(c->n, 256, c->launch_sms), 256, 0, c->stream>>>(wdeg, c->n, c->vheavy);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = stable_partition(c, c->vheavy, c->n, c->v_light, t);
  if (e == cudaSuccess) {
    c->n_light = t[0];
    c->n_heavy = t[1];
    c->v_heavy = c->v_light + t[0];
    if (c->m > 0) {
      k_edge_codes<<<grid_for(c->m, 256, c->launch_sms), 256, 0, c->stream>>>(c->eptr, c->m, code);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess) e = stable_partition(c, code, c->m, c->e_tiny, t);
  if (e == cudaSuccess) {
    c->n_tiny = 0;
    for (int cl = 0; cl <= kTinyEdge; ++cl) c->n_tiny += t[cl];
    c->n_mid_half = t[kTinyEdge + 1];
    c->n_mid_small = t[kTinyEdge + 2];
    c->n_mid = t[kTinyEdge + 3] + t[kTinyEdge + 4];
    c->n_mid_hi = t[kTinyEdge + 3];
    c->n_big = t[kTinyEdge + 5];
    c->e_mid_half = c->e_tiny + c->n_tiny;
    c->e_mid_small = c->e_mid_half + c->n_mid_half;
    c->e_mid = c->e_mid_small + c->n_mid_small;
    c->e_big = c->e_mid + c->n_mid;
  }
  cudaFreeAsync(code, c->stream);
  return e;
}

template <int KWP>
static void launch_pincounts_kwp(jet_ctx *c, const int32_t *part, int32_t *phi, bool vec, Gate gate) {
  const int g = grid_for((int64_t)c->m * kPinLanes<KWP>, 256, c->launch_sms, c->pin_bps[vec ? 1 : 0]);
  if (vec) k_pincounts<KWP, true><<<g, 256, 0, c->stream>>>(c->eptr, c->pins, part, c->m, c->k, phi, c->mask, c->cnt, gate);
  else k_pincounts<KWP, false><<<g, 256, 0, c->stream>>>(c->eptr, c->pins, part, c->m, c->k, phi, c->mask, c->cnt, gate);
}

// Resident blocks per SM of the pin-count kernels.
template <int KWP>
static cudaError_t prepare_pincounts_kwp(jet_ctx *c) {
  cudaError_t e = resident_blocks(k_pincounts<KWP, false>, 256, 0, &c->pin_bps[0]);
  if (e == cudaSuccess) e = resident_blocks(k_pincounts<KWP, true>, 256, 0, &c->pin_bps[1]);
  return e;
}

cudaError_t prepare_state_kernels(jet_ctx *c) {
  switch (c->kwp) {
    case 1: return prepare_pincounts_kwp<1>(c);
    case 2: return prepare_pincounts_kwp<2>(c);
    case 4: return prepare_pincounts_kwp<4>(c);
    default: return prepare_pincounts_kwp<8>(c);
  }
}

// phi and both bitmasks of every edge from part.
static cudaError_t launch_count_phi(jet_ctx *c, const int32_t *part, int32_t *phi, Gate gate) {
  cudaStream_t s = c->stream;
  const bool vec = c->k % 4 == 0 && ((uintptr_t)phi & 15) == 0;
  switch (c->kwp) {
    case 1: launch_pincounts_kwp<1>(c, part, phi, vec, gate); break;
    case 2: launch_pincounts_kwp<2>(c, part, phi, vec, gate); break;
    case 4: launch_pincounts_kwp<4>(c, part, phi, vec, gate); break;
    default: launch_pincounts_kwp<8>(c, part, phi, vec, gate); break;
  }
  ++c->kernel_launches;
  if (c->n_seg > 0) {  // edges above kWarpEdge pins
    const int nb = c->n_seg_block, nw = c->n_seg - nb;
    if (nb > 0)
      k_pincounts_seg<<<grid_for(nb, 1, c->launch_sms), kMaxK, 0, s>>>(c->eptr, c->pins, part, c->ab_seg, nb, c->k, c->kwp,
                                                                       phi, c->mask, c->cnt, gate);
    auto warps = [&](auto words) {
      k_pincounts_warp<decltype(words)::value><<<grid_for((int64_t)nw * 32, 256, c->launch_sms), 256, 0, s>>>(
          c->eptr, c->pins, part, c->ab_seg + nb, nw, c->k, phi, c->mask, c->cnt, gate);
    };
    if (nw > 0) switch (c->kwp) {
      case 1: warps(std::integral_constant<int, 1>()); break;
      case 2: warps(std::integral_constant<int, 2>()); break;
      case 4: warps(std::integral_constant<int, 4>()); break;
      default: warps(std::integral_constant<int, 8>()); break;
    }
    c->kernel_launches += (nb > 0) + (nw > 0);
  }
  if (c->n_slots > 0) {  // edges longer than one segment
    k_masks_from_phi<<<grid_for((int64_t)c->n_slots * 32, 256, c->launch_sms), 256, 0, s>>>(
        phi, c->n_slots, c->k, c->kwp, c->mask, c->ab_slot_edge, gate);
    ++c->kernel_launches;
  }
  return cudaGetLastError();
}

cudaError_t launch_recount(jet_ctx *c, const int32_t *part, int32_t *phi, const unsigned long long *value,
                           unsigned long long min) {
  if (c->m == 0) return cudaSuccess;
  return launch_count_phi(c, part, phi, Gate{value, min});
}

cudaError_t launch_pincounts(jet_ctx *c, const int32_t *part, int32_t *phi, int64_t *block_w) {
  cudaStream_t s = c->stream;
  cudaError_t e = cudaMemsetAsync(block_w, 0, sizeof(int64_t) * c->k, s);
  if (e != cudaSuccess) return e;
  if (c->m > 0 && phi && (e = launch_count_phi(c, part, phi, Gate{})) != cudaSuccess) return e;
  if (c->n > 0) {
    const int g = grid_for(c->n, 1024, c->launch_sms, 4);
    const long long share = ((c->n - 1ll) / (1024ll * g) + 1) * 1024;  // vertices of a block, at most
    if (share * c->cmax < (1ll << 32))
      k_block_weights<unsigned><<<g, 256, 0, s>>>(part, c->vwgt, c->n, c->k, block_w, c->cnt);
    else
      k_block_weights<unsigned long long><<<g, 256, 0, s>>>(part, c->vwgt, c->n, c->k, block_w, c->cnt);
    ++c->kernel_launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  c->phi_owner = phi;
  return cudaSuccess;
}

cudaError_t launch_masks_from_phi(jet_ctx *c, const int32_t *phi) {
  if (c->m > 0) {
    k_masks_from_phi<<<grid_for((int64_t)c->m * 32, 256, c->launch_sms), 256, 0, c->stream>>>(phi, c->m, c->k, c->kwp,
                                                                                            c->mask, nullptr, Gate{});
    ++c->kernel_launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  c->phi_owner = phi;
  return cudaSuccess;
}

cudaError_t launch_connectivity_dense(jet_ctx *c, const int32_t *phi, int64_t *out) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(int64_t), c->stream);
  if (e != cudaSuccess || c->m == 0) return e;
  const bool vec = c->k % 4 == 0 && ((uintptr_t)phi & 15) == 0;
  const int lanes = vec ? (c->k + 3) / 4 : c->k;  // lanes that one load of a row needs
  const int G = lanes > 16 ? 32 : lanes > 8 ? 16 : lanes > 4 ? 8 : lanes > 2 ? 4 : 2;
  long long *o = reinterpret_cast<long long *>(out);
  auto go = [&](auto lanes_c, auto loads_c) {  // loads_c: of rows that are not aligned
    constexpr int L = decltype(lanes_c)::value, Q = decltype(loads_c)::value;
    const int g = grid_for((int64_t)c->m * G, 256, c->launch_sms, vec ? 8 : kRowsBlocks<Q>);
    if (vec) k_connectivity_dense<L><<<g, 256, 0, c->stream>>>(phi, c->ewgt, c->m, c->k, o);
    else k_connectivity_rows<L, Q><<<g, 256, 0, c->stream>>>(phi, c->ewgt, c->m, c->k, o);
  };
  using std::integral_constant;
  switch (G) {
    case 2: go(integral_constant<int, 2>(), integral_constant<int, 1>()); break;
    case 4: go(integral_constant<int, 4>(), integral_constant<int, 1>()); break;
    case 8: go(integral_constant<int, 8>(), integral_constant<int, 1>()); break;
    case 16: go(integral_constant<int, 16>(), integral_constant<int, 1>()); break;
    default:
      switch ((lanes + 31) / 32) {  // 1 .. 8
        case 1: go(integral_constant<int, 32>(), integral_constant<int, 1>()); break;
        case 2: go(integral_constant<int, 32>(), integral_constant<int, 2>()); break;
        case 3:
        case 4: go(integral_constant<int, 32>(), integral_constant<int, 4>()); break;
        default: go(integral_constant<int, 32>(), integral_constant<int, 8>()); break;
      }
  }
  ++c->kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_objective(jet_ctx *c, const int32_t *part, const int64_t *block_w, jet_round_stats *stats,
                             int rebalance_only, RefineState *rs, int32_t limit, cudaGraphConditionalHandle h) {
  const ObjEnd o{block_w, c->k, c->Lmax, stats, rebalance_only, rs, limit, h};
  const int g = grid_for(c->m, 1024, c->launch_sms);
  if (c->m == 0) {
    k_objective_none<<<1, kMaxK, 0, c->stream>>>(c->cnt, o);
  } else if (c->graph_path) {
    const int2 *pairs = ((uintptr_t)c->pins & 7) ? nullptr : reinterpret_cast<const int2 *>(c->pins);
    k_objective_cut<<<g, 256, 0, c->stream>>>(c->pins, pairs, part, c->ewgt, c->m, c->unit_ewgt, c->cnt, o);
  } else {
    switch (c->kwp) {
      case 1: k_objective_masks<1><<<g, 256, 0, c->stream>>>(c->mask, c->ewgt, c->m, c->cnt, o); break;
      case 2: k_objective_masks<2><<<g, 256, 0, c->stream>>>(c->mask, c->ewgt, c->m, c->cnt, o); break;
      case 4: k_objective_masks<4><<<g, 256, 0, c->stream>>>(c->mask, c->ewgt, c->m, c->cnt, o); break;
      default: k_objective_masks<8><<<g, 256, 0, c->stream>>>(c->mask, c->ewgt, c->m, c->cnt, o); break;
    }
  }
  ++c->kernel_launches;
  return cudaGetLastError();
}

cudaError_t launch_build_adj(jet_ctx *c, int32_t *bad_edges) {
  cudaError_t e = cudaMemsetAsync(bad_edges, 0, sizeof(int32_t), c->stream);
  if (e != cudaSuccess) return e;
  if (c->m > 0) {
    k_count_non_pairs<<<grid_for(c->m, 256, c->launch_sms), 256, 0, c->stream>>>(c->eptr, c->pins, c->m, bad_edges);
    ++c->kernel_launches;
  }
  if (c->n > 0 && c->adj) {
    k_build_adj<<<grid_for(c->n, 256, c->launch_sms), 256, 0, c->stream>>>(c->vptr, c->inc, c->eptr, c->pins, c->n,
                                                                         c->adj);
    ++c->kernel_launches;
  }
  return cudaGetLastError();
}

}  // namespace jet
