// lines.cu -- classification, ordering, orientation and Catmull-Rom curves of
// the vortex-core lines of a sample graph (Sec. 3.4) on the GPU, parallel
// over samples: no thread walks a line.
//
// Input: the pierced-face graph of qtv_face_graph (neighbour table, degrees,
// component labels = lowest face index), the sample positions, and the face
// ids and windings (a sample's circulation direction is W times its face
// normal).
//
// Classification (per component, from the degrees of its samples): Type III
// when some degree exceeds 2 (branch points, e.g. at reconnections), Type II
// (closed loop) when every degree is 2 and the component has more than one
// sample, else Type I (an open line, or a single sample).
//
// Pieces (the simple lines, as in a walk that always takes the lowest
// unused neighbour): a Type I component is one piece from its lower end; a
// Type II component is one closed piece from its lowest sample towards the
// lower of that sample's two neighbours; a Type III component splits at its
// branch points: every chain between branch points and ends is a piece,
// started at a branch point b through neighbour v, and it is found from the
// branch side that comes first in (b, v) order (from the lower branch point;
// from the lower first neighbour for a chain that returns to b, which is then
// closed; dead ends are never starts).
//
// Ordering without walking.  "Special" samples end the chains: samples of
// degree other than 2, and the lowest sample of each Type II component.  On
// the directed edges (u -> w) of the graph (numbered compactly: sample u owns
// the edges from the exclusive scan of the degrees), the successor of (u -> w) is
// (w -> x), x the neighbour of w other than u, unless w is special.  Pointer
// jumping over this successor (double-buffered rounds of eight links, log8 of
// the sample count of them) gives every directed edge its distance to the end of its
// chain, the end sample and the sample before it.  A sample inside a chain
// then knows both ends, which end starts its piece, its position from that
// start (the distance back to it) and the piece's place in the output.
//
// Output order: pieces in ascending order of (start sample, first
// neighbour); each piece's samples in order, oriented (Sec. 3.4, right-hand
// rule) to run along their circulation direction: reversed when the sum over
// segments of (p[i+1] - p[i]) . dir[i] (with the closing segment for closed
// pieces) is negative, a closed piece keeping its first sample.  Curves:
// uniform Catmull-Rom, 'per_segment' points per segment, end points repeated
// for open pieces and wrapped for closed ones, plus the last sample of an open
// piece; lengths are the polyline lengths of the curves.  A lane computes the points
// of a segment; orientation sums (FP64) and lengths (a segment's distances in a pair of
// FP32 values, segments in FP64) go by chunks of entries in a fixed order, so results
// do not depend on timing.
#include <cstdio>

#include "qtv_internal.cuh"

namespace qtv {

struct LineWork {
  void* buf = nullptr;
  size_t cap = 0;
};

void line_work_free(LineWork* w) {
  if (!w) return;
  cudaFree(w->buf);
  delete w;
}

namespace {

constexpr int LT = 256;
constexpr int kMaxRounds = 64;  // jump rounds: log2 of 2^32 samples plus slack
constexpr int kHops = 8;        // links an edge follows in a round
constexpr uint32_t kEnded = 0x80000000u;
constexpr int kSlots = 10;

__device__ __forceinline__ unsigned long long limit_n(unsigned long long n, const uint64_t* n_dev) {
  if (n_dev) {
    const unsigned long long d = *n_dev;
    if (d < n) n = d;
  }
  return n;
}

struct LineArgs {
  unsigned long long n;
  const uint64_t* n_dev;
  const uint32_t* nbr;
  const uint8_t* deg;
  const uint32_t* comp;
  const float* xyz;
  const uint64_t* face_ids;
  const int8_t* winding;
  // workspace
  uint32_t* cflags;  // per component label: 1 = a sample of degree > 2,
                     // 2 = a sample of degree < 2
  uint8_t* special;  // per sample
  uint32_t* deg32;   // degrees as 32-bit values (scan input)
  unsigned long long* aoff;   // per sample: first directed edge (exclusive scan of degrees)
  const unsigned long long* narcs;  // device: number of directed edges
  uint32_t* atail;   // per directed edge: tail sample
  uint32_t* ahead;   // per directed edge: head sample
  // per directed edge, double-buffered: x = successor edge, y = edges from this
  // one to it; once the chain has ended (kEnded in y) x = its last edge, y =
  // edges to its end (one 8-byte gather per link)
  uint2* jmp[2];
  uint32_t* live;    // per round: 1 if an edge's chain has not ended yet
  uint32_t* fbuf;    // buffer of the final jump results
  uint32_t* pcount;  // per sample: pieces started there
  uint32_t* plen;    // per sample: nodes of the pieces started there
  unsigned long long* pfirst;  // exclusive scan of pcount
  unsigned long long* noff;    // exclusive scan of plen
  unsigned long long* edge_node_off;  // per starting edge slot: node offset of its piece
  uint32_t* tmp_nodes;   // unoriented node list
  double *left, *right;  // per chunk of node entries: orientation partials
  // outputs
  qtv_piece* pieces;
  unsigned long long piece_cap;
  uint32_t* nodes;
  unsigned long long node_cap;
};

__device__ __forceinline__ int comp_type(const LineArgs& a, uint32_t L) {
  // every degree 2 (a loop; a lone sample has degree 0) -> II; a branch -> III
  const uint32_t f = a.cflags[L];
  if (f & 1u) return 3;
  if (f == 0u) return 2;
  return 1;
}

__global__ void stats_init_kernel(LineArgs a) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  for (unsigned long long u = (unsigned long long)blockIdx.x * LT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * LT) {
    a.cflags[u] = 0;
  }
}

__global__ void stats_kernel(LineArgs a) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  for (unsigned long long u = (unsigned long long)blockIdx.x * LT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * LT) {
    const uint32_t L = a.comp[u], d = a.deg[u];
    a.deg32[u] = d;
    // only line ends and branch points mark their component (interior samples
    // of degree 2 mark nothing), and a mark already set is not set again
    if (d != 2u) {
      const uint32_t bit = d > 2u ? 1u : 2u;
      if ((a.cflags[L] & bit) == 0u) atomicOr(a.cflags + L, bit);
    }
  }
}

__global__ void special_kernel(LineArgs a) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  for (unsigned long long u = (unsigned long long)blockIdx.x * LT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * LT) {
    const uint32_t L = a.comp[u];
    const int t = comp_type(a, L);
    const int d = a.deg[u];
    a.special[u] = (t == 2) ? (uint8_t)(u == L) : (uint8_t)(d != 2);
  }
}

// slot of neighbour x in the row of w (rows are ascending, at most 10)
__device__ __forceinline__ int slot_of(const LineArgs& a, uint32_t w, uint32_t x) {
  const uint32_t* r = a.nbr + (unsigned long long)w * kSlots;
  for (int s = 0; s < kSlots; ++s)
    if (r[s] == x) return s;
  return -1;
}

// directed edges in compact order: sample u owns edges aoff[u] .. + deg[u] - 1
__global__ void arcs_kernel(LineArgs a) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  for (unsigned long long u = (unsigned long long)blockIdx.x * LT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * LT) {
    const int d = a.deg[u];
    const unsigned long long e0 = a.aoff[u];
    for (int s = 0; s < d; ++s) {
      a.atail[e0 + s] = (uint32_t)u;
      a.ahead[e0 + s] = a.nbr[u * kSlots + s];
    }
  }
}

__global__ void edges_init_kernel(LineArgs a) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long ne = *a.narcs;
  for (unsigned long long e = (unsigned long long)blockIdx.x * LT + threadIdx.x; e < ne;
       e += (unsigned long long)gridDim.x * LT) {
    const uint32_t u = a.atail[e], w = a.ahead[e];
    if (a.special[w]) {
      a.jmp[0][e] = make_uint2((uint32_t)e, 1u | kEnded);
    } else {
      // w has degree 2: continue to its other neighbour
      const int sx = (a.nbr[(unsigned long long)w * kSlots] == u) ? 1 : 0;
      a.jmp[0][e] = make_uint2((uint32_t)(a.aoff[w] + sx), 1u);
    }
  }
}

// Round r of pointer jumping (src = r & 1): kHops links a round, so a chain of m
// edges takes log(m) / log(kHops) rounds.  It is skipped once the previous
// round left no edge with a successor (every chain has ended), so the rounds
// beyond the longest chain cost a launch each; fbuf names the buffer that the
// last round run wrote.  594e3 samples, device time of all rounds: one link a
// round 225 us (20 launches), four 137 (10), eight 119 (7); with records of 8
// bytes instead of 16, 105.
__global__ void jump_kernel(LineArgs a, int src, int r) {
  pdl_wait();
  pdl_trigger();
  if (r > 0 && a.live[r - 1] == 0u) return;
  const unsigned long long ne = *a.narcs;
  const int d = src ^ 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.fbuf = (uint32_t)d;
  bool flagged = false;  // this block has seen the round's flag set
  for (unsigned long long e0 = (unsigned long long)blockIdx.x * LT; e0 < ne;
       e0 += (unsigned long long)gridDim.x * LT) {
    const unsigned long long e = e0 + threadIdx.x;
    bool more = false;
    if (e < ne) {
      uint2 J = a.jmp[src][e];
      if (J.y & kEnded) {
        // an edge whose chain ended two rounds ago already holds its final
        // values in both buffers
        if (r < 2 || !(a.jmp[d][e].y & kEnded)) a.jmp[d][e] = J;
      } else {
#pragma unroll
        for (int hop = 1; hop < kHops; ++hop)
          if (!(J.y & kEnded)) {
            const uint2 N = a.jmp[src][J.x];
            J = make_uint2(N.x, J.y + N.y);
          }
        a.jmp[d][e] = J;
        more = !(J.y & kEnded);
      }
    }
    // one flag per round, set by the first block that finds a live edge (a
    // block reads it at most once, so the flag's line sees few requests)
    if (__syncthreads_or(more) && !flagged) {
      flagged = true;
      if (threadIdx.x == 0 && *reinterpret_cast<volatile uint32_t*>(a.live + r) == 0u)
        a.live[r] = 1u;
    }
  }
}

// edges of the chain that edge e starts
__device__ __forceinline__ uint32_t chain_len(const LineArgs& a, int buf, unsigned long long e) {
  return a.jmp[buf][e].y & ~kEnded;
}

// end sample and the sample before it, of the chain that edge e starts
__device__ __forceinline__ void chain_end(const LineArgs& a, int buf, uint32_t e, uint32_t& end,
                                          uint32_t& before) {
  const uint32_t l = a.jmp[buf][e].x;
  before = a.atail[l];
  end = a.ahead[l];
}

// is the chain that starts at special sample s through neighbour y (edge e) a
// piece start?
__device__ __forceinline__ bool discovering(const LineArgs& a, int buf, uint32_t s, uint32_t y,
                                            uint32_t e) {
  uint32_t end, before;
  chain_end(a, buf, e, end, before);
  const int t = comp_type(a, a.comp[s]);
  if (t == 1) return s < end;
  if (t == 2) return y < before;
  if (a.deg[s] <= 2) return false;  // dead end
  if (end == s) return y < before;
  if (a.deg[end] > 2) return s < end;
  return true;
}

__global__ void count_kernel(LineArgs a) {
  pdl_wait();
  pdl_trigger();
  const int buf = (int)*a.fbuf;
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  for (unsigned long long u = (unsigned long long)blockIdx.x * LT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * LT) {
    uint32_t pc = 0, nl = 0;
    const int d = a.deg[u];
    if (d == 0) {
      pc = 1;
      nl = 1;
    } else if (a.special[u]) {
      for (int s = 0; s < d; ++s) {
        const unsigned long long e = a.aoff[u] + s;
        const uint32_t y = a.nbr[u * kSlots + s];
        if (!discovering(a, buf, (uint32_t)u, y, (uint32_t)e)) continue;
        uint32_t end, before;
        chain_end(a, buf, (uint32_t)e, end, before);
        ++pc;
        nl += chain_len(a, buf, e) + (end == (uint32_t)u ? 0u : 1u);
      }
    }
    a.pcount[u] = pc;
    a.plen[u] = nl;
  }
}

// piece records, and the start and end samples of every piece
__global__ void pieces_kernel(LineArgs a) {
  pdl_wait();
  pdl_trigger();
  const int buf = (int)*a.fbuf;
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  for (unsigned long long u = (unsigned long long)blockIdx.x * LT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * LT) {
    if (a.pcount[u] == 0) continue;
    unsigned long long p = a.pfirst[u], off = a.noff[u];
    const uint32_t L = a.comp[u];
    const uint8_t ct = (uint8_t)comp_type(a, L);
    const int d = a.deg[u];
    if (d == 0) {
      if (p < a.piece_cap) {
        qtv_piece r = {};
        r.first = off;
        r.count = 1;
        r.component = L;
        r.comp_type = ct;
        a.pieces[p] = r;
      }
      a.tmp_nodes[off] = (uint32_t)u;
      continue;
    }
    for (int s = 0; s < d; ++s) {
      const unsigned long long e = a.aoff[u] + s;
      const uint32_t y = a.nbr[u * kSlots + s];
      if (!discovering(a, buf, (uint32_t)u, y, (uint32_t)e)) continue;
      uint32_t end, before;
      chain_end(a, buf, (uint32_t)e, end, before);
      const bool closed = end == (uint32_t)u;
      const uint32_t cnt = chain_len(a, buf, e) + (closed ? 0u : 1u);
      if (p < a.piece_cap) {
        qtv_piece r = {};
        r.first = off;
        r.count = cnt;
        r.component = L;
        r.closed = closed ? 1 : 0;
        r.comp_type = ct;
        a.pieces[p] = r;
      }
      a.edge_node_off[e] = off;
      a.tmp_nodes[off] = (uint32_t)u;
      if (!closed) a.tmp_nodes[off + cnt - 1] = end;
      ++p;
      off += cnt;
    }
  }
}

// samples inside chains: their piece and position from its start
__global__ void interior_kernel(LineArgs a) {
  pdl_wait();
  pdl_trigger();
  const int buf = (int)*a.fbuf;
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  for (unsigned long long u = (unsigned long long)blockIdx.x * LT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * LT) {
    if (a.special[u] || a.deg[u] != 2) continue;
    const unsigned long long e0 = a.aoff[u], e1 = e0 + 1;
    uint32_t end0, bef0, end1, bef1;
    chain_end(a, buf, (uint32_t)e0, end0, bef0);
    chain_end(a, buf, (uint32_t)e1, end1, bef1);
    // the chain's end edges, seen from the ends: (end0 -> bef0), (end1 -> bef1)
    const int s0 = slot_of(a, end0, bef0), s1 = slot_of(a, end1, bef1);
    if (s0 < 0 || s1 < 0) continue;
    const unsigned long long f0 = a.aoff[end0] + s0;
    const unsigned long long f1 = a.aoff[end1] + s1;
    unsigned long long off;
    uint32_t pos;
    if (discovering(a, buf, end0, bef0, (uint32_t)f0)) {
      off = a.edge_node_off[f0];
      pos = chain_len(a, buf, e0);
    } else if (discovering(a, buf, end1, bef1, (uint32_t)f1)) {
      off = a.edge_node_off[f1];
      pos = chain_len(a, buf, e1);
    } else {
      continue;
    }
    a.tmp_nodes[off + pos] = (uint32_t)u;
  }
}

// ---------------------------------------------------------------------------
// Sums over pieces.  The entries of all pieces are cut
// into chunks of fixed length, one warp each, whatever the lengths of the
// pieces: a warp per piece left the longest one (18231 samples of 1.39e6 at
// 512^3) running alone.  A piece inside one chunk is summed there; one that
// spans chunks leaves a partial per chunk (right: it starts in this one, left:
// it started before), which are added in a fixed order.
// ---------------------------------------------------------------------------
constexpr unsigned long long kNodeChunk = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int d = 16; d; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
  return __shfl_sync(0xffffffffu, v, 0);
}

// the last of np ascending values first(p) that is <= g
template <typename F>
__device__ __forceinline__ unsigned long long last_at_most(unsigned long long lo, unsigned long long hi,
                                                           unsigned long long g, F first) {
  while (hi - lo > 1) {
    const unsigned long long mid = (lo + hi) >> 1;
    if (first(mid) <= g) lo = mid;
    else hi = mid;
  }
  return lo;
}

// sum of a piece [first, end) that spans chunks, by the calling warp
__device__ __forceinline__ double spanning_sum(const double* left, const double* right,
                                               unsigned long long first, unsigned long long end,
                                               unsigned long long chunk) {
  const unsigned long long c0 = first / chunk, c1 = (end - 1) / chunk;
  const int lane = threadIdx.x & 31;
  double v = lane == 0 ? right[c0] : 0.0;
  for (unsigned long long c = c0 + 1 + lane; c <= c1; c += 32) v += left[c];
  return warp_sum(v);
}

// outputs that do not fit are incomplete whatever they hold: the caller comes again
__device__ __forceinline__ bool too_many(const LineArgs& a, const unsigned long long* counts) {
  return counts[0] > a.piece_cap || counts[1] > a.node_cap;
}

// node entries of the pieces, and the calling warp's chunks of them
__device__ __forceinline__ unsigned long long node_total(const LineArgs& a, unsigned long long np) {
  return np ? a.pieces[np - 1].first + a.pieces[np - 1].count : 0ull;
}

// orientation sums: final for pieces inside a chunk, partials for the others
__global__ void orient_kernel(LineArgs a, const unsigned long long* counts) {
  pdl_wait();
  pdl_trigger();
  if (too_many(a, counts)) return;
  const unsigned long long np = counts[0];
  const unsigned long long total = node_total(a, np);
  const int lane = threadIdx.x & 31;
  const unsigned long long warps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
  const bool dirs = a.face_ids && a.winding;
  for (unsigned long long c = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
       c * kNodeChunk < total; c += warps) {
    const unsigned long long g0 = c * kNodeChunk, g1 = min(total, g0 + kNodeChunk);
    unsigned long long p = last_at_most(0, np, g0, [&](unsigned long long m) { return a.pieces[m].first; });
    for (; p < np; ++p) {
      const qtv_piece r = a.pieces[p];
      if (r.first >= g1) break;
      const unsigned long long end = r.first + r.count;
      double sum = 0.0;
      if (dirs && r.count >= 2) {
        const unsigned long long last = r.closed ? end : end - 1;  // one segment per entry below it
        float nan = 0.f;  // NaN once a coordinate is not finite (so is the sum then)
        for (unsigned long long i = max((unsigned long long)r.first, g0) + lane; i < min(last, g1); i += 32) {
          const uint32_t u = a.tmp_nodes[i];
          const uint32_t v = a.tmp_nodes[i + 1 == end ? r.first : i + 1];
          // (p[i+1] - p[i]) . d, d = W times the face normal: one axis (FP64
          // units are scarce)
          const int o = (int)(a.face_ids[u] & 3u);
          const int ax = o == 0 ? 2 : (o == 1 ? 0 : 1);  // z, x, y for xy, yz, zx faces
          float pu[3], pv[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            pu[k] = a.xyz[3ull * u + k];
            pv[k] = a.xyz[3ull * v + k];
            nan = fmaf(pu[k], 0.f, fmaf(pv[k], 0.f, nan));
          }
          const float cu = ax == 0 ? pu[0] : (ax == 1 ? pu[1] : pu[2]);
          const float cv = ax == 0 ? pv[0] : (ax == 1 ? pv[1] : pv[2]);
          if (o != 3) sum = fma((double)cv - (double)cu, (double)a.winding[u], sum);
        }
        sum += (double)nan;
      }
      sum = warp_sum(sum);
      if (lane == 0) {
        if (r.first < g0) a.left[c] = sum;
        else if (end > g1) a.right[c] = sum;
        else if (sum < 0.0) a.pieces[p].reversed = 1;
      }
    }
  }
}

// final node list: each piece in order, or reversed (closed: first kept); the
// first chunk of a spanning piece sets its flag
__global__ void place_kernel(LineArgs a, const unsigned long long* counts) {
  pdl_wait();
  pdl_trigger();
  if (too_many(a, counts)) return;
  const unsigned long long np = counts[0];
  const unsigned long long total = node_total(a, np);
  const int lane = threadIdx.x & 31;
  const unsigned long long warps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
  for (unsigned long long c = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
       c * kNodeChunk < total; c += warps) {
    const unsigned long long g0 = c * kNodeChunk, g1 = min(total, g0 + kNodeChunk);
    unsigned long long p = last_at_most(0, np, g0, [&](unsigned long long m) { return a.pieces[m].first; });
    for (; p < np; ++p) {
      const qtv_piece r = a.pieces[p];
      if (r.first >= g1) break;
      const unsigned long long end = r.first + r.count;
      bool rev = r.reversed != 0;
      if (r.first < g0 || end > g1) {
        rev = spanning_sum(a.left, a.right, r.first, end, kNodeChunk) < 0.0;
        if (rev && r.first >= g0 && lane == 0) a.pieces[p].reversed = 1;
      }
      for (unsigned long long i = max((unsigned long long)r.first, g0) + lane; i < min(end, g1); i += 32) {
        const unsigned long long k = i - r.first;
        unsigned long long src = k;
        if (rev) src = r.closed ? (k == 0 ? 0 : r.count - k) : r.count - 1 - k;
        a.nodes[i] = a.tmp_nodes[r.first + src];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Exclusive scan into u64, of one or two arrays at once: the sums of chunks of
// SCHUNK values, then every block scans its chunk on top of the sums before it
// (a single thread adding them took 11 us of each scan).
// ---------------------------------------------------------------------------
constexpr int SB = 1024;        // threads per scan block
constexpr int SPER = 4;         // values per thread
constexpr int SCHUNK = SB * SPER;

template <typename T>
struct ScanArgs {
  const T* in[2];
  unsigned long long* out[2];
  unsigned long long* total[2];  // of each array
  unsigned long long* bsum;   // [2][chunks]
  unsigned long long n;
  const uint64_t* n_dev;
};

// sum over the block (all threads get it)
__device__ __forceinline__ unsigned long long block_total(unsigned long long v, unsigned long long* wt) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  __syncthreads();  // wt may still be read
  if (lane == 0) wt[w] = v;
  __syncthreads();
  v = wt[lane];
#pragma unroll
  for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

template <typename T>
__global__ void __launch_bounds__(SB) scan_sums_kernel(ScanArgs<T> a) {
  pdl_wait();
  pdl_trigger();
  __shared__ unsigned long long wt[32];
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  const T* in = a.in[blockIdx.y];
  unsigned long long loc = 0;
  for (unsigned long long i = (unsigned long long)blockIdx.x * SCHUNK + threadIdx.x;
       i < min(nn, ((unsigned long long)blockIdx.x + 1) * SCHUNK); i += SB)
    loc += in[i];
  loc = block_total(loc, wt);
  if (threadIdx.x == 0) a.bsum[(unsigned long long)blockIdx.y * gridDim.x + blockIdx.x] = loc;
}

template <typename T>
__global__ void __launch_bounds__(SB) scan_apply_kernel(ScanArgs<T> a) {
  pdl_wait();
  pdl_trigger();
  __shared__ unsigned long long wt[32];
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  const T* in = a.in[blockIdx.y];
  unsigned long long* out = a.out[blockIdx.y];
  const unsigned long long* bsum = a.bsum + (unsigned long long)blockIdx.y * gridDim.x;
  unsigned long long before = 0;
  for (unsigned long long b = threadIdx.x; b < blockIdx.x; b += SB) before += bsum[b];
  before = block_total(before, wt);
  const unsigned long long base = (unsigned long long)blockIdx.x * SCHUNK + threadIdx.x * SPER;
  unsigned long long v[SPER], loc = 0;
#pragma unroll
  for (int i = 0; i < SPER; ++i) {
    v[i] = base + i < nn ? in[base + i] : 0;
    loc += v[i];
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned long long inc = loc;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= d) inc += t;
  }
  __syncthreads();  // wt may still be read
  if (lane == 31) wt[w] = inc;
  __syncthreads();
  unsigned long long run = before + inc - loc;
  for (int q = 0; q < w; ++q) run += wt[q];
#pragma unroll
  for (int i = 0; i < SPER; ++i) {
    if (base + i < nn) out[base + i] = run;
    run += v[i];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == SB - 1) *a.total[blockIdx.y] = run;
}

// bsum: one entry per chunk (at least one) and array
template <typename T>
void scan(const T* in0, const T* in1, const uint64_t* n_dev, unsigned long long n,
          unsigned long long* out0, unsigned long long* out1, unsigned long long* bsum,
          unsigned long long* total0, unsigned long long* total1, cudaStream_t st) {
  ScanArgs<T> a{{in0, in1}, {out0, out1}, {total0, total1}, bsum, n, n_dev};
  const unsigned nb = (unsigned)((n + SCHUNK - 1) / SCHUNK);
  const dim3 grid(nb > 0 ? nb : 1, in1 ? 2 : 1);
  launch_dependent(scan_sums_kernel<T>, dim3(grid), dim3(SB), 0, st, a);
  launch_dependent(scan_apply_kernel<T>, dim3(grid), dim3(SB), 0, st, a);
}

// ---------------------------------------------------------------------------
// curves
// ---------------------------------------------------------------------------
struct CurveArgs {
  const float* xyz;
  const uint32_t* nodes;
  const qtv_piece* pieces;
  unsigned long long np;
  const uint64_t* np_dev;
  int per;
  uint32_t *npts, *count;         // per piece: curve points, samples
  unsigned long long* cfirst;     // exclusive scan of npts
  unsigned long long* efirst;     // exclusive scan of count
  const unsigned long long* entries;  // samples of all pieces
  float* curve;
  unsigned long long curve_cap;
  float* length;
  double *left, *right;           // per warp of entries: length partials
};

__device__ __forceinline__ uint32_t curve_points(const qtv_piece& r, int per) {
  if (r.count < 2) return r.count;
  return r.closed ? r.count * (uint32_t)per : (r.count - 1) * (uint32_t)per + 1;
}

__global__ void curve_count_kernel(CurveArgs a) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long np = limit_n(a.np, a.np_dev);
  for (unsigned long long p = (unsigned long long)blockIdx.x * LT + threadIdx.x; p < np;
       p += (unsigned long long)gridDim.x * LT) {
    const qtv_piece r = a.pieces[p];
    a.npts[p] = curve_points(r, a.per);
    a.count[p] = r.count;
  }
}

__device__ __forceinline__ void sample_pos(const CurveArgs& a, const qtv_piece& r, long long i,
                                           float p[3]) {
  const uint32_t u = a.nodes[r.first + (unsigned long long)i];
  p[0] = a.xyz[3ull * u];
  p[1] = a.xyz[3ull * u + 1];
  p[2] = a.xyz[3ull * u + 2];
}

// One lane per sample of the pieces (in piece order): the points of the segment
// that starts there, or the one point of a last or lone sample, and the
// segment's share of the polyline length (FP32 lengths between the points, from
// exact coordinate differences, the next segment's first point being the next
// sample itself; those of a segment added in FP32 with their rounding errors
// kept, the segments in FP64 in a fixed order).  The points of a warp go
// through shared memory, kStage a sample at a time, and out in runs.  A thread
// per point that gathered its four samples (and the lengths from the points
// read back) took 70 and 50 us for 4.9e6 points; this takes 59 us, of 9 to
// write them (54% of the issue slots taken).
constexpr int kStage = 8, kStagePitch = 3 * kStage + 1;

__global__ void __launch_bounds__(LT) curve_kernel(CurveArgs a) {
  pdl_wait();
  pdl_trigger();
  __shared__ float stage[LT / 32][32 * kStagePitch];
  const unsigned long long np = limit_n(a.np, a.np_dev);
  // the pieces that fit come first and have at least a point a sample
  const unsigned long long ne = min((unsigned long long)*a.entries, a.curve_cap);
  const int lane = threadIdx.x & 31;
  float* const st = stage[threadIdx.x >> 5];
  const unsigned long long warps = ((unsigned long long)gridDim.x * LT) >> 5;
  auto first = [&](unsigned long long m) { return a.efirst[m]; };
  for (unsigned long long c = ((unsigned long long)blockIdx.x * LT + threadIdx.x) >> 5; c * 32 < ne;
       c += warps) {
    const unsigned long long g0 = c * 32, g = g0 + lane;
    const bool act = g < ne;
    // pieces of the first and the last sample, then each lane's between them
    const unsigned long long edge = lane == 0 ? g0 : min(ne, g0 + 32) - 1;
    const unsigned long long mine = lane < 2 ? last_at_most(0, np, edge, first) : 0ull;
    const unsigned long long lo = __shfl_sync(0xffffffffu, mine, 0);
    const unsigned long long hi = __shfl_sync(0xffffffffu, mine, 1) + 1;
    const unsigned long long p = act ? last_at_most(lo, hi, g, first) : lo;
    const qtv_piece r = a.pieces[p];
    const unsigned long long e0 = a.efirst[p], c0 = a.cfirst[p];
    const long long m = r.count, s = act ? (long long)(g - e0) : 0;
    // a piece whose curve does not fit is left out
    const bool fits = act && c0 + a.npts[p] <= a.curve_cap;
    const bool seg = fits && (r.closed ? m >= 2 : s + 1 < m);
    const int npt = seg ? a.per : (fits ? 1 : 0);
    const unsigned long long at = c0 + (unsigned long long)s * (unsigned)a.per;  // first point
    float p0[3] = {}, p1[3] = {}, p2[3] = {}, p3[3] = {};
    if (fits) sample_pos(a, r, s, p1);
    if (seg) {
      // closed: [P[m-1], P[0..m-1], P[0], P[1]]; open: [P[0], P[0..m-1], P[m-1]]
      auto wrap = [&](long long x) {
        if (r.closed) return x < 0 ? x + m : (x >= m ? x - m : x);
        return x < 0 ? 0ll : (x > m - 1 ? m - 1 : x);
      };
      sample_pos(a, r, wrap(s - 1), p0);
      sample_pos(a, r, wrap(s + 1), p2);
      sample_pos(a, r, wrap(s + 2), p3);
    }
    float len = 0.f, rest = 0.f;  // unevaluated sum of two (error-free additions)
    float prev[3] = {p1[0], p1[1], p1[2]};
    auto add_len = [&](const float q[3]) {
      float s2 = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float d = q[k] - prev[k];
        s2 = fmaf(d, d, s2);
        prev[k] = q[k];
      }
      const float d = sqrtf(s2), t = __fadd_rn(len, d), z = __fsub_rn(t, len);
      rest = __fadd_rn(rest, __fadd_rn(__fsub_rn(len, __fsub_rn(t, z)), __fsub_rn(d, z)));
      len = t;
    };
    const int most = __reduce_max_sync(0xffffffffu, npt);
    for (int t0 = 0; t0 < most; t0 += kStage) {
      const int left = max(0, min(npt - t0, kStage));  // points of this lane in the round
#pragma unroll
      for (int i = 0; i < kStage; ++i) {
        if (i >= left) break;
        float out[3] = {p1[0], p1[1], p1[2]};
        if (seg) {
          const float t = (float)(t0 + i) / (float)a.per, t2 = t * t, t3 = t2 * t;
#pragma unroll
          for (int k = 0; k < 3; ++k)
            out[k] = 0.5f * (2.f * p1[k] + t * (p2[k] - p0[k]) +
                             t2 * (2.f * p0[k] - 5.f * p1[k] + 4.f * p2[k] - p3[k]) +
                             t3 * (-p0[k] + 3.f * p1[k] - 3.f * p2[k] + p3[k]));
          if (t0 + i > 0) add_len(out);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) st[lane * kStagePitch + 3 * i + k] = out[k];
      }
      __syncwarp();
      const unsigned long long run = at + (unsigned)t0;
#pragma unroll 4
      for (int x = lane; x < 32 * 3 * kStage; x += 32) {
        const int l = x / (3 * kStage), f = x - l * (3 * kStage);
        const unsigned long long dst = __shfl_sync(0xffffffffu, run, l);
        const int n = __shfl_sync(0xffffffffu, left, l);
        if (f < 3 * n) a.curve[3 * dst + f] = st[l * kStagePitch + f];
      }
      __syncwarp();
    }
    if (seg) add_len(p2);
    // lengths: sums over the lanes of each piece of this warp
    for (unsigned long long q = lo; q < hi; ++q) {
      // (an infinite length has no rounding error: its rest is NaN)
      double v = act && p == q ? (double)len + (fabsf(len) <= 3.402823466e38f ? (double)rest : 0.0) : 0.0;
      v = warp_sum(v);
      if (lane == 0) {
        const unsigned long long f = a.efirst[q], end = f + a.count[q];
        if (a.cfirst[q] + a.npts[q] > a.curve_cap) continue;
        if (f < g0) a.left[c] = v;
        else if (end > g0 + 32) a.right[c] = v;
        else if (end > f) a.length[q] = (float)v;
      }
    }
  }
}

// lengths of the pieces that span warps of entries, one warp each (0 for a
// piece that does not fit)
__global__ void __launch_bounds__(LT) length_span_kernel(CurveArgs a) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long np = limit_n(a.np, a.np_dev);
  const unsigned long long warps = ((unsigned long long)gridDim.x * LT) >> 5;
  for (unsigned long long p = ((unsigned long long)blockIdx.x * LT + threadIdx.x) >> 5; p < np;
       p += warps) {
    const unsigned long long first = a.efirst[p], n = a.count[p];
    double sum = 0.0;
    if (n && a.cfirst[p] + a.npts[p] <= a.curve_cap) {
      if (first / 32 == (first + n - 1) / 32) continue;
      sum = spanning_sum(a.left, a.right, first, first + n, 32);
    }
    if ((threadIdx.x & 31) == 0) a.length[p] = (float)sum;
  }
}

// ---------------------------------------------------------------------------
// arc-length thinning of ordered pieces
// ---------------------------------------------------------------------------
constexpr double kThinUnit = 4294967296.0;  // arc-length units per length unit (2^32)

struct ThinArgs {
  const float* xyz;
  const uint32_t* nodes;
  const qtv_piece* pieces;
  unsigned long long np, ne;
  unsigned long long D;            // box length in arc-length units
  unsigned long long* v;           // per entry: rounded length of the segment ending there
  unsigned long long* X;           // exclusive scan of v
  uint32_t* flag;                  // per entry: starts a group
  unsigned long long* G;           // exclusive scan of flag
  float* out;
  unsigned long long out_cap;
  qtv_piece* out_pieces;
  const unsigned long long* total;  // groups (device)
};

// piece of node-list entry g (pieces are contiguous and in order)
__device__ __forceinline__ unsigned long long piece_of(const ThinArgs& a, unsigned long long g) {
  unsigned long long lo = 0, hi = a.np;
  while (hi - lo > 1) {
    const unsigned long long mid = (lo + hi) >> 1;
    if (a.pieces[mid].first <= g) lo = mid;
    else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ double coord(const ThinArgs& a, unsigned long long g, int c) {
  return (double)a.xyz[3ull * a.nodes[g] + c];
}

__global__ void thin_len_kernel(ThinArgs a) {
  pdl_wait();
  pdl_trigger();
  for (unsigned long long g = (unsigned long long)blockIdx.x * LT + threadIdx.x; g < a.ne;
       g += (unsigned long long)gridDim.x * LT) {
    const qtv_piece r = a.pieces[piece_of(a, g)];
    unsigned long long v = 0;
    if (g > r.first) {
      // FP64 length of the segment from the previous sample, summed in the
      // order ((dx^2 + dy^2) + dz^2) without contraction, then rounded
      const double dx = coord(a, g, 0) - coord(a, g - 1, 0);
      const double dy = coord(a, g, 1) - coord(a, g - 1, 1);
      const double dz = coord(a, g, 2) - coord(a, g - 1, 2);
      const double q = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
      v = (unsigned long long)__double2ll_rn(sqrt(q) * kThinUnit);
    }
    a.v[g] = v;
  }
}

__global__ void thin_flag_kernel(ThinArgs a) {
  pdl_wait();
  pdl_trigger();
  for (unsigned long long g = (unsigned long long)blockIdx.x * LT + threadIdx.x; g < a.ne;
       g += (unsigned long long)gridDim.x * LT) {
    const qtv_piece r = a.pieces[piece_of(a, g)];
    uint32_t f = 1;
    if (g > r.first) {
      const unsigned long long s = a.X[g] + a.v[g] - a.X[r.first];
      const unsigned long long sp = a.X[g - 1] + a.v[g - 1] - a.X[r.first];
      f = (s / a.D) != (sp / a.D) ? 1u : 0u;
    }
    a.flag[g] = f;
  }
}

__global__ void thin_mean_kernel(ThinArgs a) {
  pdl_wait();
  pdl_trigger();
  for (unsigned long long g = (unsigned long long)blockIdx.x * LT + threadIdx.x; g < a.ne;
       g += (unsigned long long)gridDim.x * LT) {
    if (!a.flag[g]) continue;
    const qtv_piece r = a.pieces[piece_of(a, g)];
    const unsigned long long end = r.first + r.count;
    double sx = 0.0, sy = 0.0, sz = 0.0;
    unsigned long long m = 0, e = g;
    do {
      sx = __dadd_rn(sx, coord(a, e, 0));
      sy = __dadd_rn(sy, coord(a, e, 1));
      sz = __dadd_rn(sz, coord(a, e, 2));
      ++m;
      ++e;
    } while (e < end && !a.flag[e]);
    const unsigned long long q = a.G[g];
    if (q < a.out_cap) {
      a.out[3 * q] = (float)(sx / (double)m);
      a.out[3 * q + 1] = (float)(sy / (double)m);
      a.out[3 * q + 2] = (float)(sz / (double)m);
    }
  }
}

__global__ void thin_pieces_kernel(ThinArgs a) {
  pdl_wait();
  pdl_trigger();
  for (unsigned long long p = (unsigned long long)blockIdx.x * LT + threadIdx.x; p < a.np;
       p += (unsigned long long)gridDim.x * LT) {
    qtv_piece r = a.pieces[p];
    const unsigned long long g0 = a.G[r.first];
    const unsigned long long g1 = p + 1 < a.np ? a.G[a.pieces[p + 1].first] : *a.total;
    r.first = g0;
    r.count = (uint32_t)(g1 - g0);
    a.out_pieces[p] = r;
  }
}

bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return false;
  return cs != cudaStreamCaptureStatusNone;
}

int ensure(qtv_handle h, size_t bytes, cudaStream_t st, void** out) {
  if (!h->lines) h->lines = new LineWork();
  LineWork* w = h->lines;
  if (bytes > w->cap) {
    if (capturing(st))
      return set_error(QTV_ERR_STATE, "line workspace must grow outside stream capture");
    cudaFree(w->buf);
    w->buf = nullptr;
    w->cap = 0;
    const cudaError_t e = cudaMalloc(&w->buf, bytes);
    if (e != cudaSuccess) return check_cuda(e, "cudaMalloc(line workspace)");
    w->cap = bytes;
  }
  *out = w->buf;
  return QTV_OK;
}

template <typename T>
T* carve(char*& p, unsigned long long count) {
  T* r = reinterpret_cast<T*>(p);
  p += ((count * sizeof(T) + 255) / 256) * 256;
  return r;
}

}  // namespace

int line_pieces_launch(qtv_handle h, uint64_t n, const uint64_t* n_dev, const uint32_t* nbr,
                       const uint8_t* deg, const uint32_t* comp, const float* xyz,
                       const uint64_t* face_ids, const int8_t* winding, qtv_piece* pieces,
                       uint64_t piece_cap, uint32_t* nodes, uint64_t node_cap, uint64_t* counts,
                       cudaStream_t st) {
  const unsigned long long ne = (unsigned long long)n * kSlots;
  // each piece holds at least one edge and adds at most two end samples to
  // its interior ones; edges <= 5 n (degree <= 10)
  const unsigned long long nodes_max = 11ull * n + 1;
  const unsigned long long nb = (n + SCHUNK - 1) / SCHUNK + 1;
  size_t bytes = 0;
  {
    // sizes must match the carve sequence below
    const unsigned long long sz[] = {n * 4, n, ne * 8, ne * 8, n * 4, n * 4, n * 8, n * 8, ne * 8,
                                     nodes_max * 4, (nodes_max / kNodeChunk + 1) * 8,
                                     (nodes_max / kNodeChunk + 1) * 8, nb * 16, 16,
                                     n * 4, n * 8, ne * 4, ne * 4, nb * 8, 8, kMaxRounds * 4 + 4};
    for (unsigned long long s : sz) bytes += ((s + 255) / 256) * 256;
  }
  void* buf = nullptr;
  int rc = ensure(h, bytes, st, &buf);
  if (rc) return rc;
  char* p = static_cast<char*>(buf);
  LineArgs a;
  a.n = n;
  a.n_dev = n_dev;
  a.nbr = nbr;
  a.deg = deg;
  a.comp = comp;
  a.xyz = xyz;
  a.face_ids = face_ids;
  a.winding = winding;
  a.cflags = carve<uint32_t>(p, n);
  a.special = carve<uint8_t>(p, n);
  a.jmp[0] = carve<uint2>(p, ne);
  a.jmp[1] = carve<uint2>(p, ne);
  a.pcount = carve<uint32_t>(p, n);
  a.plen = carve<uint32_t>(p, n);
  a.pfirst = carve<unsigned long long>(p, n);
  a.noff = carve<unsigned long long>(p, n);
  a.edge_node_off = carve<unsigned long long>(p, ne);
  a.tmp_nodes = carve<uint32_t>(p, nodes_max);
  a.left = carve<double>(p, nodes_max / kNodeChunk + 1);
  a.right = carve<double>(p, nodes_max / kNodeChunk + 1);
  unsigned long long* bs1 = carve<unsigned long long>(p, 2 * nb);
  unsigned long long* tot = carve<unsigned long long>(p, 2);
  a.deg32 = carve<uint32_t>(p, n);
  a.aoff = carve<unsigned long long>(p, n);
  a.atail = carve<uint32_t>(p, ne);
  a.ahead = carve<uint32_t>(p, ne);
  unsigned long long* bs3 = carve<unsigned long long>(p, nb);
  unsigned long long* narcs = carve<unsigned long long>(p, 1);
  a.narcs = narcs;
  a.live = carve<uint32_t>(p, kMaxRounds + 1);
  a.fbuf = a.live + kMaxRounds;
  a.pieces = pieces;
  a.piece_cap = piece_cap;
  a.nodes = nodes;
  a.node_cap = node_cap;

  long long g = ((long long)n + LT - 1) / LT;
  if (g > (long long)h->num_sms * 16) g = (long long)h->num_sms * 16;
  if (g < 1) g = 1;
  long long ge = ((long long)ne + LT - 1) / LT;
  if (ge > (long long)h->num_sms * 32) ge = (long long)h->num_sms * 32;
  if (ge < 1) ge = 1;
  TraceScope ts(h, K_LINES, st);
  launch_dependent(stats_init_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  launch_dependent(stats_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  launch_dependent(special_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  // compact directed edges: offsets by an exclusive scan of the degrees
  scan<uint32_t>(a.deg32, nullptr, n_dev, n, a.aoff, nullptr, bs3, narcs, nullptr, st);
  launch_dependent(arcs_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  launch_dependent(edges_init_kernel, dim3((unsigned)ge), dim3(LT), 0, st, a);
  int rounds = 0;
  for (unsigned long long reach = 1; reach < (unsigned long long)n + 1; reach *= kHops) ++rounds;
  if (rounds < 1) rounds = 1;
  cudaError_t e = cudaMemsetAsync(a.live, 0, (kMaxRounds + 1) * sizeof(uint32_t), st);
  if (e != cudaSuccess) return check_cuda(e, "cudaMemsetAsync(line rounds)");
  for (int r = 0; r < rounds; ++r)
    launch_dependent(jump_kernel, dim3((unsigned)ge), dim3(LT), 0, st, a, r & 1, r);
  launch_dependent(count_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  scan<uint32_t>(a.pcount, a.plen, n_dev, n, a.pfirst, a.noff, bs1, tot, tot + 1, st);
  e = cudaMemcpyAsync(counts, tot, 2 * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return check_cuda(e, "cudaMemcpyAsync(line counts)");
  launch_dependent(pieces_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  launch_dependent(interior_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  launch_dependent(orient_kernel, dim3(h->num_sms * 8), dim3(LT), 0, st, a, tot);
  launch_dependent(place_kernel, dim3(h->num_sms * 8), dim3(LT), 0, st, a, tot);
  e = cudaGetLastError();
  return check_cuda(e, "line pieces launch");
}

int piece_curves_launch(qtv_handle h, const float* xyz, const uint32_t* nodes,
                        const qtv_piece* pieces, uint64_t np, const uint64_t* np_dev, int per,
                        float* curve, uint64_t curve_cap, uint64_t* curve_first, float* length,
                        uint64_t* total, cudaStream_t st) {
  const unsigned long long nb = (np + SCHUNK - 1) / SCHUNK + 1;
  const unsigned long long pc = curve_cap / 32 + 1;  // warps of samples whose points fit
  size_t bytes = 0;
  const unsigned long long sz[] = {np * 4, np * 4, np * 8, nb * 16, pc * 8, pc * 8, 8};
  for (unsigned long long x : sz) bytes += (x + 255) / 256 * 256;
  void* buf = nullptr;
  int rc = ensure(h, bytes, st, &buf);
  if (rc) return rc;
  char* p = static_cast<char*>(buf);
  CurveArgs a;
  a.xyz = xyz;
  a.nodes = nodes;
  a.pieces = pieces;
  a.np = np;
  a.np_dev = np_dev;
  a.per = per;
  a.npts = carve<uint32_t>(p, np);
  a.count = carve<uint32_t>(p, np);
  a.efirst = carve<unsigned long long>(p, np);
  unsigned long long* bs = carve<unsigned long long>(p, 2 * nb);
  a.left = carve<double>(p, pc);
  a.right = carve<double>(p, pc);
  unsigned long long* entries = carve<unsigned long long>(p, 1);
  a.entries = entries;
  a.cfirst = reinterpret_cast<unsigned long long*>(curve_first);
  a.curve = curve;
  a.curve_cap = curve_cap;
  a.length = length;
  long long g = ((long long)np + LT - 1) / LT;
  if (g > (long long)h->num_sms * 16) g = (long long)h->num_sms * 16;
  if (g < 1) g = 1;
  TraceScope ts(h, K_CURVES, st);
  launch_dependent(curve_count_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  scan<uint32_t>(a.npts, a.count, np_dev, np, a.cfirst, a.efirst, bs,
                 reinterpret_cast<unsigned long long*>(total), entries, st);
  if (curve_cap > 0) launch_dependent(curve_kernel, dim3(h->num_sms * 8), dim3(LT), 0, st, a);
  launch_dependent(length_span_kernel, dim3(h->num_sms * 4), dim3(LT), 0, st, a);
  const cudaError_t e = cudaGetLastError();
  return check_cuda(e, "piece curves launch");
}

int thin_pieces_launch(qtv_handle h, const float* xyz, const uint32_t* nodes,
                       const qtv_piece* pieces, uint64_t np, uint64_t nnodes, float box,
                       float* out_xyz, uint64_t out_cap, qtv_piece* out_pieces, uint64_t* total,
                       cudaStream_t st) {
  const unsigned long long ne = nnodes;
  const unsigned long long nb = (ne + SCHUNK - 1) / SCHUNK + 1;
  const unsigned long long sz[] = {ne * 8, ne * 8, ne * 4, ne * 8, nb * 8, nb * 8, 16};
  size_t bytes = 0;
  for (unsigned long long x : sz) bytes += ((x + 255) / 256) * 256;
  void* buf = nullptr;
  int rc = ensure(h, bytes, st, &buf);
  if (rc) return rc;
  char* p = static_cast<char*>(buf);
  ThinArgs a;
  a.xyz = xyz;
  a.nodes = nodes;
  a.pieces = pieces;
  a.np = np;
  a.ne = ne;
  const double Dd = (double)box * kThinUnit;
  a.D = Dd >= 1.0 ? (unsigned long long)llrint(Dd) : 1ull;
  a.v = carve<unsigned long long>(p, ne);
  a.X = carve<unsigned long long>(p, ne);
  a.flag = carve<uint32_t>(p, ne);
  a.G = carve<unsigned long long>(p, ne);
  unsigned long long* bs1 = carve<unsigned long long>(p, nb);
  unsigned long long* bs2 = carve<unsigned long long>(p, nb);
  unsigned long long* tots = carve<unsigned long long>(p, 2);
  a.out = out_xyz;
  a.out_cap = out_cap;
  a.out_pieces = out_pieces;
  a.total = tots + 1;
  long long g = ((long long)ne + LT - 1) / LT;
  if (g > (long long)h->num_sms * 16) g = (long long)h->num_sms * 16;
  if (g < 1) g = 1;
  long long gp = ((long long)np + LT - 1) / LT;
  if (gp > (long long)h->num_sms * 16) gp = (long long)h->num_sms * 16;
  if (gp < 1) gp = 1;
  TraceScope ts(h, K_THIN, st);
  launch_dependent(thin_len_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  scan<unsigned long long>(a.v, nullptr, nullptr, ne, a.X, nullptr, bs1, tots, nullptr, st);
  launch_dependent(thin_flag_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  scan<uint32_t>(a.flag, nullptr, nullptr, ne, a.G, nullptr, bs2, tots + 1, nullptr, st);
  launch_dependent(thin_mean_kernel, dim3((unsigned)g), dim3(LT), 0, st, a);
  launch_dependent(thin_pieces_kernel, dim3((unsigned)gp), dim3(LT), 0, st, a);
  cudaError_t e = cudaMemcpyAsync(total, tots + 1, sizeof(uint64_t), cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaGetLastError();
  return check_cuda(e, "thin pieces launch");
}

}  // namespace qtv
