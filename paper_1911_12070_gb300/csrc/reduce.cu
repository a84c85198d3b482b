// reduce.cu -- box-mean reduction of a sample graph (Sec. 3.3.1-3.3.2) on the
// GPU, in an order-independent lattice form.
//
// The paper walks the graph: a box of side d centred on the current node takes
// the unprocessed nodes it reaches inside the box, they collapse to their mean
// with their external edges inherited, the walk moves on to an unprocessed
// neighbour, and whole passes repeat until positions settle (2 to 5 passes).
// That walk is sequential.  Here every pass is data-parallel instead: a
// lattice of boxes of side D covers space (shifted by D/2 in every axis on
// odd passes, so that no lattice boundary stays fixed), the nodes of one box
// that are connected through edges inside the box form one cluster, and each
// cluster collapses to one node at the mean of its members, keeping every
// edge that leaves it.  Passes repeat until one pass of each lattice merges
// nothing; then no further pass can change anything.
//
// Exactness.  Positions are held as 64-bit integers in units of 2^-32 of the
// input's length unit (x 2^32, exact in FP64 for an FP32 x, rounded to the
// nearest integer with ties to even; negative positions too);
// box keys are floor divisions of integers and a mean is the rounded integer
// quotient floor((sum + floor(c/2)) / c), so sums and means do not depend on the order in
// which threads add, and the result is the same on every run.
//
// Representation.  A cluster is represented by its node of lowest input index,
// which holds its position; nl[u] is the node that u went under when its cluster
// merged (u itself for a representative), so the cluster of any node is a walk
// of at most one step per pass.  Each pass works on two compact lists, the
// representatives and the edges between different clusters (with their ends
// renamed; exactly the inherited connectivity of the paper's collapse), which
// shrink as clusters merge: it links every edge whose ends have equal keys
// (union-find, as in graph.cu: the larger root goes under the smaller with a
// CAS, so roots are cluster minima), sums the members' positions, and lists the
// surviving representatives, with their means and their keys in the next
// lattice, and edges anew.  The order of the lists depends on timing, the
// results do not.  An edge list that outgrows its buffer (denser graphs than
// any of lines) is dropped and the pass reads the input edges through the walks.
//
// Bound by the latency of gathers from L2.  Scanning all nodes and input edges
// in every pass took 0.47 ms of device time for the 594e3 samples of a 384^3
// field (10 passes launched, 7 made); the lists take 0.40 ms
// (the first pass, over all nodes, 0.15 of them).
//
// Launches: one set-up kernel, then for each of max_passes passes a fixed
// sequence of three kernels; once two passes were quiet every later kernel
// returns at once, so the call synchronises nothing and can be captured into a
// CUDA graph.  A launch gets its pass as an argument and each pass has counters
// of its own, written by earlier launches than the ones that read them: a block
// may start after others of its launch have finished, so none may act on a
// word that its own launch rewrites.  Each kernel is
// launched behind the previous one (pdl_wait), as those of graph.cu and lines.cu:
// about sixty short launches of a vectorization, 1360 -> 1265 us at 384^3.
#include "qtv_internal.cuh"

namespace qtv {

struct ReduceWork {
  long long* sum = nullptr;        // [cap][3] cluster sums of one pass (two's complement)
  unsigned int* cnt = nullptr;     // [cap] members of a new cluster
  unsigned long long* key = nullptr;  // [cap] packed box key of a representative
  unsigned int* par = nullptr;     // [cap] union-find parents of one pass
  unsigned int* nl = nullptr;      // [cap] the node that a node merged into
  unsigned int* reps[2] = {nullptr, nullptr};  // [cap] representatives, by pass parity
  uint2* edges[2] = {nullptr, nullptr};        // [kEdgesPerNode cap] edges between clusters
  unsigned long long* status = nullptr;  // kStatus*
  uint64_t cap = 0;
};

void reduce_work_free(ReduceWork* w) {
  if (!w) return;
  cudaFree(w->sum);
  cudaFree(w->cnt);
  cudaFree(w->key);
  cudaFree(w->par);
  cudaFree(w->nl);
  for (int i = 0; i < 2; ++i) {
    cudaFree(w->reps[i]);
    cudaFree(w->edges[i]);
  }
  cudaFree(w->status);
  delete w;
}

namespace {

constexpr int RT = 256;
// Room of an edge list: line graphs have about an edge a node, the graph of vortex
// nodes (6-connectivity) 1.7, most of them between clusters still after a pass of
// small boxes.  With room for one a node such passes fell to the input edges: 1.45e6
// vortex nodes of 384^3 at box 1.5, 1147 us, now 925 (1072 without lists); room for
// three gave 919.
constexpr uint64_t kEdgesPerNode = 2;
constexpr int kMaxTries = 1 << 20;     // CAS retries of one link before giving up
constexpr uint32_t kNoNode = 0xFFFFFFFFu;
constexpr double kFix = 4294967296.0;  // fixed-point units per length unit

constexpr int kMostPasses = 64;

// status words; a pass starts with the lists that the pass before it left
enum {
  kGaveUp = 0,                               // a bounded retry loop ran out
  kMerges,                                   // [pass]
  kNumReps = kMerges + kMostPasses,          // [pass], and after the last one
  kNumEdges = kNumReps + kMostPasses + 1,    // above the buffer: no list, use the input edges
  kStatusWords = kNumEdges + kMostPasses + 1
};
static_assert(kStatusWords <= RT, "one block sets them");

struct ReduceArgs {
  unsigned long long n;
  const uint64_t* n_dev;
  const uint32_t* nbr;
  const uint8_t* deg;
  int stride;
  long long D;          // box side in fixed point
  int max_passes;
  long long* q;         // [n][3] positions (valid at representatives)
  long long* sum;
  unsigned int* cnt;
  unsigned long long* key;
  unsigned int* par;
  unsigned int* nl;
  unsigned int* reps[2];
  uint2* edges[2];
  unsigned long long edge_cap;
  unsigned long long* status;
};

__device__ __forceinline__ unsigned long long limit_n(unsigned long long n, const uint64_t* n_dev) {
  if (n_dev) {
    const unsigned long long d = *n_dev;
    if (d < n) n = d;
  }
  return n;
}

// two passes before this one were quiet: it is not made (and merges nothing, so the
// ones after it are not either)
__device__ __forceinline__ bool done(const ReduceArgs& a, int pass) {
  return pass >= 2 && (a.status[kMerges + pass - 1] | a.status[kMerges + pass - 2]) == 0ull;
}

// floor(x / d) for d > 0
__device__ __forceinline__ long long floor_div(long long x, long long d) {
  const long long qt = x / d;
  return (x % d != 0 && x < 0) ? qt - 1 : qt;
}

// 21 bits per axis (two's complement), enough for any grid below 2^20 boxes
__device__ __forceinline__ unsigned long long pack_key(long long kx, long long ky, long long kz) {
  const unsigned long long m = (1ull << 21) - 1ull;
  return ((unsigned long long)kx & m) | (((unsigned long long)ky & m) << 21) |
         (((unsigned long long)kz & m) << 42);
}

// representative u starts a pass whose lattice is shifted (odd) or not: its box
// key, a fresh union-find parent, zero sums
__device__ __forceinline__ void start_pass(const ReduceArgs& a, unsigned long long u, bool odd,
                                           const long long q[3]) {
  const long long off = odd ? a.D / 2 : 0;
  a.key[u] = pack_key(floor_div(q[0] - off, a.D), floor_div(q[1] - off, a.D),
                      floor_div(q[2] - off, a.D));
  a.par[u] = (uint32_t)u;
  a.sum[3 * u] = a.sum[3 * u + 1] = a.sum[3 * u + 2] = 0;
  a.cnt[u] = 0u;
}

__global__ void __launch_bounds__(RT) reduce_init_kernel(ReduceArgs a, const float* xyz) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  if (blockIdx.x == 0 && threadIdx.x < kStatusWords) {
    // every node is a representative; no edge list yet
    const int i = threadIdx.x;
    a.status[i] = i == kNumReps ? nn : (i == kNumEdges ? ~0ull : 0ull);
  }
  for (unsigned long long u = (unsigned long long)blockIdx.x * RT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * RT) {
    long long q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) a.q[3 * u + c] = q[c] = __double2ll_rn((double)xyz[3 * u + c] * kFix);
    a.nl[u] = (uint32_t)u;
    a.reps[0][u] = (uint32_t)u;
    start_pass(a, u, false, q);
  }
}

__device__ __forceinline__ uint32_t find_root(uint32_t* parent, uint32_t x) {
  uint32_t p = *((volatile uint32_t*)parent + x);
  while (p != x) {
    const uint32_t g = *((volatile uint32_t*)parent + p);
    if (g != p) *((volatile uint32_t*)parent + x) = g;  // halving: parents only decrease
    x = p;
    p = g;
  }
  return x;
}

__device__ __forceinline__ uint32_t find_root_ro(const uint32_t* parent, uint32_t x) {
  uint32_t p = *((const volatile uint32_t*)parent + x);
  while (p != x) {
    x = p;
    p = *((const volatile uint32_t*)parent + x);
  }
  return x;
}

// the cluster of node u (read-only walk)
__device__ __forceinline__ uint32_t cluster_of(const ReduceArgs& a, uint32_t u) {
  return find_root_ro(a.nl, u);
}

// f(ends) for the input edges (u, v), u < v, that join different clusters
template <typename F>
__device__ __forceinline__ void node_edges(const ReduceArgs& a, unsigned long long nn,
                                           unsigned long long u, F f) {
  const int m = a.deg[u];
  uint32_t lu = kNoNode;
  for (int x = 0; x < m; ++x) {
    const uint32_t v = a.nbr[u * (unsigned long long)a.stride + x];
    if (v <= (uint32_t)u || v >= nn) continue;
    if (lu == kNoNode) lu = cluster_of(a, (uint32_t)u);
    const uint32_t lv = cluster_of(a, v);
    if (lv != lu) f(make_uint2(lu, lv));
  }
}

// f(ends) for the calling thread's share of the edges between clusters of this
// pass: from the list, or, without one, the input edges
template <typename F>
__device__ __forceinline__ void for_edges(const ReduceArgs& a, unsigned long long nn, int pass, F f) {
  const unsigned long long ne = a.status[kNumEdges + pass];
  const unsigned long long t0 = (unsigned long long)blockIdx.x * RT + threadIdx.x;
  const unsigned long long step = (unsigned long long)gridDim.x * RT;
  if (ne <= a.edge_cap) {
    for (unsigned long long e = t0; e < ne; e += step) f(a.edges[pass & 1][e]);
    return;
  }
  for (unsigned long long u = t0; u < nn; u += step) node_edges(a, nn, u, f);
}

// every edge between two clusters of equal key
__global__ void __launch_bounds__(RT) reduce_link_kernel(ReduceArgs a, int pass) {
  pdl_wait();
  pdl_trigger();
  if (done(a, pass)) return;
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  for_edges(a, nn, pass, [&](uint2 e) {
    if (a.key[e.x] != a.key[e.y]) return;
    int tries = 0;
    while (true) {
      uint32_t ra = find_root(a.par, e.x), rb = find_root(a.par, e.y);
      if (ra == rb) break;
      if (ra > rb) {
        const uint32_t t = ra;
        ra = rb;
        rb = t;
      }
      if (atomicCAS(a.par + rb, rb, ra) == rb) break;
      if (++tries >= kMaxTries) {
        atomicOr(a.status + kGaveUp, 1ull);
        break;
      }
    }
  });
}

// representatives: the root (lowest index of the merged cluster), and the
// position added to the new cluster's sum
__global__ void __launch_bounds__(RT) reduce_merge_kernel(ReduceArgs a, int pass) {
  pdl_wait();
  pdl_trigger();
  if (done(a, pass)) return;
  const int cur = pass & 1;
  const unsigned long long nr = a.status[kNumReps + pass];
  unsigned long long merges = 0;
  for (unsigned long long i = (unsigned long long)blockIdx.x * RT + threadIdx.x; i < nr;
       i += (unsigned long long)gridDim.x * RT) {
    const uint32_t u = a.reps[cur][i];
    const uint32_t r = find_root_ro(a.par, u);
    a.nl[u] = r;
    merges += r != u ? 1ull : 0ull;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      atomicAdd(reinterpret_cast<unsigned long long*>(a.sum + 3ull * r + c),
                (unsigned long long)a.q[3ull * u + c]);
    atomicAdd(a.cnt + r, 1u);
  }
#pragma unroll
  for (int d = 16; d; d >>= 1) merges += __shfl_down_sync(0xffffffffu, merges, d);
  if ((threadIdx.x & 31) == 0 && merges) atomicAdd(a.status + kMerges + pass, merges);
}

// First place in a list for the k entries of the calling thread: one atomic a
// block and call (all threads call; one atomic a warp made the counters' lines
// the bottleneck).
__device__ __forceinline__ unsigned long long append(unsigned long long* count, uint32_t k) {
  __shared__ uint32_t part[RT / 32];
  __shared__ unsigned long long base;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t inc = k;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= d) inc += t;
  }
  __syncthreads();  // part and base may still be read
  if (lane == 31) part[w] = inc;
  __syncthreads();
  uint32_t before = 0, total = 0;
#pragma unroll
  for (int i = 0; i < RT / 32; ++i) {
    if (i < w) before += part[i];
    total += part[i];
  }
  if (threadIdx.x == 0 && total) base = atomicAdd(count, (unsigned long long)total);
  __syncthreads();
  return base + before + inc - k;
}

// The next pass's lists: surviving representatives with the rounded mean of
// their cluster and their key in its lattice, and the edges that still join
// different clusters.
__global__ void __launch_bounds__(RT) reduce_list_kernel(ReduceArgs a, int pass) {
  pdl_wait();
  pdl_trigger();
  if (done(a, pass)) return;
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  const int cur = pass & 1, next = cur ^ 1;
  const unsigned long long nr = a.status[kNumReps + pass], ne = a.status[kNumEdges + pass];
  unsigned long long* const nreps = a.status + kNumReps + pass + 1;
  unsigned long long* const nedges = a.status + kNumEdges + pass + 1;
  const unsigned long long b0 = (unsigned long long)blockIdx.x * RT, step = (unsigned long long)gridDim.x * RT;
  for (unsigned long long i0 = b0; i0 < nr; i0 += step) {
    const unsigned long long i = i0 + threadIdx.x;
    const uint32_t u = i < nr ? a.reps[cur][i] : 0u;
    const bool stays = i < nr && a.nl[u] == u;
    const unsigned long long at = append(nreps, stays ? 1u : 0u);
    if (!stays) continue;
    a.reps[next][at] = u;
    const long long c = (long long)a.cnt[u];
    long long q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) a.q[3ull * u + k] = q[k] = floor_div(a.sum[3ull * u + k] + c / 2, c);
    start_pass(a, u, next != 0, q);
  }
  if (ne <= a.edge_cap) {
    for (unsigned long long i0 = b0; i0 < ne; i0 += step) {
      const unsigned long long i = i0 + threadIdx.x;
      uint2 e = i < ne ? a.edges[cur][i] : make_uint2(0u, 0u);
      e.x = a.nl[e.x];
      e.y = a.nl[e.y];
      const unsigned long long at = append(nedges, e.x != e.y ? 1u : 0u);
      if (e.x != e.y && at < a.edge_cap) a.edges[next][at] = e;
    }
  } else {
    for (unsigned long long i0 = b0; i0 < nn; i0 += step) {
      const unsigned long long u = i0 + threadIdx.x;
      uint32_t k = 0;
      if (u < nn) node_edges(a, nn, u, [&](uint2) { ++k; });
      unsigned long long at = append(nedges, k);
      if (k)
        node_edges(a, nn, u, [&](uint2 e) {
          if (at < a.edge_cap) a.edges[next][at] = e;
          ++at;
        });
    }
  }
}

// labels of all nodes; representatives: positions back to the length unit
// (exact in FP64); counts = (clusters, passes)
__global__ void __launch_bounds__(RT) reduce_out_kernel(ReduceArgs a, uint32_t* __restrict__ label,
                                                        double* __restrict__ out, uint64_t* counts) {
  pdl_wait();
  pdl_trigger();
  const unsigned long long nn = limit_n(a.n, a.n_dev);
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    int passes = a.max_passes;  // the first that was not made
    for (int p = threadIdx.x; p < a.max_passes; p += 32)
      if (done(a, p)) {
        passes = p;
        break;
      }
    passes = __reduce_min_sync(0xffffffffu, passes);
    if (threadIdx.x == 0) {
      counts[0] = a.status[kGaveUp] ? QTV_COUNT_TIMEOUT : a.status[kNumReps + passes];
      counts[1] = (uint64_t)passes;
    }
  }
  for (unsigned long long u = (unsigned long long)blockIdx.x * RT + threadIdx.x; u < nn;
       u += (unsigned long long)gridDim.x * RT) {
    const uint32_t r = cluster_of(a, (uint32_t)u);
    label[u] = r;
    if (r != (uint32_t)u) continue;
#pragma unroll
    for (int c = 0; c < 3; ++c) out[3 * u + c] = (double)a.q[3 * u + c] / kFix;
  }
}

bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return false;
  return cs != cudaStreamCaptureStatusNone;
}

}  // namespace

int box_reduce_launch(qtv_handle h, uint64_t n, const uint64_t* n_dev, const uint32_t* nbr,
                      const uint8_t* deg, int stride, const float* xyz, float box, int max_passes,
                      uint32_t* label, double* out_xyz, uint64_t* counts, cudaStream_t st) {
  if (!h->reduce || h->reduce->cap < n) {
    if (capturing(st))
      return set_error(QTV_ERR_STATE, "reduction workspace must grow outside stream capture");
    reduce_work_free(h->reduce);
    h->reduce = nullptr;
    ReduceWork* w = new ReduceWork();
    const uint64_t c = n > 0 ? n : 1;
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&w->sum), c * 3 * sizeof(long long));
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&w->cnt), c * sizeof(unsigned int));
    if (e == cudaSuccess)
      e = cudaMalloc(reinterpret_cast<void**>(&w->key), c * sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&w->par), c * sizeof(unsigned int));
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&w->nl), c * sizeof(unsigned int));
    for (int i = 0; i < 2; ++i) {
      if (e == cudaSuccess)
        e = cudaMalloc(reinterpret_cast<void**>(&w->reps[i]), c * sizeof(unsigned int));
      if (e == cudaSuccess)
        e = cudaMalloc(reinterpret_cast<void**>(&w->edges[i]), kEdgesPerNode * c * sizeof(uint2));
    }
    if (e == cudaSuccess)
      e = cudaMalloc(reinterpret_cast<void**>(&w->status), kStatusWords * sizeof(unsigned long long));
    if (e != cudaSuccess) {
      reduce_work_free(w);
      return check_cuda(e, "cudaMalloc(reduction workspace)");
    }
    w->cap = c;
    h->reduce = w;
  }
  ReduceWork* w = h->reduce;
  if (n == 0)
    return check_cuda(cudaMemsetAsync(counts, 0, 2 * sizeof(uint64_t), st),
                      "cudaMemsetAsync(reduction counts)");
  ReduceArgs a;
  a.n = n;
  a.n_dev = n_dev;
  a.nbr = nbr;
  a.deg = deg;
  a.stride = stride;
  a.D = (long long)((double)box * kFix);
  a.max_passes = max_passes;
  // positions live in the output array as fixed-point integers until the end
  a.q = reinterpret_cast<long long*>(out_xyz);
  a.sum = w->sum;
  a.cnt = w->cnt;
  a.key = w->key;
  a.par = w->par;
  a.nl = w->nl;
  for (int i = 0; i < 2; ++i) {
    a.reps[i] = w->reps[i];
    a.edges[i] = w->edges[i];
  }
  a.edge_cap = kEdgesPerNode * w->cap;
  a.status = w->status;
  long long blocks = ((long long)n + RT - 1) / RT;
  if (blocks > (long long)h->num_sms * 8) blocks = (long long)h->num_sms * 8;
  TraceScope ts(h, K_REDUCE, st);
  launch_dependent(reduce_init_kernel, dim3((unsigned)blocks), dim3(RT), 0, st, a, xyz);
  for (int p = 0; p < max_passes; ++p) {
    launch_dependent(reduce_link_kernel, dim3((unsigned)blocks), dim3(RT), 0, st, a, p);
    launch_dependent(reduce_merge_kernel, dim3((unsigned)blocks), dim3(RT), 0, st, a, p);
    launch_dependent(reduce_list_kernel, dim3((unsigned)blocks), dim3(RT), 0, st, a, p);
  }
  launch_dependent(reduce_out_kernel, dim3((unsigned)blocks), dim3(RT), 0, st, a, label, out_xyz,
                   counts);
  const cudaError_t e = cudaGetLastError();
  return check_cuda(e, "box reduction launch");
}

}  // namespace qtv
