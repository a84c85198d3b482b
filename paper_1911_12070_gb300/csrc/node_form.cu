// node_form.cu -- the node form of the circulation (Sec. 2.2.2) and the
// density error of Eq. 7 (Sec. 5) on the GPU.
//
// Node form.  For every node and each of the three grid planes through it, the
// circulation of Eq. 5 around the ring of the node's eight in-plane neighbours
// (the 2h x 2h square centred on the node, counter-clockwise about the plane
// normal; (u, v) = (x, y), (y, z), (z, x) for the planes xy, yz, zx), as the
// integer S = C / (2 pi).  A node is a vortex node when the largest |C| of its
// three planes exceeds pi, i.e. when some S != 0.  S = 0 where the ring leaves
// the grid or passes through a NaN/Inf node (the node itself is not on its
// ring).
//
// Arithmetic.  Every directed edge a -> b contributes the integer branch
// crossing r (its wrapped phase difference minus theta_b - theta_a, over
// 2 pi), decided from the sign bits of Im a, Im b and the sign of the
// determinant Re a Im b - Im a Re b; the theta terms telescope around the
// ring, so S is the sum of the ring's eight r.  Each grid edge is evaluated once,
// in its forward direction, and a ring that runs it backwards adds -r (the
// argument of the conjugate is the exact negation).  The ring encloses the four
// plaquettes of its plane at the node, and the edges between them cancel, so S is
// the sum of their four-edge sums, whatever the r are:
//   W_xy(i,j) = r_x(i,j) + r_y(i+1,j) - r_x(i,j+1) - r_y(i,j), and so on,
//   S_xy(i,j) = W_xy(i-1,j-1) + W_xy(i,j-1) + W_xy(i-1,j) + W_xy(i,j),
// and each W serves four rings.  The sums are kept mod 8: S in [-3, 4], exact
// because only a ring whose eight differences are all exact +-pi ties reaches
// |S| = 4 (read as 4).
//
// Layout (bit-sliced).  A warp owns 30 columns (lanes 1..30; lanes 0 and 31
// hold the neighbour columns) of a band of NB = 18 rows, and each lane keeps
// one bit per row (rows j0 - 1 .. j0 + NB, halo rows included) in words: the
// sign bit of Im psi and the sign bits of the FP32 cross products of its x, y
// and z edges, as the identification sweep does.  An edge term is +1 when s_a =
// 0, s_b = 1 and the cross sign is 0, -1 when s_a = 1, s_b = 0 and the sign is 1;
// edges that touch a zero node count 0.  W and S are three words each; adding
// two of them is five 3-input operations.  The warp marches z over a chunk of
// planes, streaming each lane's column through a 2-slot ring in shared memory
// with cp.async; the previous plane's values stay in registers.
//
// Output.  Vortex nodes in ascending linear node index with their three S: each
// lane with vortex nodes in a sub-band of 9 rows of a step stages one record, its
// S words there, contiguously in a chunk of the staging buffer that the warp
// reserved (one atomic per chunk), and the step writes a table entry {staging
// base, lane mask} per sub-band; after an exclusive scan of the (plane, sub-band)
// totals one warp per (plane, sub-band) lists the nodes row by row.  Optionally the dense S field [3][nz][ny][nx].
//
// Bound by issue (69% of the slots taken).  With eight ring terms added per ring, records per node and
// the previous plane read from shared memory it took 3.2 warp instructions a
// node and 218 us at 384^3, the scatter 63; now 140 and 35 (512^3: 500 and 110,
// now 298 and 64).
//
// Density error.  e = sum_q |rho(p_q)| / (n rho_bar), rho the density |psi|^2
// of the trilinearly interpolated field at the sample points, rho_bar the mean
// density over all nodes.  Sums run in FP32 over short runs and in FP64 across
// runs, over a partition fixed by the launch shape, so a call is reproducible.
#include <algorithm>
#include <cstdio>

#include "qtv_internal.cuh"

namespace qtv {

struct NodeWork {
  uint4* recs = nullptr;               // staged records: words 0..3
  uint64_t recs_cap = 0;
  uint32_t* recs4 = nullptr;           // word 4
  uint64_t recs4_cap = 0;
  uint2* table = nullptr;              // per (plane, band, column segment)
  uint64_t table_cap = 0;
  unsigned int* segtot = nullptr;      // vortex nodes per (plane, band)
  uint64_t segtot_cap = 0;
  unsigned long long* seg_off = nullptr;
  uint64_t seg_off_cap = 0;
  unsigned long long* top = nullptr;   // staging bump counter, work item counter, sums of the scan
  double* partial = nullptr;           // density sums per block
  uint64_t partial_cap = 0;
  int resident_warps = 0;
};

void node_work_free(NodeWork* w) {
  if (!w) return;
  cudaFree(w->recs);
  cudaFree(w->recs4);
  cudaFree(w->table);
  cudaFree(w->segtot);
  cudaFree(w->seg_off);
  cudaFree(w->top);
  cudaFree(w->partial);
  delete w;
}

namespace {

// Rows, warps and slots: the copies pass through the L1 cache, which gets what
// shared memory leaves; 200 KB of rings a multiprocessor slow them (384^3: 17 rows,
// 16 warps, 3 slots, 209 KB 182 us; 22, 12, 3, 203 KB 188).  More rows a lane share
// the word logic: 20 rows, 16 warps, 2 slots, 164 KB 140 us; 18, 16, 2 140; 20, 12,
// 3 146; 32, 8, 2 145; 24, 10, 3 152.
constexpr int NT = 20;          // rows held: bit t = row j0 - 1 + t
constexpr int NB = NT - 2;      // owned rows per band: bits 1..NB
constexpr uint32_t kOwnedRows = (1u << (NB + 1)) - 2u;
constexpr uint32_t kRowsHeld = (1u << NT) - 1u;
constexpr int NSUB = 2;         // sub-bands of a band: the output's segments
constexpr int SUBR = NB / NSUB; // rows of a sub-band
constexpr uint32_t kSubRows = (2u << SUBR) - 2u;  // bits 1..SUBR
constexpr int NCOL = 30;        // owned columns per warp (lanes 1..30)
constexpr int NODE_WARPS = 4;   // warps per CTA
constexpr int kSlots = 2;       // plane slots of a warp's ring: p, p + 1
constexpr long long kItemsPerWarp = 4;  // work items per resident warp
constexpr uint32_t kChunk = 1024;  // staging records a warp reserves at a time (20 KB)
constexpr int kSlotLen = NT * 32;  // elements of a slot: rows of the warp's 32 columns
__host__ __device__ constexpr int slot_at(int t) { return t * 32; }  // of lane 0
constexpr size_t kNodeSmem = (size_t)NODE_WARPS * kSlots * kSlotLen * sizeof(float2);
static_assert(SUBR * NSUB == NB && SUBR < 16, "sub-bands fill a band, 16 bits a row word of a record");
constexpr int DENS_THREADS = 256;
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ bool fin(float v) { return fabsf(v) <= 3.402823466e38f; }

// acc' = (acc << 1) | sign bit of x
__device__ __forceinline__ uint32_t push1(uint32_t acc, float x) {
  return __funnelshift_l(__float_as_uint(x), acc, 1);
}

// FP32 value of Re a Im b - Im a Re b with one rounding of the second product
// absorbed by the FMA; its sign bit decides the edge term
__device__ __forceinline__ float cross_f(float2 a, float2 b) { return fmaf(a.x, b.y, -(a.y * b.x)); }

// packed product of the (Re, Im) values: zero if a component of a node is
// zero, non-finite if a node is (or on FP32 under- or overflow, which merely
// selects the masking path)
__device__ __forceinline__ unsigned long long prod_step(unsigned long long acc, float2 v) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;"
      : "=l"(d)
      : "l"(acc), "l"((unsigned long long)__float_as_uint(v.x) |
                      ((unsigned long long)__float_as_uint(v.y) << 32)));
  return d;
}
__device__ __forceinline__ bool prod_special(unsigned long long acc) {
  const float px = fabsf(__uint_as_float((uint32_t)acc));
  const float py = fabsf(__uint_as_float((uint32_t)(acc >> 32)));
  return !(px > 0.f && px <= 3.402823466e38f && py > 0.f && py <= 3.402823466e38f);
}
constexpr unsigned long long kProdOne = 0x3f8000003f800000ull;  // (1.f, 1.f)

// edge words of a -> b from sign words, the cross-sign word n and the edges E
// that touch a zero node (which count 0): P = crossing +1, N = crossing -1
struct EW {
  uint32_t P, N;
};
__device__ __forceinline__ EW edge_w(uint32_t sa, uint32_t sb, uint32_t n, uint32_t E) {
  EW e;
  e.P = ~sa & sb & ~n & ~E;
  e.N = sa & ~sb & n & ~E;
  return e;
}
__device__ __forceinline__ EW shr(EW e) { return EW{e.P >> 1, e.N >> 1}; }
__device__ __forceinline__ EW sh_dn(EW e) {
  return EW{__shfl_down_sync(FULL, e.P, 1), __shfl_down_sync(FULL, e.N, 1)};
}

// bit-sliced residues mod 8
struct Mod8 {
  uint32_t b0, b1, b2;
};

// a + b - c - d (each -1, 0 or 1): #nonzero - 2 #negative
__device__ __forceinline__ Mod8 loop_sum(EW a, EW b, EW c, EW d) {
  const uint32_t za = a.P | a.N, zb = b.P | b.N, zc = c.P | c.N, zd = d.P | d.N;
  const uint32_t ab = za & zb, cd = zc & zd, xab = za ^ zb, xcd = zc ^ zd;
  const uint32_t z1 = ab ^ cd ^ (xab & xcd);
  // negative terms: a, b where -1; c, d where +1
  const uint32_t gab = a.N ^ b.N, gcd = c.P ^ d.P;
  const uint32_t g0 = gab ^ gcd, g1 = (a.N & b.N) ^ (c.P & d.P) ^ (gab & gcd);
  Mod8 r;
  r.b0 = xab ^ xcd;
  r.b1 = z1 ^ g0;
  r.b2 = (ab & cd) ^ g1 ^ (~z1 & g0);
  return r;
}

__device__ __forceinline__ Mod8 add8(Mod8 a, Mod8 b) {
  const uint32_t c0 = a.b0 & b.b0;
  const uint32_t c1 = (a.b1 & b.b1) | (c0 & (a.b1 ^ b.b1));
  return Mod8{a.b0 ^ b.b0, a.b1 ^ b.b1 ^ c0, a.b2 ^ b.b2 ^ c1};
}
// with the row below (bit t: rows t - 1 and t), with the column to the left
__device__ __forceinline__ Mod8 add_row(Mod8 a) {
  return add8(a, Mod8{a.b0 << 1, a.b1 << 1, a.b2 << 1});
}
__device__ __forceinline__ Mod8 add_col(Mod8 a) {
  return add8(a, Mod8{__shfl_up_sync(FULL, a.b0, 1), __shfl_up_sync(FULL, a.b1, 1),
                      __shfl_up_sync(FULL, a.b2, 1)});
}
__device__ __forceinline__ uint32_t nonzero8(Mod8 a) { return a.b0 | a.b1 | a.b2; }

// value in [-3, 4] of row t of a residue
__device__ __forceinline__ int mod8_at(const Mod8& m, int t) {
  const int v = (int)((m.b0 >> t) & 1u) | (int)(((m.b1 >> t) & 1u) << 1) |
                (int)(((m.b2 >> t) & 1u) << 2);
  return v >= 5 ? v - 8 : v;
}

struct NodeArgs {
  const float2* psi;
  int nx, ny, nz;
  int nbands, nxseg, kchunk;
  long long nitems;               // z chunks * bands * column segments
  uint4* recs;                    // words 0..3 of the records
  uint32_t* recs4;                // word 4
  unsigned long long recs_cap;
  unsigned long long* top;        // staging chunk counter, work item counter
  uint2* table;                   // [nz][nbands][nxseg] {staging base, lane mask}
  unsigned int* segtot;           // [nz][nbands], zeroed before the launch
  int8_t* dense;                  // [3][nz][ny][nx] or null
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src)
               : "memory");
}

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Each lane streams its column of the band through the warp's ring with
// cp.async; a lane also reads its right neighbour's column, so every slot is
// fenced by __syncwarp after its copies complete and before it is refilled.
// Rows, columns and planes outside the grid hold (1, 1): finite and nonzero, and
// only ever on rings that the validity masks reject.
__global__ void __launch_bounds__(NODE_WARPS * 32, 4) node_form_kernel(const __grid_constant__ NodeArgs a) {
  extern __shared__ float2 node_ring[];
  const int lane = threadIdx.x & 31;
  float2* ring = node_ring + (size_t)(threadIdx.x >> 5) * kSlots * kSlotLen;
  const long long nwarps = (long long)gridDim.x * NODE_WARPS;
  const long long nxyz = (long long)a.nx * a.ny * a.nz;
  const unsigned lt = (1u << lane) - 1u;
  const int ln = lane < 31 ? lane + 1 : 31;
  unsigned long long chunk_at = 0;  // next free staging record of the warp's chunk
  uint32_t chunk_left = 0;
  const long long first = (long long)blockIdx.x * NODE_WARPS + (threadIdx.x >> 5);
  // the first items by warp, the others as warps get free
  auto next = [&]() {
    unsigned long long v = 0;
    if (lane == 0) v = atomicAdd(a.top + 1, 1ull);
    return nwarps + (long long)__shfl_sync(FULL, v, 0);
  };
  for (long long it = first; it < a.nitems; it = next()) {
    const int xs = (int)(it % a.nxseg);
    const long long rest = it / a.nxseg;
    const int band = (int)(rest % a.nbands);
    const int zc = (int)(rest / a.nbands);
    const int x = xs * NCOL + lane - 1;
    const int j0 = band * NB;  // row t of the band is j0 - 1 + t
    const int kz0 = zc * a.kchunk;
    const int kz1 = min(a.nz, kz0 + a.kchunk);
    const bool xin = x >= 0 && x < a.nx;
    const bool own = lane >= 1 && lane <= NCOL && x < a.nx;
    const bool colring = x >= 1 && x <= a.nx - 2;
    // rows in the grid (t in [lo, hi)), rows whose y-ring fits
    const int lo = j0 == 0 ? 1 : 0, hi = min(NT, a.ny - j0 + 1);
    const uint32_t rload = ((1u << hi) - 1u) & ~((1u << lo) - 1u);
    const uint32_t rin = rload & kOwnedRows;
    const uint32_t rring = rload & (rload << 1) & (rload >> 1) & kOwnedRows;
    const float2* const col = a.psi + (long long)(j0 - 1) * a.nx + x;
    const long long plane = (long long)a.nx * a.ny;

    auto issue = [&](int q, int slot) {
      float2* d = ring + slot * kSlotLen + lane;
      const bool qin = q >= 0 && q < a.nz && xin;
      const float2* src = col + (long long)q * plane;
      if (qin && rload == kRowsHeld) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          cp_async8(d + slot_at(t), src);
          src += a.nx;
        }
      } else {
#pragma unroll 1
        for (int t = 0; t < NT; ++t) {
          if (qin && ((rload >> t) & 1u)) cp_async8(d + slot_at(t), src);
          else d[slot_at(t)] = make_float2(1.f, 1.f);
          src += a.nx;
        }
      }
      cp_commit();
    };
    // planes kz0 - 1 .. kz1; plane q in slot (q - kz0 + 1) mod kSlots
    __syncwarp();
    issue(kz0 - 1, 0);
    issue(kz0, 1);
    int sp = 0;  // slot of plane p

    float2 V[NT];  // values of the previous plane
#pragma unroll
    for (int t = 0; t < NT; ++t) V[t] = make_float2(1.f, 1.f);
    EW RXc{0, 0}, RYc{0, 0};
    Mod8 S0c{0, 0, 0}, Tc{0, 0, 0}, Uc{0, 0, 0};  // xy ring sums of plane p - 1; yz, zx sums of
                                                  // the layer below it
    uint32_t Sprev = 0, ZBc = 0, Bm = 0, Bc = 0;

    for (int p = kz0 - 1; p <= kz1; ++p) {
      cp_wait<kSlots - 1>();  // plane p has landed (this lane's copies)
      __syncwarp();  // ... and every lane's
      const float2* cur = ring + sp * kSlotLen;
      uint32_t Sp = 0, NX = 0, NY = 0, NZ = 0;
      unsigned long long prod = kProdOne;
#pragma unroll
      for (int t = NT - 1; t >= 0; --t) {
        const float2 v = cur[t * 32 + lane];
        const float2 nb = cur[t * 32 + ln];
        Sp = push1(Sp, v.y);
        NX = push1(NX, cross_f(v, nb));
        NZ = push1(NZ, cross_f(V[t], v));
        if (t < NT - 1) NY = push1(NY, cross_f(v, V[t + 1]));
        prod = prod_step(prod, v);
        V[t] = v;
      }
      __syncwarp();  // every lane is done with the slot
      if (p + kSlots <= kz1) issue(p + kSlots, sp);
      else cp_commit();
      sp = sp + 1 == kSlots ? 0 : sp + 1;
      uint32_t ZBp = 0, Bn = 0;
      if (__any_sync(FULL, prod_special(prod))) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const float2 v = V[t];
          if (((__float_as_uint(v.x) | __float_as_uint(v.y)) << 1) == 0u) ZBp |= 1u << t;
          if (!(fin(v.x) && fin(v.y))) Bn |= 1u << t;
        }
        Bn &= xin ? rload : 0u;
      }
      const uint32_t Spn = __shfl_down_sync(FULL, Sp, 1);
      const uint32_t ZBpn = __shfl_down_sync(FULL, ZBp, 1);
      const EW RXn = edge_w(Sp, Spn, NX, ZBp | ZBpn);
      const EW RYn = edge_w(Sp, Sp >> 1, NY, ZBp | (ZBp >> 1));
      const EW RZ = edge_w(Sprev, Sp, NZ, ZBc | ZBp);  // edges p - 1 -> p
      const Mod8 S0n = add_col(add_row(loop_sum(RXn, sh_dn(RYn), shr(RXn), RYn)));
      // layer p - 1 -> p
      const Mod8 T = add_row(loop_sum(RYc, shr(RZ), RYn, RZ));
      const Mod8 U = add_col(loop_sum(RZ, RXn, sh_dn(RZ), RXc));
      if (p > kz0) {
        // node plane k = p - 1
        const int k = p - 1;
        const bool kring = k >= 1 && k <= a.nz - 2;
        const Mod8 S1 = add8(Tc, T), S2 = add8(Uc, U);
        uint32_t ok0 = (own && colring) ? rring : 0u;
        uint32_t ok1 = (own && kring) ? rring : 0u;
        uint32_t ok2 = (own && colring && kring) ? rin : 0u;
        if (__any_sync(FULL, (Bm | Bc | Bn) != 0u)) {  // rings through non-finite nodes
          const uint32_t Bl = __shfl_up_sync(FULL, Bc, 1), Br = __shfl_down_sync(FULL, Bc, 1);
          const uint32_t H = Bl | Bc | Br;
          const uint32_t V = Bm | Bc | Bn;
          ok0 &= ~((H << 1) | (H >> 1) | Bl | Br);
          ok1 &= ~((V << 1) | (V >> 1) | Bm | Bn);
          ok2 &= ~(__shfl_up_sync(FULL, V, 1) | __shfl_down_sync(FULL, V, 1) | Bm | Bn);
        }
        const uint32_t F = (nonzero8(S0c) & ok0) | (nonzero8(S1) & ok1) | (nonzero8(S2) & ok2);
        if (a.dense && own) {
#pragma unroll 1
          for (int t = 1; t <= NB; ++t) {
            if (!((rin >> t) & 1u)) continue;
            const long long q = ((long long)k * a.ny + (j0 - 1 + t)) * a.nx + x;
            a.dense[q] = (int8_t)(((ok0 >> t) & 1u) ? mod8_at(S0c, t) : 0);
            a.dense[nxyz + q] = (int8_t)(((ok1 >> t) & 1u) ? mod8_at(S1, t) : 0);
            a.dense[2 * nxyz + q] = (int8_t)(((ok2 >> t) & 1u) ? mod8_at(S2, t) : 0);
          }
        }
        // records of this step, by sub-band: contiguous in the warp's staging chunk
#pragma unroll
        for (int sb = 0; sb < NSUB; ++sb) {
          const int sh = sb * SUBR;
          const uint32_t Fs = (F >> sh) & kSubRows;
          const uint32_t cnt = __reduce_add_sync(FULL, (uint32_t)__popc(Fs));
          const uint32_t bal = __ballot_sync(FULL, Fs != 0u);
          const uint32_t nrec = (uint32_t)__popc(bal);
          if (nrec > chunk_left) {
            unsigned long long b = 0;
            if (lane == 0) b = atomicAdd(a.top, (unsigned long long)kChunk);
            chunk_at = __shfl_sync(FULL, b, 0);
            chunk_left = kChunk;
          }
          const unsigned long long base = chunk_at;
          chunk_at += nrec;
          chunk_left -= nrec;
          if (Fs) {
            const unsigned long long q = base + (unsigned)__popc(bal & lt);
            if (q < a.recs_cap) {
              auto two = [&](uint32_t u, uint32_t v) {
                return ((u >> sh) & kSubRows) | (((v >> sh) & kSubRows) << 16);
              };
              a.recs[q] = make_uint4(two(S0c.b0 & ok0, S0c.b1 & ok0), two(S0c.b2 & ok0, S1.b0 & ok1),
                                     two(S1.b1 & ok1, S1.b2 & ok1), two(S2.b0 & ok2, S2.b1 & ok2));
              a.recs4[q] = (((S2.b2 & ok2) >> sh) & kSubRows) | ((uint32_t)lane << 16);
            }
          }
          if (lane == 0) {
            const long long sg = (long long)k * (a.nbands * NSUB) + band * NSUB + sb;
            if (cnt) atomicAdd(a.segtot + sg, cnt);
            a.table[sg * a.nxseg + xs] = make_uint2((uint32_t)base, bal);
          }
        }
      }
      RXc = RXn;
      RYc = RYn;
      S0c = S0n;
      Tc = T;
      Uc = U;
      Sprev = Sp;
      ZBc = ZBp;
      Bm = Bc;
      Bc = Bn;
    }
    cp_wait<0>();
    __syncwarp();
  }
}

// Exclusive scan of the per-(plane, sub-band) totals, whose order is ascending node
// order.  A block per chunk of totals.  Up to kScanAlone totals the chunks are one tile
// and a block adds the totals before its chunk itself (one block over all of them: 12 us
// for 1e4 totals); above, that would grow with their square (3.2e7 totals: a call 91 ms, now 21), so at
// most kScanChunks larger chunks are summed by a launch before it.
constexpr int kScanPer = 4;  // consecutive totals per thread
constexpr int kScanTile = 1024 * kScanPer;
constexpr long long kScanAlone = 64LL * kScanTile;
constexpr long long kScanChunks = 2048;

// (all threads get the sum)
__device__ __forceinline__ unsigned long long scan_block_sum(unsigned long long v, unsigned long long* wb) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
  __syncthreads();  // wb may still be read
  if (lane == 0) wb[w] = v;
  __syncthreads();
  v = wb[lane];
#pragma unroll
  for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
  return v;
}

__global__ void __launch_bounds__(1024) node_sums_kernel(const unsigned int* __restrict__ segtot,
                                                         long long nseg, long long chunk,
                                                         unsigned long long* __restrict__ sums) {
  __shared__ unsigned long long wb[32];
  const long long c0 = blockIdx.x * chunk, c1 = min(nseg, c0 + chunk);
  unsigned long long v = 0;
#pragma unroll 8
  for (long long i = c0 + threadIdx.x; i < c1; i += 1024) v += segtot[i];
  v = scan_block_sum(v, wb);
  if (threadIdx.x == 0) sums[blockIdx.x] = v;
}

// sums: of the chunks, or null (then a chunk is one tile)
__global__ void __launch_bounds__(1024) node_scan_kernel(const unsigned int* __restrict__ segtot,
                                                         long long nseg, long long chunk,
                                                         const unsigned long long* __restrict__ sums,
                                                         unsigned long long* __restrict__ seg_off,
                                                         uint64_t* __restrict__ count) {
  __shared__ unsigned long long wb[32], wt[32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const long long c0 = blockIdx.x * chunk, c1 = min(nseg, c0 + chunk);
  unsigned long long before = 0;
  if (sums) {
    for (long long i = tid; i < blockIdx.x; i += 1024) before += sums[i];
  } else {
#pragma unroll 8
    for (long long i = tid; i < c0; i += 1024) before += segtot[i];
  }
  before = scan_block_sum(before, wb);
  for (long long t0 = c0; t0 < c1; t0 += kScanTile) {
    const long long s = t0 + tid * kScanPer;
    unsigned long long v[kScanPer], local = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
      v[i] = s + i < c1 ? segtot[s + i] : 0u;
      local += v[i];
    }
    unsigned long long incl = local;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long u = __shfl_up_sync(FULL, incl, d);
      if (lane >= d) incl += u;
    }
    __syncthreads();  // wt may still be read
    if (lane == 31) wt[w] = incl;
    __syncthreads();
    unsigned long long run = before + incl - local;
    for (int q = 0; q < 32; ++q) {
      run += q < w ? wt[q] : 0ull;
      before += wt[q];
    }
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
      if (s + i < c1) seg_off[s + i] = run;
      run += v[i];
    }
  }
  if (c1 == nseg && tid == 0) *count = before;
}

// One warp per (plane, band): its records, by column segment and lane, i.e. by
// ascending x, give its nodes row by row: per row and 32 records one ballot ranks
// the records with a node there.  Records of up to kHeldRecs x 32 lanes stay in
// registers (a sub-band of a 512-column tangle has about 100); larger segments read
// them again for each row.
constexpr int kHeldRecs = 5;
constexpr int kMaxSegs = (64 * kMaxWarpsX + NCOL - 1) / NCOL;
constexpr int kMaxE = (kMaxSegs + 31) / 32;  // table entries per lane
static_assert(kMaxE == 3, "the entry selection below handles three entries per lane");

struct NodeRec {
  uint4 w;
  uint32_t w4, x;
  __device__ __forceinline__ uint32_t rows() const {
    const uint32_t m = w.x | w.y | w.z | w.w;
    return (m | (m >> 16) | w4) & 0xFFFFu;
  }
};

__global__ void __launch_bounds__(256) node_expand_kernel(
    const uint2* __restrict__ table, const unsigned long long* __restrict__ seg_off, long long nseg,
    int nbands, int nxseg, int nx, int ny, const uint4* __restrict__ recs,
    const uint32_t* __restrict__ recs4, unsigned long long recs_cap, uint64_t* __restrict__ node_ids,
    int8_t* __restrict__ circ, unsigned long long capacity) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
  const int E = (nxseg + 31) >> 5, NL = (nxseg + E - 1) / E;  // lane l holds segments l E ..
  for (long long s = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nseg;
       s += warps) {
    uint2 en[kMaxE];
    uint32_t n = 0;
#pragma unroll
    for (int j = 0; j < kMaxE; ++j) {
      const int i = lane * E + j;
      en[j] = (j < E && i < nxseg) ? table[s * nxseg + i] : make_uint2(0u, 0u);
      n += __popc(en[j].y);
    }
    const unsigned long long off = seg_off[s];
    uint32_t incl = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(FULL, incl, d);
      if (lane >= d) incl += u;
    }
    const uint32_t start = lane < NL ? incl - n : 0xFFFFFFFFu;
    const uint32_t rtot = __shfl_sync(FULL, incl, 31);
    if (rtot == 0) continue;
    const long long k = s / nbands;
    const long long j0 = (s - k * nbands) * SUBR;
    const unsigned long long lin0 =  // of row t = 0 (only rows t >= 1 are used)
        ((unsigned long long)k * ny + (unsigned long long)j0) * (unsigned long long)nx - (unsigned long long)nx;
    // record of index g0 + lane in x order (no rows past the end)
    auto load = [&](uint32_t g0) -> NodeRec {
      const uint32_t g = g0 + lane;
      int lo = 0;
#pragma unroll
      for (int st = 16; st >= 1; st >>= 1) {
        const int cand = lo + st;
        const uint32_t sv = __shfl_sync(FULL, start, cand & 31);
        if (cand < NL && sv <= g) lo = cand;
      }
      uint32_t qi = g - __shfl_sync(FULL, start, lo);
      uint2 e = make_uint2(__shfl_sync(FULL, en[0].x, lo), __shfl_sync(FULL, en[0].y, lo));
      int j = 0;
      if (E > 1) {  // uniform
        const uint2 e1 = make_uint2(__shfl_sync(FULL, en[1].x, lo), __shfl_sync(FULL, en[1].y, lo));
        const uint2 e2 = make_uint2(__shfl_sync(FULL, en[2].x, lo), __shfl_sync(FULL, en[2].y, lo));
        const uint32_t c0 = __popc(e.y), c1 = __popc(e1.y);
        if (qi >= c0) {
          qi -= c0;
          j = 1;
          e = e1;
          if (qi >= c1) {
            qi -= c1;
            j = 2;
            e = e2;
          }
        }
      }
      NodeRec r;
      r.w = make_uint4(0u, 0u, 0u, 0u);
      r.w4 = r.x = 0u;
      const unsigned long long idx = (unsigned long long)e.x + qi;
      if (g < rtot && idx < recs_cap) {
        r.w = recs[idx];
        r.w4 = recs4[idx];
        r.x = (uint32_t)((lo * E + j) * NCOL - 1) + (r.w4 >> 16);
      }
      return r;
    };
    uint32_t run = 0;  // nodes of the segment so far
    // the records' nodes of row t, after those already listed
    auto emit = [&](const NodeRec& r, int t) {
      const bool has = (r.rows() >> t) & 1u;
      const unsigned bal = __ballot_sync(FULL, has);
      if (has) {
        const unsigned long long dst = off + run + (unsigned)__popc(bal & lt);
        if (dst < capacity) {
          auto val = [&](uint32_t b0, uint32_t b1, uint32_t b2) {
            const int v = (int)(b0 & 1u) | (int)((b1 & 1u) << 1) | (int)((b2 & 1u) << 2);
            return (int8_t)(v >= 5 ? v - 8 : v);
          };
          node_ids[dst] = lin0 + (unsigned long long)((uint32_t)t * (uint32_t)nx + r.x);
          circ[3 * dst] = val(r.w.x >> t, r.w.x >> (t + 16), r.w.y >> t);
          circ[3 * dst + 1] = val(r.w.y >> (t + 16), r.w.z >> t, r.w.z >> (t + 16));
          circ[3 * dst + 2] = val(r.w.w >> t, r.w.w >> (t + 16), r.w4 >> t);
        }
      }
      run += (uint32_t)__popc(bal);
    };
    if (rtot <= 32u * kHeldRecs) {
      NodeRec held[kHeldRecs];
#pragma unroll
      for (int c = 0; c < kHeldRecs; ++c)
        if (32u * c < rtot) held[c] = load(32u * c);
#pragma unroll 1
      for (int t = 1; t <= SUBR; ++t) {
#pragma unroll
        for (int c = 0; c < kHeldRecs; ++c)
          if (32u * c < rtot) emit(held[c], t);
      }
    } else {
#pragma unroll 1
      for (int t = 1; t <= SUBR; ++t)
        for (uint32_t g0 = 0; g0 < rtot; g0 += 32u) emit(load(g0), t);
    }
  }
}

// FP64 sum of the block's per-thread values; thread 0 gets it.
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int d = 16; d; d >>= 1) v += __shfl_down_sync(FULL, v, d);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
  return r;
}

// Sum of |psi|^2 over all nodes: FP32 runs of up to 4 nodes (8 squares),
// FP64 across runs.
__global__ void __launch_bounds__(DENS_THREADS) density_mean_kernel(const float2* __restrict__ psi,
                                                                    long long n,
                                                                    double* __restrict__ partial) {
  __shared__ double sh[DENS_THREADS / 32];
  const long long stride = (long long)gridDim.x * DENS_THREADS;
  double acc = 0.0;
  long long q = (long long)blockIdx.x * DENS_THREADS + threadIdx.x;
  for (; q + 3 * stride < n; q += 4 * stride) {
    const float2 a = __ldg(psi + q), b = __ldg(psi + q + stride), c = __ldg(psi + q + 2 * stride),
                 d = __ldg(psi + q + 3 * stride);
    float run = a.x * a.x;
    run = fmaf(a.y, a.y, run);
    run = fmaf(b.x, b.x, run);
    run = fmaf(b.y, b.y, run);
    run = fmaf(c.x, c.x, run);
    run = fmaf(c.y, c.y, run);
    run = fmaf(d.x, d.x, run);
    run = fmaf(d.y, d.y, run);
    acc += (double)run;
  }
  for (; q < n; q += stride) {
    const float2 a = __ldg(psi + q);
    acc += (double)fmaf(a.y, a.y, a.x * a.x);
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

struct DensArgs {
  const float2* psi;
  int nx, ny, nz;
  float h, ox, oy, oz;
  const float* xyz;
  unsigned long long n;
  const uint64_t* n_dev;
  float* rho;
  double* partial;
};

// Trilinear density at the points (grid coordinates (p - origin) / h; NaN
// outside [0, n - 1] per axis) and the FP64 sum of |rho| per block.
__global__ void __launch_bounds__(DENS_THREADS) density_points_kernel(DensArgs a) {
  __shared__ double sh[DENS_THREADS / 32];
  unsigned long long nn = a.n;
  if (a.n_dev) {
    const unsigned long long d = *a.n_dev;
    if (d < nn) nn = d;
  }
  double acc = 0.0;
  for (unsigned long long q = (unsigned long long)blockIdx.x * DENS_THREADS + threadIdx.x; q < nn;
       q += (unsigned long long)gridDim.x * DENS_THREADS) {
    const float x = (__ldg(a.xyz + 3 * q) - a.ox) / a.h;
    const float y = (__ldg(a.xyz + 3 * q + 1) - a.oy) / a.h;
    const float z = (__ldg(a.xyz + 3 * q + 2) - a.oz) / a.h;
    float r;
    if (!(x >= 0.f && y >= 0.f && z >= 0.f && x <= (float)(a.nx - 1) && y <= (float)(a.ny - 1) &&
          z <= (float)(a.nz - 1))) {
      r = __int_as_float(0x7fc00000);
    } else {
      const int i = min((int)floorf(x), max(a.nx - 2, 0));
      const int j = min((int)floorf(y), max(a.ny - 2, 0));
      const int k = min((int)floorf(z), max(a.nz - 2, 0));
      const float fx = x - (float)i, fy = y - (float)j, fz = z - (float)k;
      const int i1 = i + 1 < a.nx ? i + 1 : i, j1 = j + 1 < a.ny ? j + 1 : j,
                k1 = k + 1 < a.nz ? k + 1 : k;
      float re = 0.f, im = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int ii = (c & 1) ? i1 : i, jj = (c & 2) ? j1 : j, kk = (c & 4) ? k1 : k;
        const float w = ((c & 1) ? fx : 1.f - fx) * ((c & 2) ? fy : 1.f - fy) *
                        ((c & 4) ? fz : 1.f - fz);
        const float2 v = __ldg(a.psi + ((long long)kk * a.ny + jj) * a.nx + ii);
        re = fmaf(w, v.x, re);
        im = fmaf(w, v.y, im);
      }
      r = fmaf(re, re, im * im);
    }
    if (a.rho) a.rho[q] = r;
    acc += (double)fabsf(r);
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) a.partial[blockIdx.x] = s;
}

// out = {e, mean |rho| over the points, rho_bar}; the partial sums are added
// in a fixed order by one warp.
__global__ void density_final_kernel(const double* __restrict__ pm, int nbm,
                                     const double* __restrict__ pp, int nbp, long long nodes,
                                     unsigned long long n, const uint64_t* n_dev,
                                     double* __restrict__ out) {
  const int lane = threadIdx.x;
  double sm = 0.0, sp = 0.0;
  for (int b = lane; b < nbm; b += 32) sm += pm[b];
  for (int b = lane; b < nbp; b += 32) sp += pp[b];
#pragma unroll
  for (int d = 16; d; d >>= 1) {
    sm += __shfl_down_sync(FULL, sm, d);
    sp += __shfl_down_sync(FULL, sp, d);
  }
  if (lane == 0) {
    unsigned long long nn = n;
    if (n_dev && *n_dev < nn) nn = *n_dev;
    const double rho_bar = nodes > 0 ? sm / (double)nodes : 0.0;
    out[0] = nn ? sp / (rho_bar * (double)nn) : 0.0;
    out[1] = nn ? sp / (double)nn : 0.0;
    out[2] = rho_bar;
  }
}

bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return false;
  return cs != cudaStreamCaptureStatusNone;
}

template <typename T>
int grow(T*& p, uint64_t& cap, uint64_t want, cudaStream_t st, const char* what) {
  if (want <= cap && p) return QTV_OK;
  if (capturing(st))
    return set_error(QTV_ERR_STATE, "%s: workspace must grow during stream capture", what);
  cudaFree(p);
  p = nullptr;
  cap = 0;
  const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&p), want * sizeof(T));
  if (e != cudaSuccess) {
    p = nullptr;
    return check_cuda(e, what);
  }
  cap = want;
  return QTV_OK;
}

NodeWork* work_of(qtv_handle h, cudaStream_t st, int* rc) {
  *rc = QTV_OK;
  if (h->node) return h->node;
  if (capturing(st)) {
    *rc = set_error(QTV_ERR_STATE, "node-form workspace must be created outside stream capture");
    return nullptr;
  }
  NodeWork* w = new NodeWork();
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&w->top), (2 + kScanChunks) * sizeof(unsigned long long));
  if (e != cudaSuccess) {
    delete w;
    *rc = check_cuda(e, "cudaMalloc(node-form counter)");
    return nullptr;
  }
  int bps = 0;
  e = cudaFuncSetAttribute(node_form_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kNodeSmem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, node_form_kernel, NODE_WARPS * 32,
                                                      kNodeSmem);
  if (e != cudaSuccess) {
    node_work_free(w);
    *rc = check_cuda(e, "occupancy(node_form_kernel)");
    return nullptr;
  }
  w->resident_warps = (bps > 0 ? bps : 1) * NODE_WARPS * h->num_sms;
  h->node = w;
  return w;
}

int launch_blocks(const NodeWork* w, long long nitems) {
  long long blocks = (nitems + NODE_WARPS - 1) / NODE_WARPS;
  const long long maxb = w->resident_warps / NODE_WARPS;
  if (blocks > maxb) blocks = maxb;
  if (blocks < 1) blocks = 1;
  return (int)blocks;
}

}  // namespace

int node_circulation_launch(qtv_handle h, const qtv_grid& g, const float2* psi,
                            uint64_t* node_ids, int8_t* circ, uint64_t capacity, uint64_t* count,
                            int8_t* dense, cudaStream_t st) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const long long nodes = (long long)nx * ny * nz;
  if (nodes == 0) {
    const cudaError_t e = cudaMemsetAsync(count, 0, sizeof(uint64_t), st);
    return check_cuda(e, "cudaMemsetAsync(count)");
  }
  int rc = QTV_OK;
  NodeWork* w = work_of(h, st, &rc);
  if (!w) return rc;
  const int nbands = (ny + NB - 1) / NB;
  const int nxseg = (nx + NCOL - 1) / NCOL;
  const long long per_chunk = (long long)nbands * nxseg;
  // z chunks: about kItems per resident warp, of at least 8 planes
  const long long want = (kItemsPerWarp * (long long)w->resident_warps + per_chunk - 1) / per_chunk;
  int kchunk = (int)((nz + want - 1) / want);
  if (kchunk < 8) kchunk = nz < 8 ? nz : 8;
  const int nzchunks = (nz + kchunk - 1) / kchunk;
  const long long nitems = (long long)nzchunks * per_chunk;
  const long long nseg = (long long)nz * nbands * NSUB;
  const uint64_t ntab = (uint64_t)nseg * nxseg;
  // staging: the records (at least one node each, at most one for the column of a
  // sub-band), plus what chunk switches leave unused (under one step of at most NCOL
  // <= kChunk / 8 records per chunk, i.e. at most 1/7 of the records) and the open
  // chunk of every warp
  const long long launch_warps = (long long)launch_blocks(w, nitems) * NODE_WARPS;
  const uint64_t most = std::min(capacity, (uint64_t)nseg * (uint64_t)nx);
  const uint64_t recs_need = most + most / 7 + 1 + (uint64_t)launch_warps * kChunk;
  static_assert(NCOL * 8 <= (int)kChunk, "chunk slack bound");
  // table entries keep 32-bit staging offsets
  if (recs_need > 0xFFFFFFFFull)
    return set_error(QTV_ERR_ARG, "node form: %llu staging records (capacity %llu) exceed 2^32",
                     (unsigned long long)recs_need, (unsigned long long)capacity);
  rc = grow(w->recs, w->recs_cap, recs_need, st, "cudaMalloc(node records)");
  if (!rc) rc = grow(w->recs4, w->recs4_cap, recs_need, st, "cudaMalloc(node records)");
  if (!rc) rc = grow(w->table, w->table_cap, ntab, st, "cudaMalloc(node table)");
  if (!rc) rc = grow(w->segtot, w->segtot_cap, (uint64_t)nseg, st, "cudaMalloc(node totals)");
  if (!rc) rc = grow(w->seg_off, w->seg_off_cap, (uint64_t)nseg, st, "cudaMalloc(node offsets)");
  if (rc) return rc;

  cudaError_t e = cudaMemsetAsync(w->top, 0, 2 * sizeof(unsigned long long), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(w->segtot, 0, nseg * sizeof(unsigned int), st);
  if (e != cudaSuccess) return check_cuda(e, "cudaMemsetAsync(node-form state)");
  NodeArgs a;
  a.psi = psi;
  a.nx = nx;
  a.ny = ny;
  a.nz = nz;
  a.nbands = nbands;
  a.nxseg = nxseg;
  a.kchunk = kchunk;
  a.nitems = nitems;
  a.recs = w->recs;
  a.recs4 = w->recs4;
  a.recs_cap = w->recs_cap < w->recs4_cap ? w->recs_cap : w->recs4_cap;
  a.top = w->top;
  a.table = w->table;
  a.segtot = w->segtot;
  a.dense = dense;
  {
    TraceScope ts(h, K_NODE_FORM, st);
    node_form_kernel<<<launch_blocks(w, nitems), NODE_WARPS * 32, kNodeSmem, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return check_cuda(e, "node_form_kernel launch");
  }
  {
    TraceScope ts(h, K_NODE_SCAN, st);
    long long chunk = kScanTile;
    unsigned long long* sums = nullptr;
    if (nseg > kScanAlone) {
      sums = w->top + 2;
      const long long tiles = (nseg + kScanTile - 1) / kScanTile;
      chunk = (tiles + kScanChunks - 1) / kScanChunks * kScanTile;
    }
    const unsigned blocks = (unsigned)((nseg + chunk - 1) / chunk);
    if (sums) node_sums_kernel<<<blocks, 1024, 0, st>>>(w->segtot, nseg, chunk, sums);
    node_scan_kernel<<<blocks, 1024, 0, st>>>(w->segtot, nseg, chunk, sums, w->seg_off, count);
    e = cudaGetLastError();
    if (e != cudaSuccess) return check_cuda(e, "node_scan_kernel launch");
  }
  if (capacity > 0 && node_ids && circ) {
    long long blocks = (nseg + 7) / 8;
    const long long maxb = (long long)h->num_sms * 16;
    if (blocks > maxb) blocks = maxb;
    TraceScope ts(h, K_NODE_SCATTER, st);
    node_expand_kernel<<<(int)blocks, 256, 0, st>>>(w->table, w->seg_off, nseg, nbands * NSUB, nxseg, nx, ny,
                                                    w->recs, w->recs4, a.recs_cap, node_ids, circ,
                                                    capacity);
    e = cudaGetLastError();
    if (e != cudaSuccess) return check_cuda(e, "node_expand_kernel launch");
  }
  return QTV_OK;
}

int density_error_launch(qtv_handle h, const qtv_grid& g, const float2* psi, const float* xyz,
                         uint64_t n, const uint64_t* n_dev, float* rho, double* out,
                         cudaStream_t st) {
  int rc = QTV_OK;
  NodeWork* w = work_of(h, st, &rc);
  if (!w) return rc;
  const long long nodes = (long long)g.nx * g.ny * g.nz;
  const int nbm = h->num_sms * 4;
  long long nbp_l = ((long long)n + DENS_THREADS - 1) / DENS_THREADS;
  if (nbp_l > h->num_sms * 4) nbp_l = h->num_sms * 4;
  if (nbp_l < 1) nbp_l = 1;
  const int nbp = (int)nbp_l;
  rc = grow(w->partial, w->partial_cap, (uint64_t)(nbm + nbp), st, "cudaMalloc(density sums)");
  if (rc) return rc;
  TraceScope ts(h, K_DENSITY, st);
  density_mean_kernel<<<nbm, DENS_THREADS, 0, st>>>(psi, nodes, w->partial);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return check_cuda(e, "density_mean_kernel launch");
  DensArgs a;
  a.psi = psi;
  a.nx = g.nx;
  a.ny = g.ny;
  a.nz = g.nz;
  a.h = g.h;
  a.ox = g.origin[0];
  a.oy = g.origin[1];
  a.oz = g.origin[2];
  a.xyz = xyz;
  a.n = n;
  a.n_dev = n_dev;
  a.rho = rho;
  a.partial = w->partial + nbm;
  density_points_kernel<<<nbp, DENS_THREADS, 0, st>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return check_cuda(e, "density_points_kernel launch");
  density_final_kernel<<<1, 32, 0, st>>>(w->partial, nbm, w->partial + nbm, nbp, nodes, n, n_dev,
                                         out);
  e = cudaGetLastError();
  if (e != cudaSuccess) return check_cuda(e, "density_final_kernel launch");
  return QTV_OK;
}

}  // namespace qtv
