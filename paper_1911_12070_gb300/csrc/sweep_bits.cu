// sweep_bits.cu -- bit-sliced identification sweep (Sec. 2.2.2, Eq. 5).
//
// Decomposition.  A CTA owns a band of 16 rows (+1 halo row) of an x tile and
// marches z.  Lane l of warp w owns the grid column x = 31 w + l of the tile;
// lane 31 is the halo column of the warp (the first column of the next warp)
// and owns no faces, so every quantity of column x + 1 that a lane needs comes
// from lane l + 1 by a shuffle.  Each lane walks its 17 rows and keeps one bit
// per row in 32-bit words: the sign bit of Im psi (the half-plane of the node)
// and the sign bits of the cross products of its x, y and z edges.
//
// Edge test.  As in the nibble sweep (sweep_bulk.cu): with s the sign bit of
// Im psi (IEEE atan2 convention) and n the sign bit of the FP32 FMA value of
// cross(a, b) = Re a Im b - Im a Re b, the branch-crossing integer of edge
// a -> b is +1 when s_a = 0, s_b = 1, n = 0, and -1 when s_a = 1, s_b = 0,
// n = 1, else 0.  Per word of 17 rows: P = ~s_a & s_b & ~n, N = s_a & ~s_b &
// n, and Z = P | N.
//
// Plaquette sums.  W = r1 + r2 - r3 - r4 lies in {-1, 0, 1, 2} (four wrapped
// differences in (-pi, pi] add to a multiple of 2 pi in (-4 pi, 4 pi]), so W
// is fixed by W mod 4.  A term t = +-r has the 2-bit code (Z, N) for +r and
// (Z, P) for -r (1 = 01, -1 = 11); the sum of four codes mod 4 has low bit
// L = xor of the four Z and high bit H = xor of the four high bits xor the
// parity of the pairs of Z (the carry), so W = 1, 2, -1 for (L, H) = (1, 0),
// (0, 1), (1, 1).  Each orientation takes nine 3-input logic operations for
// 16 rows.
//
// Zero and non-finite nodes.  A warp-uniform test per plane (a packed FP32x2
// product of the Re and Im values, zero if a component of a node is, or
// non-finite) selects a path that builds zero-node bits (their edges count 0:
// phase 0) and non-finite bits (their faces are dropped).  Padding holds
// (1, 1), finite with nonzero components.
//
// Staging.  Planes of the band arrive by cp.async.bulk row copies (one per row,
// issued by the lanes of warp 0) into a ring of shared-memory slots with a
// "full" mbarrier (transaction bytes) and an "empty" mbarrier (one arrival per
// warp after it has read the slot) per slot, so warps are not held in lockstep.
// A lane keeps the 17 values of plane k in registers while it reads plane
// k + 1.  Waits are bounded (about 2^32 SM cycles); a timeout sets a status
// bit that turns the reported count into QTV_COUNT_TIMEOUT.
//
// Stacked last tiles.  A CTA's plane step costs about the same whatever the
// tile width (the sweep is latency-bound per CTA), so a last tile of a row
// that is narrower than one warp (16 columns at nx = 512) would cost a whole
// CTA unit per band and plane.  Instead the last tiles of NW consecutive
// bands share one unit: warp v takes band band0 + v as if it were warp 0 of
// that band's last tile, in its own 32-column strip of the slot rows.  Strip
// rows are too short for bulk copies to pay (each bulk copy has a fixed cost),
// so each warp fills its own strip with 16-byte cp.async copies, one commit
// group per plane, and the warps of a stacked unit run independently.
//
// Unaligned rows (UNAL).  With odd nx, or a field on an 8-byte boundary, a row
// starts 8 bytes off a 16-byte boundary in some or all rows.  Its bulk copy is
// widened to the boundaries (the neighbours in the field come along), which
// shifts the row by one element in its slot row; a lane reads the even and the
// odd rows of a plane at two column offsets.  Such fields took the register
// sweep (identify.cu), whose edge test is exact, so this instantiation decides
// the same windings: per edge it keeps the margin by which |cross| clears its
// rounding errors.  Where an x, y or z edge of a lane is within reach of them the
// edge matters only if its nodes lie in different half-planes (else it crosses
// nothing whatever the sign), and only then the warp's edges of that row, direction and
// plane are taken again with the comparison of exact_edge: ties of equal neighbours,
// real fields and regions of zeros cost a vote, single ties a row.  Bound, as the
// aligned instantiation, by the latency of a CTA's plane steps (47% of the issue slots
// and 41% of HBM taken at 275 x 301 x 253), with a quarter more instructions a node.  512 x 512 x 511: 0.284 ms against 0.785 for the register
// sweep (0.222 aligned at 512^3); 256 x 256 x 255: 0.054 against 0.094.  Whole steps of
// 275 x 301 x 253, in us against the register sweep: waves 98 (147), the same scaled by
// 1e-19 101 (154), a real field 89 (122), constant along z 107 (146), zero outside a
// ball 135 (130); with ties in every warp, integers up to 3, 172 (157), and with a
// Gaussian that leaves FP32's range within the grid 163 (135).
// Holding the smallest |cross| against a per-plane bound from the largest
// component instead took 0.413 ms: near-parallel neighbours tripped it; redoing every
// plane with a doubtful edge or a product of components that underflows took 170 to
// 190 us for fields with zeros, ties or vanishing amplitude.
//
// Output and finalize.  Each lane with faces in a plane writes one 16-byte
// record (L and H words of the three orientations, 16 rows each, and the lane)
// into the fixed slot block of its (plane, band, tile, warp) step (32 records,
// one per lane); the step's table entry (ballot of the lanes with records,
// face count) is held by lane t % 32 and 32 consecutive planes' entries are
// stored at once; face totals per (plane, band) segment accumulate in shared
// memory for the CTA's run of planes and are added to the segment totals at
// its end.  The scan of the nibble sweep gives segment offsets, and the expand
// pass (expand_bits.cu) writes faces in ascending face-id order (row, then x,
// then orientation).
#include <algorithm>

#include "bits_layout.cuh"
#include "qtv_internal.cuh"
#include "sweep_common.cuh"

namespace qtv {
namespace {

using namespace sweep;
using namespace bits;

constexpr int kMaxRun = 256;      // planes per run (bounds the shared face totals)
constexpr int kTail = 8;          // padding elements after the ring (stacked strips)

// acc' = (acc << 1) | sign bit of x
__device__ __forceinline__ uint32_t push1(uint32_t acc, float x) {
  return __funnelshift_l(__float_as_uint(x), acc, 1);
}

struct Edge {
  uint32_t P, N, Z;
};

// edges a -> b from the sign words of a and b, the cross-sign word n, and the
// edges E that touch a zero node (contribute 0)
__device__ __forceinline__ Edge edge_words(uint32_t sa, uint32_t sb, uint32_t n, uint32_t E) {
  Edge e;
  e.P = ~sa & sb & ~n & ~E;
  e.N = sa & ~sb & n & ~E;
  e.Z = e.P | e.N;
  return e;
}

__device__ __forceinline__ Edge edge_words(uint32_t sa, uint32_t sb, uint32_t n) {
  Edge e;
  e.P = ~sa & sb & ~n;
  e.N = sa & ~sb & n;
  e.Z = e.P | e.N;
  return e;
}

// packed product of the (Re, Im) values of a plane: zero when a component of
// a node is zero, non-finite when a node is (or on FP32 under- or overflow,
// which merely selects the masking path)
__device__ __forceinline__ unsigned long long prod_step(unsigned long long acc, float2 v) {
  return mul_f32x2(acc, (unsigned long long)__float_as_uint(v.x) |
                            ((unsigned long long)__float_as_uint(v.y) << 32));
}
__device__ __forceinline__ bool prod_special(unsigned long long acc) {
  const float px = fabsf(__uint_as_float((uint32_t)acc)), py = fabsf(__uint_as_float((uint32_t)(acc >> 32)));
  return !(px > 0.f && px <= 3.402823466e38f && py > 0.f && py <= 3.402823466e38f);
}
constexpr unsigned long long kProdOne = 0x3f8000003f800000ull;  // (1.f, 1.f)

// sum mod 4 of four terms given as (low, high) bit words
__device__ __forceinline__ void mod4(uint32_t a, uint32_t a1, uint32_t b, uint32_t b1, uint32_t c,
                                     uint32_t c1, uint32_t d, uint32_t d1, uint32_t& L,
                                     uint32_t& H) {
  const uint32_t x = a ^ b, y = c ^ d;
  L = x ^ y;
  const uint32_t e2 = (a & b) ^ (c & d) ^ (x & y);
  H = a1 ^ b1 ^ c1 ^ d1 ^ e2;
}

// ---- exact edge test of the unaligned instantiation (see "Unaligned rows")
// exact_edge holds the FP32 value c of cross(a, b) against e, the rounding error of its
// second product p: |e| <= 2^-24 |p| (an error too small for FP32 is 0).  So c alone
// decides where |c| > 2^-21 |p|, eight times that: where the margin |c| - 2^-21 |p| is
// positive, which one FMA decides without a false positive, underflow or not.
// cross_m gives the value and the margin.
constexpr float kTieFar = 3.402823466e38f;
constexpr uint32_t kRowsHeld = (1u << BRH) - 1u;
__device__ __forceinline__ float cross_m(float2 a, float2 b, float& m) {
  const float p = a.y * b.x;
  const float c = fmaf(a.x, b.y, -p);
  m = fmaf(-4.76837158203125e-7f, fabsf(p), fabsf(c));
  return c;
}
// Padding of rows past the grid: vectors whose x-, y- and z-neighbours differ,
// so that no edge between them is a tie.
__device__ __forceinline__ float2 pad_value(int row, int col, int slot) {
  return make_float2(1.f, (float)(1 + (col & 1) + 2 * (row & 1) + 4 * slot));
}
// the comparisons of exact_edge(a, b): bit into G where c > e, into L where c < e
__device__ __forceinline__ void exact_compare(float2 a, float2 b, uint32_t bit, uint32_t& G, uint32_t& L) {
  const float p = __fmul_rn(a.y, b.x);
  const float e = fmaf(a.y, b.x, -p);
  const float c = fmaf(a.x, b.y, -p);
  if (c > e) G |= bit;
  if (c < e) L |= bit;
}
// zero if both components are finite, else NaN, added to acc
__device__ __forceinline__ unsigned long long finite_step(unsigned long long acc, float2 v) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"((unsigned long long)__float_as_uint(v.x) | ((unsigned long long)__float_as_uint(v.y) << 32)),
        "l"(0ull), "l"(acc));
  return d;
}
__device__ __forceinline__ bool not_finite(unsigned long long acc) {
  return (acc & 0x7fffffff7fffffffull) != 0ull;
}
// minima that keep a NaN
__device__ __forceinline__ float min_nan(float a, float b) {
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float min_nan(float a, float b, float c) {
  float d;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ Edge edge_pn(uint32_t P, uint32_t N) {
  Edge e;
  e.P = P;
  e.N = N;
  e.Z = P | N;
  return e;
}
__device__ __forceinline__ Edge edge_dn(const Edge& e) {
  return edge_pn(__shfl_down_sync(0xffffffffu, e.P, 1), __shfl_down_sync(0xffffffffu, e.N, 1));
}

__device__ __forceinline__ uint32_t zero_bit(float2 v) {
  return ((__float_as_uint(v.x) | __float_as_uint(v.y)) << 1) == 0u ? 1u : 0u;
}
__device__ __forceinline__ uint32_t bad_bit(float2 v) {
  return (finite_f(v.x) && finite_f(v.y)) ? 0u : 1u;
}

template <int NW, int MINB, int STAGES, bool UNAL>
__global__ void __launch_bounds__(NW * 32, MINB) sweep_bits_kernel(const __grid_constant__ BulkParams a) {
  extern __shared__ __align__(128) unsigned char dsm[];
  pdl_trigger();  // the segment scan may queue behind this grid's blocks
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int w = tid >> 5;
  constexpr int W2 = BL * NW + (UNAL ? 4 : 2);  // row pitch of a slot, in elements
  float2* ring = reinterpret_cast<float2*>(dsm);
  uint64_t* full =
      reinterpret_cast<uint64_t*>(dsm + ((size_t)STAGES * BRH * W2 + kTail) * sizeof(float2));
  uint64_t* empty = full + STAGES;
  unsigned int* s_faces = reinterpret_cast<unsigned int*>(empty + STAGES);  // [kMaxRun]
  // per warp: first node of its band's rows in the tile
  const float2** s_src = reinterpret_cast<const float2**>(s_faces + kMaxRun);
  const int xl = BL * w + lane;  // tile-local column of this lane

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1u);
      mbar_init(&empty[s], (uint32_t)NW);
    }
    fence_mbar_init();
  }
  __syncthreads();

  uint32_t fill = 0, use = 0;  // planes issued (warp 0) / consumed, counted over the whole CTA
  bool timeout = false;
  int valid_w = W2, valid_r = BRH;  // padding bookkeeping, as in the nibble sweep
  bool stk_padded = false;          // the ring holds padding outside the stacked strips
  // padding past the last slot: the lanes of the last stacked strip read up to
  // 32 NW - W2 elements beyond a slot row
  for (int i = tid; i < kTail; i += blockDim.x)
    ring[(size_t)STAGES * BRH * W2 + i] = make_float2(1.f, 1.f);

  const long long U = a.units;
  long long u = U * blockIdx.x / gridDim.x;
  const long long uend = U * (blockIdx.x + 1) / gridDim.x;

  while (u < uend) {
    int si = 0;
    while (si + 1 < a.nsnap && a.s[si + 1].unit0 <= u) ++si;
    const SnapDesc& sd = a.s[si];
    const int nx = sd.nx, ny = sd.ny, nz = sd.nz, ntx = sd.ntx;
    // columns: (band, tile) of the tiles before the last, then (with
    // stacking) groups of NW bands whose narrow last tiles share a CTA, one
    // band per warp, else (band, tile) of every tile
    const int ntn = sd.nstk ? ntx - 1 : ntx;
    const long long nnorm = (long long)sd.nbands * ntn;
    long long col;
    int kb, kblk;
    unit_pos(u - sd.unit0, nnorm + sd.nstk, nz, sd.hblock, col, kb, kblk);
    const bool stk = col >= nnorm;
    const int band0 = stk ? (int)(col - nnorm) * NW : 0;  // first band of a stacked group
    const int band = stk ? band0 + w : (int)(col / ntn);  // this warp's band
    const int tile = stk ? ntx - 1 : (int)(col % ntn);
    const bool wok = band < sd.nbands;  // a stacked group may hold fewer than NW bands
    const int ke = (int)min(min((long long)kblk, (long long)kb + (uend - u)), (long long)kb + kMaxRun);
    u += ke - kb;
    const int j0 = band * BR;
    const int nrows = wok ? min(BRH, ny - j0) : 0;
    const int klast = min(ke, nz - 1);
    const int nplanes = klast - kb + 1;
    const int nsteps = ke - kb;
    const int xt0 = tile * sd.st;
    const bool last_tile = tile == ntx - 1;
    // (an odd row may leave its last tile one column, which the tile before
    // stages as its halo)
    const int tw = last_tile ? nx - xt0 : (UNAL ? min(sd.st + 2, nx - xt0) : sd.st + 2);
    const int own_end = last_tile ? tw : sd.st;
    const uint32_t row_bytes = (uint32_t)tw * 8u;
    // first node of this warp's band (stacked) or the CTA's band in the tile,
    // kept in shared memory (read once per plane by the copying lanes)
    __syncwarp();
    if (lane == 0) s_src[w] = sd.psi + (size_t)(wok ? band * BR : 0) * nx + xt0;
    __syncwarp();
    // tile-local column of this lane, and its column in a slot (a stacked
    // group puts band band0 + v at slot columns 32 v ..)
    const int xs = stk ? lane : xl;
    const int xc = stk ? 32 * w + lane : xl;

    if (stk) {
      if (!stk_padded) {
        for (int idx = tid; idx < STAGES * BRH * W2; idx += blockDim.x)
          ring[idx] = UNAL ? pad_value(idx / W2 % BRH, idx % W2, idx / (BRH * W2))
                           : make_float2(1.f, 1.f);
        fence_proxy_async();
        __syncthreads();
        stk_padded = true;
      }
      valid_w = W2;  // a later unstacked run re-pads what it needs
      valid_r = BRH;
    } else {
      stk_padded = false;
      // unaligned rows shift within their slot rows from plane to plane, so no
      // column padding holds; lanes past the tile are left out of the test for
      // special values instead (colv)
      const int vw = UNAL ? W2 : tw;
      if (vw < valid_w || nrows < valid_r) {
        const int cw = valid_w - vw;
        if (cw > 0)
          for (int idx = tid; idx < STAGES * BRH * cw; idx += blockDim.x)
            ring[(size_t)(idx / cw) * W2 + vw + idx % cw] = make_float2(1.f, 1.f);
        const int rr = valid_r - nrows;
        if (rr > 0) {
          const int per = rr * W2;
          for (int idx = tid; idx < STAGES * per; idx += blockDim.x) {
            const int sl = idx / per, rem = idx % per;
            ring[((size_t)sl * BRH + nrows + rem / W2) * W2 + rem % W2] =
                UNAL ? pad_value(nrows + rem / W2, rem % W2, sl) : make_float2(1.f, 1.f);
          }
        }
        fence_proxy_async();
        __syncthreads();
      }
      valid_w = vw;
      valid_r = nrows;
    }
    for (int i = tid; i < nsteps; i += blockDim.x) s_faces[i] = 0u;
    __syncthreads();

    // unaligned rows: shift of the even rows of the band in their slot rows
    // in plane m (the odd rows' is the other one where nx is odd)
    const uint32_t sh0 = UNAL && !stk
                             ? (uint32_t)(reinterpret_cast<uintptr_t>(sd.psi) >> 3) ^
                                   (uint32_t)((j0 & nx) ^ xt0)
                             : 0u;
    const uint32_t shm = UNAL && !stk ? (uint32_t)(nx & ny & 1) : 0u;
    const uint32_t shr = UNAL && !stk ? (uint32_t)(nx & 1) : 0u;
    auto shift = [&](int m) -> uint32_t { return (sh0 ^ ((uint32_t)m & shm)) & 1u; };
    const bool colv = !UNAL || (wok && xs < tw);  // this lane's column is in the tile

    // warp 0: plane m into the next slot once every warp has released it
    auto produce = [&](int m) {
      const uint32_t q = fill;
      const int sl = (int)(q % STAGES);
      if (q >= (uint32_t)STAGES && !mbar_wait(&empty[sl], ((q / STAGES) - 1u) & 1u)) timeout = true;
      if constexpr (UNAL) {
        // Row `lane`, elements [lo, hi): widened to 16-byte boundaries, which
        // adds neighbours in the field.
        const float2* src = s_src[0] + (size_t)m * ((size_t)nx * ny) + (size_t)lane * nx;
        const uint32_t she = shift(m), sho = she ^ shr;
        const int sh = (int)(lane & 1 ? sho : she);
        float2* dst = ring + ((size_t)sl * BRH + lane) * W2 + sh;  // element 0 of the row
        if (m != 0 && m != nz - 1) {
          const uint32_t be = (((uint32_t)tw + she + 1u) & ~1u) * 8u;
          const uint32_t bo = (((uint32_t)tw + sho + 1u) & ~1u) * 8u;
          if (lane == 0) {
            fence_proxy_async();
            mbar_arrive_expect_tx(&full[sl], be * (uint32_t)((nrows + 1) >> 1) +
                                                 bo * (uint32_t)(nrows >> 1));
          }
          __syncwarp();
          if (lane < nrows) bulk_g2s(dst - sh, src - sh, lane & 1 ? bo : be, &full[sl]);
          ++fill;
          return;
        }
        // The first and the last plane: nothing lies before the field's first
        // element and after its last one; there one element is left to a plain
        // copy.
        int lo = -sh, hi = tw + ((tw + sh) & 1);
        if (lane < nrows) {
          if (sh && src == sd.psi) {
            lo = 1;
            dst[0] = src[0];
            fence_proxy_async();
          }
          if (hi > tw && src + tw == sd.psi + (size_t)nx * ny * nz) {
            hi = tw - 1;
            dst[hi] = src[hi];
            fence_proxy_async();
          }
        } else {
          lo = hi = 0;
        }
        const uint32_t bytes = hi > lo ? (uint32_t)(hi - lo) * 8u : 0u;
        const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
        __syncwarp();  // the plain copies come before the arrival
        if (lane == 0) {
          fence_proxy_async();
          mbar_arrive_expect_tx(&full[sl], total);
        }
        __syncwarp();
        if (bytes) bulk_g2s(dst + lo, src + lo, bytes, &full[sl]);
        ++fill;
        return;
      }
      if (lane == 0) {
        fence_proxy_async();
        mbar_arrive_expect_tx(&full[sl], row_bytes * (uint32_t)nrows);
      }
      __syncwarp();
      if (lane < nrows)
        bulk_g2s(ring + ((size_t)sl * BRH + lane) * W2,
                 s_src[0] + (size_t)m * ((size_t)nx * ny) + (size_t)lane * nx, row_bytes, &full[sl]);
      ++fill;
    };
    // Stacked group: each warp fills and reads only its own strip, so the
    // warps run independently, with 16-byte cp.async copies (a strip row is
    // too short for a bulk copy to pay) in one commit group per plane.  Lane
    // chunks: (row, 16-byte column pair) = (r0, c0) + i (dr, dc), row-major.
    // (plane m of a run sits in slot (m - kb) % STAGES)
    auto sfill = [&](int m) {
      if (m <= klast && wok) {
        // 16-byte chunks of a strip row (tw is even), 8-byte ones unaligned
        constexpr int CE = UNAL ? 1 : 2;
        const int nch = UNAL ? tw : (int)(row_bytes >> 4);
        const float2* src = s_src[w] + (size_t)m * ((size_t)nx * ny);
        float2* dst = ring + (size_t)((m - kb) % STAGES) * BRH * W2 + 32 * w;
        const int dr = 32 / nch, dc = 32 - dr * nch;
        int r = lane / nch, c = lane - (lane / nch) * nch;
        while (r < nrows) {
          if constexpr (UNAL) cp_async8(dst + r * W2 + c, src + (size_t)r * nx + c);
          else cp_async16(dst + r * W2 + CE * c, src + (size_t)r * nx + CE * c);
          r += dr;
          c += dc;
          if (c >= nch) {
            c -= nch;
            ++r;
          }
        }
      }
      cp_async_commit();
    };
    auto acquire = [&](int m) -> const float2* {
      if (stk) {
        cp_async_wait<STAGES - 1>();
        __syncwarp();
        return ring + (size_t)((m - kb) % STAGES) * BRH * W2;
      }
      const int sl = (int)(use % STAGES);
      if (!mbar_wait(&full[sl], (use / STAGES) & 1u)) timeout = true;
      return ring + (size_t)sl * BRH * W2;
    };
    // done with plane m (a stacked warp refills its strip's slot at once)
    auto release = [&](int m) {
      __syncwarp();
      if (stk) {
        sfill(m + STAGES);
        return;
      }
      if (lane == 0) mbar_arrive(&empty[use % STAGES]);
      ++use;
    };

    // masks of the faces this lane owns (rows 0..15 of the band)
    const int avail = wok ? ny - j0 : 0;  // rows of the band that exist
    const uint32_t rv = avail >= BR ? kRows16 : ((1u << avail) - 1u);
    const uint32_t rv1 = avail - 1 >= BR ? kRows16 : (avail > 1 ? ((1u << (avail - 1)) - 1u) : 0u);
    const bool own = wok && lane < BL && xs < own_end;
    const uint32_t m_xy = (own && xs + 1 < tw) ? rv1 : 0u;
    const uint32_t m_yz = (own && xs < tw) ? rv1 : 0u;
    const uint32_t m_zx = (own && xs + 1 < tw) ? rv : 0u;
    // table entries of this (band, tile, warp): one per plane, contiguous in k;
    // records of entry e in the fixed slots 32 e .. 32 e + 31 (one per lane).
    // A stacked warp is warp 0 of its band's last tile; that tile's other
    // warps own no columns and get empty entries.
    const unsigned long long ebase =
        (unsigned long long)sd.tab0 +
        (((unsigned long long)band * ntx + tile) * NW + (stk ? 0 : w)) * nz;
    uint2* const table = reinterpret_cast<uint2*>(a.table);
    uint4* const recs = reinterpret_cast<uint4*>(a.recs);
    uint2 tent = make_uint2(0u, 0u);  // entry of step t held by lane t % 32

    if (stk) {
      for (int i = 0; i < STAGES; ++i) sfill(kb + i);
    } else if (w == 0) {
      for (int i = 0; i < min(STAGES, nplanes); ++i) produce(kb + i);
    }

    // unaligned rows: whether the lane's x edges count, exact half-planes and edges
    // of a plane
    const bool xedges = colv && lane < BL && xs + 1 < tw;
    auto half_planes = [&](const float2(&V)[BRH]) -> uint32_t {
      uint32_t b = 0;
#pragma unroll
      for (int r = 0; r < BRH; ++r) b |= (V[r].y < 0.f ? 1u : 0u) << r;
      return b;
    };
    // Edges of one direction again: in the rows in which a doubtful lane (bad) has an
    // edge between half-planes (Sa and Sb, exact), for all lanes.  to(r) is the node at
    // the other end of V's edge in row r.  Whether there was such a row.
    auto redo = [&](const float2(&V)[BRH], bool bad, uint32_t Sa, uint32_t Sb, uint32_t mask, Edge& E,
                    auto to) -> bool {
      const uint32_t rows = __reduce_or_sync(0xffffffffu, bad ? (Sa ^ Sb) & mask : 0u);
      if (!rows) return false;
      uint32_t G = 0, L = 0;
#pragma unroll
      for (int r = 0; r < BRH; ++r) {
        if (!((rows >> r) & 1u)) continue;
        exact_compare(V[r], to(r), 1u << r, G, L);
      }
      E = edge_pn((E.P & ~rows) | (~Sa & Sb & G), (E.N & ~rows) | (Sa & ~Sb & L));
      return true;
    };
    auto redo_xy = [&](const float2(&V)[BRH], bool badx, bool bady, uint32_t S, uint32_t Sn, Edge& X,
                       Edge& Y, Edge& Yn) -> bool {
      const bool ox = redo(V, badx, S, Sn, kRowsHeld, X, [&](int r) {
        return make_float2(__shfl_down_sync(0xffffffffu, V[r].x, 1), __shfl_down_sync(0xffffffffu, V[r].y, 1));
      });
      const bool oy = redo(V, bady, S, S >> 1, kRows16, Y, [&](int r) { return V[r < BR ? r + 1 : r]; });
      if (oy) Yn = edge_dn(Y);
      return ox || oy;
    };

    // ---- prologue: plane kb (values into vA)
    float2 vA[BRH], vB[BRH];
    uint32_t S0, S0n, ZB0 = 0, ZB0n = 0, BB0 = 0, BB0n = 0;
    Edge X0, Y0, Y0n;
    bool bad0;         // aligned: a special node in plane k; unaligned: one that is not finite
    bool redone0 = false;  // unaligned: edges of plane k taken again
    {
      const float2* sp = acquire(kb);
      const int xe = xc + (UNAL ? (int)shift(kb) : 0), xo = UNAL ? xc + (int)(shift(kb) ^ shr) : xe;
      uint32_t SX = 0, SY = 0;
      unsigned long long prod = UNAL ? 0ull : kProdOne;
      float mx = kTieFar, my = kTieFar;
      S0 = 0;
#pragma unroll
      for (int r = BRH - 1; r >= 0; --r) {
        const float2 v = sp[r * W2 + (r & 1 ? xo : xe)];
        const float2 nb = sp[r * W2 + (r & 1 ? xo : xe) + 1];
        S0 = push1(S0, v.y);
        if constexpr (UNAL) {
          float m1, m2 = kTieFar;
          SX = push1(SX, cross_m(v, nb, m1));
          mx = min_nan(mx, m1);
          if (r < BR) SY = push1(SY, cross_m(v, vA[r + 1], m2));
          my = min_nan(my, m2, fabsf(v.y));
        } else {
          SX = push1(SX, cross_f(v.x, v.y, nb.x, nb.y));
          if (r < BR) SY = push1(SY, cross_f(v.x, v.y, vA[r + 1].x, vA[r + 1].y));
        }
        prod = UNAL ? finite_step(prod, v) : prod_step(prod, v);
        vA[r] = v;
      }
      release(kb);
      if (w == 0 && !stk && kb + STAGES <= klast) produce(kb + STAGES);
      bool badx = false, bady = false, again = false;
      if constexpr (UNAL) {
        badx = xedges && !(mx > 0.f);
        bady = colv && !(my > 0.f);
        again = __any_sync(0xffffffffu, badx || bady);
        bad0 = __any_sync(0xffffffffu, colv && not_finite(prod));
        if (again) S0 = half_planes(vA);
      } else {
        bad0 = __any_sync(0xffffffffu, prod_special(prod));
      }
      if (bad0) {
#pragma unroll
        for (int r = 0; r < BRH; ++r) {
          if constexpr (!UNAL) ZB0 |= zero_bit(vA[r]) << r;
          BB0 |= bad_bit(vA[r]) << r;
        }
      }
      S0n = __shfl_down_sync(0xffffffffu, S0, 1);
      const uint32_t SYn = __shfl_down_sync(0xffffffffu, SY, 1);
      ZB0n = __shfl_down_sync(0xffffffffu, ZB0, 1);
      BB0n = __shfl_down_sync(0xffffffffu, BB0, 1);
      X0 = edge_words(S0, S0n, SX, ZB0 | ZB0n);
      Y0 = edge_words(S0, S0 >> 1, SY, ZB0 | (ZB0 >> 1));
      Y0n = edge_words(S0n, S0n >> 1, SYn, ZB0n | (ZB0n >> 1));
      if constexpr (UNAL)
        if (again) redone0 = redo_xy(vA, badx, bady, S0, S0n, X0, Y0, Y0n);
    }

    // one z step: plane k = kb + t in V0 (values) and the plane-k words,
    // plane k + 1 read into V1
    auto step = [&](float2(&V0)[BRH], float2(&V1)[BRH], int t) {
      const int k = kb + t;
      const bool has_up = k + 1 < nz;
      uint32_t Lxy, Hxy, Lyz = 0, Hyz = 0, Lzx = 0, Hzx = 0;
      // xy faces of plane k: +x(r), +y_{x+1}(r), -x(r+1), -y_x(r)
      mod4(X0.Z, X0.N, Y0n.Z, Y0n.N, X0.Z >> 1, X0.P >> 1, Y0.Z, Y0.P, Lxy, Hxy);
      uint32_t Mxy = (Lxy | Hxy) & m_xy, Myz = 0, Mzx = 0;
      uint32_t S1 = 0, S1n = 0, ZB1 = 0, ZB1n = 0, BB1 = 0, BB1n = 0;
      Edge X1{0, 0, 0}, Y1{0, 0, 0}, Y1n{0, 0, 0};
      bool bad1 = false, redone1 = false, redonez = false;
      if (has_up) {
        const float2* sp = acquire(k + 1);
        const int xe = xc + (UNAL ? (int)shift(k + 1) : 0);
        const int xo = UNAL ? xc + (int)(shift(k + 1) ^ shr) : xe;
        uint32_t SX = 0, SY = 0, SZ = 0;
        unsigned long long prod = UNAL ? 0ull : kProdOne;
        float mx = kTieFar, my = kTieFar, mz = kTieFar, hx = 0.f, hz = 0.f;
#pragma unroll
        for (int r = BRH - 1; r >= 0; --r) {
          const float2 v = sp[r * W2 + (r & 1 ? xo : xe)];
          const float2 nb = sp[r * W2 + (r & 1 ? xo : xe) + 1];
          S1 = push1(S1, v.y);
          if constexpr (UNAL) {
            float m1, m2 = kTieFar, m3;
            SX = push1(SX, cross_m(v, nb, m1));
            SZ = push1(SZ, cross_m(V0[r], v, m3));
            if (r < BR) SY = push1(SY, cross_m(v, V1[r + 1], m2));
            my = min_nan(my, m2, fabsf(v.y));
            // the margins of two rows in one minimum
            if (r & 1) {
              mx = min_nan(mx, hx, m1);
              mz = min_nan(mz, hz, m3);
            } else if (r == 0) {
              mx = min_nan(mx, m1);
              mz = min_nan(mz, m3);
            } else {
              hx = m1;
              hz = m3;
            }
          } else {
            SX = push1(SX, cross_f(v.x, v.y, nb.x, nb.y));
            SZ = push1(SZ, cross_f(V0[r].x, V0[r].y, v.x, v.y));
            if (r < BR) SY = push1(SY, cross_f(v.x, v.y, V1[r + 1].x, V1[r + 1].y));
          }
          prod = UNAL ? finite_step(prod, v) : prod_step(prod, v);
          V1[r] = v;
        }
        release(k + 1);
        if (w == 0 && !stk && k + 1 + STAGES <= klast) produce(k + 1 + STAGES);
        Edge Zk, Zkn;
        if constexpr (UNAL) {
          const bool badx = xedges && !(mx > 0.f), bady = colv && !(my > 0.f), badz = colv && !(mz > 0.f);
          const bool again = __any_sync(0xffffffffu, badx || bady || badz);
          bad1 = __any_sync(0xffffffffu, colv && not_finite(prod));
          if (again) S1 = half_planes(V1);
          S1n = __shfl_down_sync(0xffffffffu, S1, 1);
          const uint32_t SYn = __shfl_down_sync(0xffffffffu, SY, 1);
          const uint32_t SZn = __shfl_down_sync(0xffffffffu, SZ, 1);
          if (bad1) {
#pragma unroll
            for (int r = 0; r < BRH; ++r) BB1 |= bad_bit(V1[r]) << r;
            BB1n = __shfl_down_sync(0xffffffffu, BB1, 1);
          }
          X1 = edge_words(S1, S1n, SX);
          Y1 = edge_words(S1, S1 >> 1, SY);
          Y1n = edge_words(S1n, S1n >> 1, SYn);
          Zk = edge_words(S0, S1, SZ);
          Zkn = edge_words(S0n, S1n, SZn);
          if (again) {
            redone1 = redo_xy(V1, badx, bady, S1, S1n, X1, Y1, Y1n);
            redonez = redo(V0, badz, S0, S1, kRowsHeld, Zk, [&](int r) { return V1[r]; });
            if (redonez) Zkn = edge_dn(Zk);
          }
        } else {
          bad1 = __any_sync(0xffffffffu, prod_special(prod));
          S1n = __shfl_down_sync(0xffffffffu, S1, 1);
          const uint32_t SYn = __shfl_down_sync(0xffffffffu, SY, 1);
          const uint32_t SZn = __shfl_down_sync(0xffffffffu, SZ, 1);
          if (bad0 || bad1) {
            if (bad1) {
#pragma unroll
              for (int r = 0; r < BRH; ++r) {
                ZB1 |= zero_bit(V1[r]) << r;
                BB1 |= bad_bit(V1[r]) << r;
              }
            }
            ZB1n = __shfl_down_sync(0xffffffffu, ZB1, 1);
            BB1n = __shfl_down_sync(0xffffffffu, BB1, 1);
            X1 = edge_words(S1, S1n, SX, ZB1 | ZB1n);
            Y1 = edge_words(S1, S1 >> 1, SY, ZB1 | (ZB1 >> 1));
            Y1n = edge_words(S1n, S1n >> 1, SYn, ZB1n | (ZB1n >> 1));
            Zk = edge_words(S0, S1, SZ, ZB0 | ZB1);
            Zkn = edge_words(S0n, S1n, SZn, ZB0n | ZB1n);
          } else {
            X1 = edge_words(S1, S1n, SX);
            Y1 = edge_words(S1, S1 >> 1, SY);
            Y1n = edge_words(S1n, S1n >> 1, SYn);
            Zk = edge_words(S0, S1, SZ);
            Zkn = edge_words(S0n, S1n, SZn);
          }
        }
        // yz faces of plane k: +y_k(r), +z(r+1), -y_{k+1}(r), -z(r)
        mod4(Y0.Z, Y0.N, Zk.Z >> 1, Zk.N >> 1, Y1.Z, Y1.P, Zk.Z, Zk.P, Lyz, Hyz);
        // zx faces of plane k: +z_x(r), +x_{k+1}(r), -z_{x+1}(r), -x_k(r)
        mod4(Zk.Z, Zk.N, X1.Z, X1.N, Zkn.Z, Zkn.P, X0.Z, X0.P, Lzx, Hzx);
        Myz = (Lyz | Hyz) & m_yz;
        Mzx = (Lzx | Hzx) & m_zx;
      }
      if (bad0 || bad1) {  // drop faces that touch a non-finite node
        Mxy &= ~(BB0 | BB0n | (BB0 >> 1) | (BB0n >> 1));
        Myz &= ~(BB0 | (BB0 >> 1) | BB1 | (BB1 >> 1));
        Mzx &= ~(BB0 | BB0n | BB1 | BB1n);
      }
      // W = -2 shares the code of 2; a sum of -2 needs an edge whose determinant
      // underflows or overflows between half-planes, so the expand pass takes it from psi
      uint32_t mark = 0;
      if constexpr (UNAL)
        if (redone0 || redone1 || redonez)
          mark = ((~Lxy & Hxy & Mxy) | (~Lyz & Hyz & Myz) | (~Lzx & Hzx & Mzx)) ? kRecordTwos : 0u;
      Lxy &= Mxy;
      Hxy &= Mxy;
      Lyz &= Myz;
      Hyz &= Myz;
      Lzx &= Mzx;
      Hzx &= Mzx;
      const uint32_t cnt = __popc(Mxy) + __popc(Myz) + __popc(Mzx);
      const bool anyf = cnt != 0u;

      // ---- output: records in the fixed slots of this warp step, the
      // table entry (lane mask, faces) held by lane t % 32 and stored for 32
      // steps at once, the face total added to the CTA's count of plane k
      const uint32_t faces_w = __reduce_add_sync(0xffffffffu, cnt);
      const uint32_t bal = __ballot_sync(0xffffffffu, anyf);
      const unsigned long long e = ebase + (unsigned long long)k;
      if (anyf && e * 32ull + lane < a.recs_cap)
        recs[e * 32ull + lane] =
            make_uint4(Lxy | (Hxy << 16), Lyz | (Hyz << 16), Lzx | (Hzx << 16), (uint32_t)lane | mark);
      if (lane == (t & 31)) tent = make_uint2(bal, faces_w);
      if (((t & 31) == 31 || t == nsteps - 1) && wok) {
        if (lane <= (t & 31)) {
          const unsigned long long ei = ebase + (unsigned long long)(kb + (t & ~31) + lane);
          table[ei] = tent;
          if (stk)
            for (int v = 1; v < NW; ++v) table[ei + (unsigned long long)v * nz] = make_uint2(0u, 0u);
        }
      }
      if (lane == 0 && faces_w) {
        if (stk) atomicAdd(&a.segf[sd.seg0 + (size_t)k * sd.nbands + band], faces_w);
        else atomicAdd(&s_faces[t], faces_w);
      }
      // plane k + 1 becomes plane k
      S0 = S1;
      S0n = S1n;
      ZB0 = ZB1;
      ZB0n = ZB1n;
      BB0 = BB1;
      BB0n = BB1n;
      X0 = X1;
      Y0 = Y1;
      Y0n = Y1n;
      bad0 = bad1;
      redone0 = redone1;
    };

    for (int t = 0; t < nsteps; t += 2) {
      step(vA, vB, t);
      if (t + 1 < nsteps) step(vB, vA, t + 1);
    }
    if (stk) cp_async_wait<0>();  // only empty groups are left
    __syncthreads();
    // face totals of the run's planes into the (plane, band) segments
    for (int i = tid; i < nsteps; i += blockDim.x)
      if (s_faces[i]) atomicAdd(&a.segf[sd.seg0 + (size_t)(kb + i) * sd.nbands + band], s_faces[i]);
    __syncthreads();
  }
  if (timeout) atomicOr(reinterpret_cast<unsigned int*>(a.counters + 1), 1u);
}

using BitsFn = void (*)(BulkParams);

template <int STAGES, bool UNAL>
BitsFn bits_fn_stages(int nw) {
  if (nw <= 2) return sweep_bits_kernel<2, 8, STAGES, UNAL>;
  if (nw <= 4) return sweep_bits_kernel<4, 4, STAGES, UNAL>;
  return sweep_bits_kernel<8, 2, STAGES, UNAL>;
}

BitsFn bits_fn(int nw, int stages, bool unal) {
  if (unal) return stages <= 2 ? bits_fn_stages<2, true>(nw) : bits_fn_stages<3, true>(nw);
  return stages <= 2 ? bits_fn_stages<2, false>(nw) : bits_fn_stages<3, false>(nw);
}

int bits_fn_index(int nw, int stages, bool unal) {
  return (nw <= 2 ? 0 : (nw <= 4 ? 1 : 2)) + (stages <= 2 ? 0 : 3) + (unal ? 6 : 0);
}

}  // namespace

size_t bits_smem_bytes(int nw, int stages, bool unal) {
  return ((size_t)stages * BRH * (BL * nw + (unal ? 4 : 2)) + kTail) * sizeof(float2) +
         2 * stages * sizeof(uint64_t) + kMaxRun * sizeof(unsigned int) +
         (size_t)nw * sizeof(const float2*);
}

int bits_variant_occupancy(int nw, int stages, bool unal, int* ctas_per_sm, size_t* smem) {
  static bool attr_set[12] = {};
  if (nw != 2 && nw != 4 && nw != 8)
    return set_error(QTV_ERR_ARG, "bit-sliced sweep: %d warps per tile (2, 4 or 8)", nw);
  const int which = bits_fn_index(nw, stages, unal);
  BitsFn fn = bits_fn(nw, stages, unal);
  if (!attr_set[which]) {
    cudaError_t e =
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return check_cuda(e, "cudaFuncSetAttribute(sweep_bits)");
    attr_set[which] = true;
  }
  *smem = bits_smem_bytes(nw, stages, unal);
  int bps = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn, nw * 32, *smem);
  if (e != cudaSuccess) return check_cuda(e, "occupancy(sweep_bits)");
  if (bps < 1) return set_error(QTV_ERR_ARG, "sweep_bits: no resident CTA with %d warps", nw);
  *ctas_per_sm = bps;
  return QTV_OK;
}

void bits_sweep_launch(const BulkParams& p, int grid, int nw, int stages, bool unal, size_t smem,
                       cudaStream_t st) {
  bits_fn(nw, stages, unal)<<<grid, nw * 32, smem, st>>>(p);
}


}  // namespace qtv
