// refine.cu -- sample refinement of Sec. 3.3.3 ("Locating more accurate
// sample points") on the GPU: an estimate x0 of a core sample is moved to a
// minimizer of the density rho = |psi|^2 (Eq. 6) within the plane through x0
// perpendicular to the local core direction t, which the paper takes from the
// pseudo-vorticity t = grad Re psi x grad Im psi.
//
// Arithmetic, per sample (one thread; FP32):
//   - psi between nodes is the trilinear interpolant; rho and grad rho are
//     those of the interpolant within the cell floor(x) (cell index clamped
//     to [0, n - 2]);
//   - grad Re psi and grad Im psi at x0 are the central-difference node
//     gradients (one-sided on the boundary, 0 along an axis of one node),
//     interpolated trilinearly; t is their cross product, normalized;
//   - descent on g = grad rho - (grad rho . t) t: each step starts at
//     alpha = 2 rho / |g|^2 (the exact step for a round bowl whose minimum is
//     0) and halves alpha until rho(x - alpha g) <= rho(x) - 1e-4 alpha |g|^2
//     with the new point in the grid and in the box |x - x0|_inf <= 1 (a step
//     leaving either is rejected, not projected); it stops, converged, when
//     no step of length >= tol decreases rho that way, or after max_iter
//     accepted steps.
// Positions are carried as an integer base (the cell of x0) plus an FP32
// offset, so steps far below the FP32 spacing of absolute coordinates still
// move the point.  Warps are persistent and each lane takes a new sample when
// its search ends (the number of steps varies from 0 to max_iter).
#include <climits>
#include <cstdio>

#include "qtv_internal.cuh"

namespace qtv {
namespace {

constexpr int REF_THREADS = 128, REF_CTAS = 5;

struct RefArgs {
  const float2* psi;
  int nx, ny, nz;
  float h, ox, oy, oz;
  const float* xyz0;          // world positions [n][3], or null
  const uint64_t* face_ids;   // faces whose centres are x0, or null
  unsigned long long n;
  const uint64_t* n_dev;
  int max_iter;
  float tol;
  float* xyz;
  float* rho;
  float* tangent;
  float* detj;
  int32_t* iters;
  uint8_t* flags;
};

struct Field {
  const float2* psi;
  int n[3];
  __device__ __forceinline__ float2 at(int i, int j, int k) const {
    return __ldg(psi + ((long long)k * n[1] + j) * n[0] + i);
  }
};

// cell and fraction of base + off along an axis of m nodes
__device__ __forceinline__ void cell_frac(int base, float off, int m, int& c, float& f) {
  const float fl = floorf(off);
  c = base + (int)fl;
  f = off - fl;
  const int hi = max(m - 2, 0);
  if (c > hi) {
    f += (float)(c - hi);
    c = hi;
  }
  if (c < 0) {
    f += (float)c;
    c = 0;
  }
}

// trilinear psi at the point (cells c, fractions f) and its partial derivatives
__device__ __forceinline__ float2 tri_eval(const Field& F, const int c[3], const float f[3],
                                           float2 d[3]) {
  float2 acc = make_float2(0.f, 0.f);
  d[0] = d[1] = d[2] = make_float2(0.f, 0.f);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    int idx[3];
    float w[3], s[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int bit = (q >> a) & 1;
      idx[a] = c[a] + bit < F.n[a] ? c[a] + bit : c[a];
      w[a] = bit ? f[a] : 1.f - f[a];
      s[a] = bit ? 1.f : -1.f;
    }
    const float2 v = F.at(idx[0], idx[1], idx[2]);
    const float wt = w[0] * w[1] * w[2];
    acc.x = fmaf(wt, v.x, acc.x);
    acc.y = fmaf(wt, v.y, acc.y);
    const float dd[3] = {s[0] * w[1] * w[2], w[0] * s[1] * w[2], w[0] * w[1] * s[2]};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      d[a].x = fmaf(dd[a], v.x, d[a].x);
      d[a].y = fmaf(dd[a], v.y, d[a].y);
    }
  }
  return acc;
}

// central-difference gradient of psi at node (i,j,k) along axis a
__device__ __forceinline__ float2 node_grad(const Field& F, int i, int j, int k, int a) {
  int p[3] = {i, j, k}, q[3] = {i, j, k};
  const int m = F.n[a];
  if (m < 2) return make_float2(0.f, 0.f);
  float s = 0.5f;
  if (p[a] == 0) {
    q[a] = 1;
    s = 1.f;
  } else if (p[a] == m - 1) {
    p[a] = m - 2;
    s = 1.f;
  } else {
    p[a] -= 1;
    q[a] += 1;
  }
  const float2 lo = F.at(p[0], p[1], p[2]), hi = F.at(q[0], q[1], q[2]);
  return make_float2(s * (hi.x - lo.x), s * (hi.y - lo.y));
}

struct Pos {
  int base[3];    // integer base (cell of x0)
  float off[3];   // offset from the base
};

__device__ __forceinline__ bool pos_inside(const Pos& P, const int n[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float v = (float)P.base[a] + P.off[a];
    if (!(P.off[a] >= -(float)P.base[a] && v <= (float)(n[a] - 1))) return false;
  }
  return true;
}

// The eight corner values of the cell last evaluated: a search rarely
// leaves its cell, so most evaluations read no memory.
struct CellCache {
  int c[3];
  float2 v[8];
};

// x . y with the roundings of fma(x2, y2, fma(x0, y0, x1 y1)).  Where products
// meet sums in this file the roundings are written out: a search of 200 steps
// amplifies any other choice.
__device__ __forceinline__ float dot3(const float x[3], const float y[3]) {
  return fmaf(x[2], y[2], fmaf(x[0], y[0], __fmul_rn(x[1], y[1])));
}

// rho and grad rho at P: trilinear psi and its derivatives from the corners
// in the same order and arithmetic as tri_eval
__device__ __forceinline__ float rho_at(const Field& F, const Pos& P, float g[3], CellCache& C) {
  int c[3];
  float f[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) cell_frac(P.base[a], P.off[a], F.n[a], c[a], f[a]);
  if (c[0] != C.c[0] || c[1] != C.c[1] || c[2] != C.c[2]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      int idx[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int bit = (q >> a) & 1;
        idx[a] = c[a] + bit < F.n[a] ? c[a] + bit : c[a];
      }
      C.v[q] = F.at(idx[0], idx[1], idx[2]);
    }
    C.c[0] = c[0];
    C.c[1] = c[1];
    C.c[2] = c[2];
  }
  float2 v = make_float2(0.f, 0.f);
  float2 d[3];
  d[0] = d[1] = d[2] = make_float2(0.f, 0.f);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    float w[3], s[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int bit = (q >> a) & 1;
      w[a] = bit ? f[a] : 1.f - f[a];
      s[a] = bit ? 1.f : -1.f;
    }
    const float2 u = C.v[q];
    const float wt = w[0] * w[1] * w[2];
    v.x = fmaf(wt, u.x, v.x);
    v.y = fmaf(wt, u.y, v.y);
    const float dd[3] = {s[0] * w[1] * w[2], w[0] * s[1] * w[2], w[0] * w[1] * s[2]};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      d[a].x = fmaf(dd[a], u.x, d[a].x);
      d[a].y = fmaf(dd[a], u.y, d[a].y);
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) g[a] = __fmul_rn(2.f, fmaf(v.x, d[a].x, __fmul_rn(v.y, d[a].y)));
  return fmaf(v.x, v.x, __fmul_rn(v.y, v.y));
}

// state of one sample's search
struct RState {
  Pos P0, P;
  float t[3];
  float rho;
  float grad[3];  // in-plane gradient of the running line search once it has begun
  float gg, gn;   // its square and length
  float alpha;    // step of the next candidate
  int it;
  uint8_t fl;
  unsigned long long qi;
  CellCache cache;
};

// x0, tangent, rho and grad rho at x0; true when the descent is to run
__device__ __forceinline__ bool ref_init(const RefArgs& A, const Field& F, unsigned long long qi,
                                         RState& S) {
  const float org[3] = {A.ox, A.oy, A.oz};
  S.qi = qi;
  S.it = 0;
  S.cache.c[0] = -1;  // no cell loaded
  S.t[0] = S.t[1] = S.t[2] = 0.f;
  S.rho = __int_as_float(0x7fc00000);
  bool in0 = true;
  if (A.face_ids) {
    const uint64_t id = A.face_ids[qi];
    const int o = (int)(id & 3u);
    const unsigned long long lin = id >> 2;
    long long i, j, k;
    split_lin(lin, A.nx, A.ny, i, j, k);
    S.P0.base[0] = (int)i;
    S.P0.base[1] = (int)j;
    S.P0.base[2] = (int)k;
    // face centre: half a cell along the two in-plane axes
    S.P0.off[0] = (o == 0 || o == 2) ? 0.5f : 0.f;
    S.P0.off[1] = (o == 0 || o == 1) ? 0.5f : 0.f;
    S.P0.off[2] = (o == 1 || o == 2) ? 0.5f : 0.f;
    in0 = pos_inside(S.P0, F.n);
  } else {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float g = (__ldg(A.xyz0 + 3 * qi + a) - org[a]) / A.h;
      const float fl = floorf(g);
      in0 = in0 && g >= 0.f && g <= (float)(F.n[a] - 1);
      S.P0.base[a] = in0 ? (int)fl : 0;
      S.P0.off[a] = in0 ? g - fl : g;
    }
  }
  S.P = S.P0;
  if (!in0) {
    S.fl = QTV_REFINE_NO_TANGENT;
    return false;
  }
  // pseudo-vorticity at x0
  int c[3];
  float f[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) cell_frac(S.P0.base[a], S.P0.off[a], F.n[a], c[a], f[a]);
  float gr[3] = {0.f, 0.f, 0.f}, gi[3] = {0.f, 0.f, 0.f};
  for (int q = 0; q < 8; ++q) {
    int idx[3];
    float wt = 1.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int bit = (q >> a) & 1;
      idx[a] = c[a] + bit < F.n[a] ? c[a] + bit : c[a];
      wt *= bit ? f[a] : 1.f - f[a];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float2 g = node_grad(F, idx[0], idx[1], idx[2], a);
      gr[a] = fmaf(wt, g.x, gr[a]);
      gi[a] = fmaf(wt, g.y, gi[a]);
    }
  }
  float t[3];
  t[0] = fmaf(gr[1], gi[2], -__fmul_rn(gr[2], gi[1]));
  t[1] = fmaf(gr[2], gi[0], -__fmul_rn(gr[0], gi[2]));
  t[2] = fmaf(gr[0], gi[1], -__fmul_rn(gr[1], gi[0]));
  const float tn = sqrtf(dot3(t, t));
  S.rho = rho_at(F, S.P, S.grad, S.cache);
  if (!(tn > 0.f) || !(tn <= 3.402823466e38f)) {
    S.fl = QTV_REFINE_NO_TANGENT;
    return false;
  }
  S.t[0] = t[0] / tn;
  S.t[1] = t[1] / tn;
  S.t[2] = t[2] / tn;
  S.fl = QTV_REFINE_MAX_ITER;
  return true;
}

// start of a line search: the in-plane gradient and the first step; true when the
// sample is done
__device__ __forceinline__ bool ref_begin(const RefArgs& A, RState& S) {
  if (S.it >= A.max_iter) return true;  // flag stays QTV_REFINE_MAX_ITER
  const float gt = dot3(S.grad, S.t);
#pragma unroll
  for (int a = 0; a < 3; ++a) S.grad[a] = fmaf(-gt, S.t[a], S.grad[a]);
  S.gg = dot3(S.grad, S.grad);
  if (!(S.gg > 0.f)) {
    S.fl = QTV_REFINE_CONVERGED;
    return true;
  }
  S.gn = sqrtf(S.gg);
  S.alpha = __fdiv_rn(__fmul_rn(2.f, S.rho), S.gg);
  if (S.alpha > 3.402823466e38f) S.alpha = 3.402823466e38f;  // infinity never halves below tol
  return false;
}

// candidate at step alpha along g from off: in the box around x0 (same base as
// x0) and inside the grid
__device__ __forceinline__ bool candidate(const Field& F, const int base[3], const float off[3],
                                          const float off0[3], const float g[3], float alpha, Pos& Pn) {
  bool ok = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Pn.base[a] = base[a];
    Pn.off[a] = fmaf(-alpha, g[a], off[a]);
    ok = ok && fabsf(Pn.off[a] - off0[a]) <= 1.f;
  }
  return ok && pos_inside(Pn, F.n);
}

__device__ __forceinline__ bool descends(float rn, float alpha, float gg, float rho) {
  return rn <= fmaf(-__fmul_rn(1e-4f, alpha), gg, rho);
}

// Evaluations of a line search by one lane, to its end; from step `whole` of the
// search on, one candidate that can be taken.
enum { kGoesOn, kTaken, kEnded };
__device__ __forceinline__ int ref_search(const RefArgs& A, const Field& F, RState& S, int whole, int& evals) {
  Pos Pn;
  float rn = 0.f, gnext[3];
  int st = kEnded;
  while (S.alpha * S.gn >= A.tol) {
    if (candidate(F, S.P.base, S.P.off, S.P0.off, S.grad, S.alpha, Pn)) {
      rn = rho_at(F, Pn, gnext, S.cache);
      ++evals;
      if (descends(rn, S.alpha, S.gg, S.rho)) {
        st = kTaken;
        break;
      }
      if (S.it >= whole) {
        S.alpha *= 0.5f;
        st = kGoesOn;
        break;
      }
    }
    S.alpha *= 0.5f;
  }
  if (st == kEnded) S.fl = QTV_REFINE_CONVERGED;
  if (st == kTaken) {
    ++S.it;
    S.P = Pn;
    S.rho = rn;
#pragma unroll
    for (int a = 0; a < 3; ++a) S.grad[a] = gnext[a];
  }
  return st;
}

// conditioning at the result and the outputs of the sample
__device__ __forceinline__ void ref_finish(const RefArgs& A, const Field& F, const RState& S) {
  float dj = 0.f;
  if (!(S.fl & QTV_REFINE_NO_TANGENT)) {
    // in-plane Jacobian of psi at the result: basis e1 = normalize(t x a), a
    // the axis least aligned with t; e2 = t x e1
    const float t[3] = {S.t[0], S.t[1], S.t[2]};
    int m = 0;
    float am = fabsf(t[0]);
    if (fabsf(t[1]) < am) {
      m = 1;
      am = fabsf(t[1]);
    }
    if (fabsf(t[2]) < am) m = 2;
    const float ax[3] = {m == 0 ? 1.f : 0.f, m == 1 ? 1.f : 0.f, m == 2 ? 1.f : 0.f};
    float e1[3] = {t[1] * ax[2] - t[2] * ax[1], t[2] * ax[0] - t[0] * ax[2],
                   t[0] * ax[1] - t[1] * ax[0]};  // exact: one component of ax is 1
    const float en = sqrtf(dot3(e1, e1));
    e1[0] /= en;
    e1[1] /= en;
    e1[2] /= en;
    const float e2[3] = {fmaf(t[1], e1[2], -__fmul_rn(t[2], e1[1])),
                         fmaf(t[2], e1[0], -__fmul_rn(t[0], e1[2])),
                         fmaf(t[0], e1[1], -__fmul_rn(t[1], e1[0]))};
    int cc[3];
    float ff[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) cell_frac(S.P.base[a], S.P.off[a], F.n[a], cc[a], ff[a]);
    float2 d[3];
    (void)tri_eval(F, cc, ff, d);
    float a1r = 0.f, a1i = 0.f, a2r = 0.f, a2i = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      a1r = fmaf(d[a].x, e1[a], a1r);
      a1i = fmaf(d[a].y, e1[a], a1i);
      a2r = fmaf(d[a].x, e2[a], a2r);
      a2i = fmaf(d[a].y, e2[a], a2i);
    }
    dj = fmaf(a1r, a2i, -__fmul_rn(a2r, a1i));
  }
  const float org[3] = {A.ox, A.oy, A.oz};
  const unsigned long long qi = S.qi;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    A.xyz[3 * qi + a] = fmaf(A.h, (float)S.P.base[a] + S.P.off[a], org[a]);
    if (A.tangent) A.tangent[3 * qi + a] = S.t[a];
  }
  if (A.rho) A.rho[qi] = S.rho;
  if (A.detj) A.detj[qi] = dj;
  if (A.iters) A.iters[qi] = S.it;
  A.flags[qi] = S.fl;
}

// A search put off (88 bytes): inside a line search, or (alpha -1) before the next.
struct Waiting {
  int base[3];
  float off0[3], off[3], t[3], grad[3];
  float rho, gg, gn, alpha;
  int it;
  unsigned long long qi;
};

// Searches differ by a factor of 180 in length (76 evaluations on average, up to
// 3300 for 179e3 face centres of a 256^3 field: 200 steps of many halvings), and one
// search is a chain of dependent evaluations.
//
// refine_kernel: persistent warps, one search a lane.  A turn is a line search; with
// PUT_OFF from step `whole` of a search on it is one evaluation, since a warp waits
// for the lane that halves longest (179e3 centres 830 us, whole line searches
// throughout 1000).  The first steps stay whole: lists of short searches keep their
// lanes in step, so that they end and refill together (300e3 converged points of
// 512^3 114 us, with single evaluations 136).  16, 8 or 4 steps, the fewer the fuller
// the lanes (60e3 centres of 256^3 528 us with 8, 535 with 16; 104e3 of 214^3 618 with 4,
// 660 with 8).  A lane whose search ends waits until
// kRefill lanes of its warp have (or none is searching); then those lanes write their
// results and take the next samples from the counter together (one atomic per warp
// and refill), so the long set-up and result code runs with many lanes at once.
// PUT_OFF: a warp that has no samples to come and whose searches have all taken
// `patience` evaluations leaves them to the list, which has room for every lane.
//
// refine_long_kernel: the searches of the list, kGroup lanes each.  The lanes take
// kGroup successive halvings of a line search at once, and the first that ends it as
// ref_search would (taken, or a step below tol) counts: the same result with a chain
// about as long as the number of steps, for up to kGroup times the work a step.
//
// Rules (refine_launch).  PUT_OFF for up to four samples a lane: above, the long
// searches run beside the others' (1.39e6 centres 3150 us without, 3230 with a list)
// and all forms of short ones lose (5 steps 388 against 706).  Not below kManySteps
// steps, where no chain is long enough for the second kernel (20 steps of 10e3 centres
// 80 us without, 93 with).  patience grows with the samples in flight: with few of
// them the longest chain counts, with all lanes in use the groups' work does.
//
// Each sample is computed exactly as alone.  Face centres of 256^3, lists of 1000 /
// 10000 / 50000 / 179473: 210 / 402 / 478 / 830 us; with whole line searches and no list
// 358 / 950 / 982 / 1230.  The same points refined again (few steps), 100 / 1000 /
// 100000 of them: 30 / 51 / 268 us against 31 / 49 / 811; 10000: 67 against 58, the one
// kind of list that stays slower, as its longest chain is just above the patience.
constexpr int kRefill = 12;
constexpr int kPatience = 32;
constexpr int kManySteps = 32;
constexpr int kPerTurn = 1024;  // samples in flight for one evaluation of patience more
constexpr int kGroup = 16;

// Counters, ahead of the list in memory.  plain_next (without PUT_OFF) is zeroed by
// the call; the others are zero between calls: the last block of each kernel of a
// call leaves those that it used so, which saves a launch.
struct RefCounters {
  unsigned long long plain_next;
  unsigned long long next_sample;
  unsigned long long count;  // entries of the list
  unsigned long long taken;
  unsigned long long finished;  // blocks of the running kernel
};
constexpr size_t kRefHead = 128;
static_assert(sizeof(RefCounters) <= kRefHead, "counters");

__device__ __forceinline__ void put_off(const RState& S, Waiting& W) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    W.base[a] = S.P0.base[a];
    W.off0[a] = S.P0.off[a];
    W.off[a] = S.P.off[a];
    W.t[a] = S.t[a];
    W.grad[a] = S.grad[a];
  }
  W.rho = S.rho;
  W.gg = S.gg;
  W.gn = S.gn;
  W.alpha = S.alpha;
  W.it = S.it;
  W.qi = S.qi;
}

__device__ __forceinline__ void take_up(const Waiting& W, RState& S) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    S.P0.base[a] = S.P.base[a] = W.base[a];
    S.P0.off[a] = W.off0[a];
    S.P.off[a] = W.off[a];
    S.t[a] = W.t[a];
    S.grad[a] = W.grad[a];
  }
  S.rho = W.rho;
  S.gg = W.gg;
  S.gn = W.gn;
  S.alpha = W.alpha;
  S.it = W.it;
  S.qi = W.qi;
  S.fl = QTV_REFINE_MAX_ITER;
  S.cache.c[0] = -1;  // no cell loaded
}

// the last block of a kernel to get here (called by one thread, after the others of
// its block are done)
__device__ __forceinline__ bool last_block(RefCounters* counter) {
  __threadfence();
  return atomicAdd(&counter->finished, 1ull) == gridDim.x - 1ull;
}

template <bool PUT_OFF>
__global__ void __launch_bounds__(REF_THREADS, REF_CTAS) refine_kernel(
    RefArgs A, RefCounters* counter, Waiting* list, int patience, int whole) {
  if (PUT_OFF) pdl_trigger();
  unsigned long long nn = A.n;
  if (A.n_dev) {
    const unsigned long long d = *A.n_dev;
    if (d < nn) nn = d;
  }
  unsigned long long* const next = PUT_OFF ? &counter->next_sample : &counter->plain_next;
  Field F;
  F.psi = A.psi;
  F.n[0] = A.nx;
  F.n[1] = A.ny;
  F.n[2] = A.nz;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  RState S;
  int evals = 0;
  bool begin = false;  // the next line search is to begin
  // no sample left to take (same in all lanes): with a lane for each, from the first refill on
  bool last = nn <= (unsigned long long)gridDim.x * REF_THREADS;
  // active: searching; done: search ended, result not yet written;
  // drained: no sample left for this lane
  bool active = false, done = false, drained = false;
  while (true) {
    const unsigned idle = __ballot_sync(0xffffffffu, !active && !drained);
    const unsigned busy = __ballot_sync(0xffffffffu, active);
    if (idle && (__popc(idle) >= kRefill || busy == 0u)) {
      if (done) {
        ref_finish(A, F, S);
        done = false;
      }
      const int leader = __ffs(idle) - 1;
      unsigned long long base = 0;
      if (lane == leader) base = atomicAdd(next, (unsigned long long)__popc(idle));
      base = __shfl_sync(0xffffffffu, base, leader);
      if (!active && !drained) {
        const unsigned long long qi = base + (unsigned long long)__popc(idle & lt);
        if (qi < nn) {
          evals = 0;
          if (ref_init(A, F, qi, S)) active = begin = true;
          else ref_finish(A, F, S);
        } else {
          drained = true;
        }
      }
      last = last || __any_sync(0xffffffffu, drained);
    }
    if (!__any_sync(0xffffffffu, active || done || !drained)) break;
    if (active) {
      int st = kGoesOn;
      if (!PUT_OFF || begin) st = ref_begin(A, S) ? kEnded : kGoesOn;
      if (st == kGoesOn) st = ref_search(A, F, S, PUT_OFF ? whole : INT_MAX, evals);
      begin = st == kTaken;
      if (st == kEnded) {
        active = false;
        done = true;
      }
    }
    if (PUT_OFF && last && !__any_sync(0xffffffffu, active && evals < patience)) break;
  }
  if (PUT_OFF) {  // (out of the loop: inside it this code cost the loop a third of its speed)
    if (done) ref_finish(A, F, S);
    if (active) {
      if (begin) S.alpha = -1.f;
      put_off(S, list[atomicAdd(&counter->count, 1ull)]);
    }
    __syncthreads();
    if (threadIdx.x == 0 && last_block(counter)) counter->next_sample = counter->finished = 0ull;
  }
}

__global__ void __launch_bounds__(REF_THREADS, REF_CTAS) refine_long_kernel(
    RefArgs A, RefCounters* counter, const Waiting* waiting) {
  constexpr unsigned full = 0xffffffffu;
  pdl_wait();
  const unsigned long long nw = *(volatile unsigned long long*)&counter->count;
  if (nw == 0) return;
  Field F;
  F.psi = A.psi;
  F.n[0] = A.nx;
  F.n[1] = A.ny;
  F.n[2] = A.nz;
  const int lane = threadIdx.x & 31, j = lane % kGroup, lead = lane - j;
  const unsigned group = ((1u << kGroup) - 1u) << lead;
  RState S;  // the same in all lanes of a group, but for the cache
  S.cache.c[0] = -1;
  S.alpha = S.gg = S.gn = S.rho = 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    S.P.base[a] = S.P0.base[a] = 0;
    S.P.off[a] = S.P0.off[a] = S.grad[a] = 0.f;
  }
  bool active = false, drained = false;
  while (true) {
    if (__any_sync(full, !active && !drained)) {
      unsigned long long w = 0;
      if (!active && !drained && j == 0) w = atomicAdd(&counter->taken, 1ull);
      w = __shfl_sync(full, w, lead);
      if (!active && !drained) {
        if (w < nw) {
          take_up(waiting[w], S);
          active = !(S.alpha == -1.f && ref_begin(A, S));
          if (!active && j == 0) ref_finish(A, F, S);
        } else {
          drained = true;
        }
      }
    }
    if (!__any_sync(full, active || !drained)) break;
    float alpha = S.alpha;
    for (int i = 0; i < j; ++i) alpha *= 0.5f;
    const bool below = !(alpha * S.gn >= A.tol);
    Pos Pn = {};
    float rn = 0.f, gnext[3] = {0.f, 0.f, 0.f};
    bool taken = false;
    if (active && !below && candidate(F, S.P.base, S.P.off, S.P0.off, S.grad, alpha, Pn)) {
      rn = rho_at(F, Pn, gnext, S.cache);
      taken = descends(rn, alpha, S.gg, S.rho);
    }
    const unsigned ends = __ballot_sync(full, below || taken) & group;
    const unsigned takes = __ballot_sync(full, taken);
    const int first = ends ? __ffs(ends) - 1 : lead + kGroup - 1;
    rn = __shfl_sync(full, rn, first);
    alpha = __shfl_sync(full, alpha, first);
    float off[3], g[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      off[a] = __shfl_sync(full, Pn.off[a], first);
      g[a] = __shfl_sync(full, gnext[a], first);
    }
    if (!active) continue;
    bool ended = false;
    if (!ends) {
      S.alpha = alpha * 0.5f;
    } else if (!((takes >> first) & 1u)) {
      S.fl = QTV_REFINE_CONVERGED;
      ended = true;
    } else {
      ++S.it;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        S.P.off[a] = off[a];
        S.grad[a] = g[a];
      }
      S.rho = rn;
      ended = ref_begin(A, S);
    }
    if (ended) {
      if (j == 0) ref_finish(A, F, S);
      active = false;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && last_block(counter)) counter->count = counter->taken = counter->finished = 0ull;
}

}  // namespace

int refine_launch(qtv_handle h, const qtv_grid& g, const float2* psi, const float* xyz0,
                  const uint64_t* face_ids, uint64_t n, const uint64_t* n_dev, int max_iter,
                  float tol, float* xyz, float* rho, float* tangent, float* detj, int32_t* iters,
                  uint8_t* flags, cudaStream_t st) {
  if (n == 0) return QTV_OK;
  RefArgs a;
  a.psi = psi;
  a.nx = g.nx;
  a.ny = g.ny;
  a.nz = g.nz;
  a.h = g.h;
  a.ox = g.origin[0];
  a.oy = g.origin[1];
  a.oz = g.origin[2];
  a.xyz0 = xyz0;
  a.face_ids = face_ids;
  a.n = n;
  a.n_dev = n_dev;
  a.max_iter = max_iter;
  a.tol = tol;
  a.xyz = xyz;
  a.rho = rho;
  a.tangent = tangent;
  a.detj = detj;
  a.iters = iters;
  a.flags = flags;
  // persistent: as many blocks as fit at once, fewer for short lists
  static int per_sm[2] = {0, 0};
  for (int i = 0; i < 2; ++i)
    if (per_sm[i] == 0) {
      int b = 0;
      const cudaError_t e =
          i ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, refine_kernel<true>, REF_THREADS, 0)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, refine_kernel<false>, REF_THREADS, 0);
      per_sm[i] = e == cudaSuccess && b > 0 ? b : 1;
    }
  const unsigned long long cap = (unsigned long long)h->num_sms * per_sm[1] * REF_THREADS;
  const bool longs = max_iter >= kManySteps && n <= 4 * cap;
  const long long maxb = (long long)h->num_sms * per_sm[longs ? 1 : 0];
  long long blocks = ((long long)n + REF_THREADS - 1) / REF_THREADS;
  if (blocks > maxb) blocks = maxb;
  // counters and list of one size for every call, so that a captured call keeps its
  // pointers
  if (!h->refine_counter) {
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&h->refine_counter),
                               kRefHead + cap * sizeof(Waiting));
    if (e != cudaSuccess) {
      h->refine_counter = nullptr;
      return check_cuda(e, "cudaMalloc(refine counter)");
    }
    e = cudaMemset(h->refine_counter, 0, kRefHead);
    if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
    if (e != cudaSuccess) {
      cudaFree(h->refine_counter);
      h->refine_counter = nullptr;
      return check_cuda(e, "cudaMemset(refine counter)");
    }
  }
  RefCounters* const counter = reinterpret_cast<RefCounters*>(h->refine_counter);
  Waiting* const list =
      reinterpret_cast<Waiting*>(reinterpret_cast<char*>(h->refine_counter) + kRefHead);
  TraceScope ts(h, K_REFINE, st);
  cudaError_t e = cudaSuccess;
  if (!longs) {
    e = cudaMemsetAsync(&counter->plain_next, 0, sizeof(counter->plain_next), st);
    if (e != cudaSuccess) return check_cuda(e, "cudaMemsetAsync(refine counter)");
    refine_kernel<false><<<(int)blocks, REF_THREADS, 0, st>>>(a, counter, list, 0, 0);
    return check_cuda(cudaGetLastError(), "refine_kernel launch");
  }
  const int patience = kPatience + (int)((n < cap ? n : cap) / kPerTurn);
  // the fuller the lanes, the more a warp's waiting costs
  const int whole = n <= cap / 4 ? 16 : (n <= cap ? 8 : 4);
  refine_kernel<true><<<(int)blocks, REF_THREADS, 0, st>>>(a, counter, list, patience, whole);
  e = cudaGetLastError();
  if (e != cudaSuccess) return check_cuda(e, "refine_kernel launch");
  long long lb = ((long long)(n < cap ? n : cap) * kGroup + REF_THREADS - 1) / REF_THREADS;
  if (lb > maxb) lb = maxb;
  // (its blocks wait beside a launch that leaves room for them: 3 us; beside a full
  // one it is no gain)
  if (2 * blocks <= maxb) {
    e = launch_dependent(refine_long_kernel, dim3((unsigned)lb), dim3(REF_THREADS), 0, st, a, counter,
                         (const Waiting*)list);
  } else {
    refine_long_kernel<<<(int)lb, REF_THREADS, 0, st>>>(a, counter, list);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) cudaMemsetAsync(counter, 0, kRefHead, st);  // the list was not taken up
  return check_cuda(e, "refine_long_kernel launch");
}

}  // namespace qtv
