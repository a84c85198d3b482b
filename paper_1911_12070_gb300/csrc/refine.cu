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

// two FP32 values in one register pair, IEEE roundings per value
using F2 = unsigned long long;
__device__ __forceinline__ F2 pair(float2 v) {
  return (F2)__float_as_uint(v.x) | ((F2)__float_as_uint(v.y) << 32);
}
__device__ __forceinline__ F2 both(float v) { return pair(make_float2(v, v)); }
__device__ __forceinline__ float2 unpair(F2 v) {
  return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ F2 neg2(F2 a) { return a ^ 0x8000000080000000ull; }

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
  // Re and Im side by side (packed FP32, the same roundings per component); the
  // weights are pairs of equal halves
  F2 w[2][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    w[0][a] = both(1.f - f[a]);
    w[1][a] = both(f[a]);
  }
  F2 vv = both(0.f), dv[3] = {both(0.f), both(0.f), both(0.f)};
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int b0 = q & 1, b1 = (q >> 1) & 1, b2 = q >> 2;
    const F2 u = pair(C.v[q]);
    vv = fma2(mul2(mul2(w[b0][0], w[b1][1]), w[b2][2]), u, vv);
    // derivatives: the weight of the axis is -1 or 1
    dv[0] = b0 ? fma2(mul2(w[b1][1], w[b2][2]), u, dv[0]) : fma2(neg2(mul2(w[b1][1], w[b2][2])), u, dv[0]);
    dv[1] = b1 ? fma2(mul2(w[b0][0], w[b2][2]), u, dv[1]) : fma2(neg2(mul2(w[b0][0], w[b2][2])), u, dv[1]);
    dv[2] = b2 ? fma2(mul2(w[b0][0], w[b1][1]), u, dv[2]) : fma2(neg2(mul2(w[b0][0], w[b1][1])), u, dv[2]);
  }
  const float2 v = unpair(vv);
  const float2 d[3] = {unpair(dv[0]), unpair(dv[1]), unpair(dv[2])};
#pragma unroll
  for (int a = 0; a < 3; ++a)
    g[a] = __fmul_rn(2.f, fmaf(v.x, d[a].x, __fmul_rn(v.y, d[a].y)));
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

// The next candidate of the line search that can be taken: one evaluation.  True
// when the sample is done.  (With the whole search inside a step a lane that
// halved twenty times held its warp.)
__device__ __forceinline__ bool ref_try(const RefArgs& A, const Field& F, RState& S) {
  Pos Pn;
  while (true) {
    if (!(S.alpha * S.gn >= A.tol)) {
      S.fl = QTV_REFINE_CONVERGED;
      return true;
    }
    if (candidate(F, S.P.base, S.P.off, S.P0.off, S.grad, S.alpha, Pn)) break;
    S.alpha *= 0.5f;
  }
  float gnext[3];
  const float rn = rho_at(F, Pn, gnext, S.cache);
  if (!descends(rn, S.alpha, S.gg, S.rho)) {
    S.alpha *= 0.5f;
    return false;
  }
  ++S.it;
  S.P = Pn;
  S.rho = rn;
#pragma unroll
  for (int a = 0; a < 3; ++a) S.grad[a] = gnext[a];
  return ref_begin(A, S);
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

// A search put off: what ref_try needs (88 bytes).
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
// refine_kernel: persistent warps; each lane keeps one search and evaluates one
// candidate of it per turn (with a whole line search inside a turn 9 of 32 threads
// were active, now 18: 609e3 samples in 908 us instead of 1932, without the searches
// put off).  A lane whose search ends waits until kRefill lanes of its warp have (or
// none is searching); then those lanes write their results and take the next samples
// from the counter together (one atomic per warp and refill), so the long set-up and
// result code runs with many lanes at once.  Once there are no more, a search of
// more than `patience` evaluations is put off into list 0, which has room for every
// lane in flight (with less, the searches left over made the launch as long as the
// longest chain: 4.3 ms instead of 3.2 for 1.39e6 samples).
//
// refine_long_kernel: the searches of a list, kGroup lanes each.  The lanes take
// kGroup successive halvings of a line search at once, and the first that ends it as
// ref_try would (taken, or a step below tol) counts: the same result with a chain
// about as long as the number of steps, for eight times the work a step.
//
// Rules (refine_launch).  Up to four samples a lane, list 0 goes to the groups
// directly and the patience grows with the samples in flight: with few of them the
// longest chain counts (33 evaluations 235 us for 1000 samples, 100 258), with all
// lanes in use the groups' work does (179e3 samples: 128 evaluations 824 us, 64 941).
// Above, a second launch first takes list 0 by full warps and puts off after
// another kPatience2 evaluations into list 1 (609e3 samples 1865 us, without it
// 1988 to 2019; 179e3 samples 1041 with it).
//
// Each sample is computed exactly as alone.  Face centres of 256^3, lists of 1000 /
// 10000 / 50000 / 179473: 239 / 284 / 371 / 826 us; with one lane and a line search a turn 348 /
// 761 / 885 / 1180 us; 512^3 (1.39e6) 3217 -> 3132, means of thinned lines there
// (235e3) 1627 -> 1093.  Slower: 1e5 points in random order that have converged
// already, whose searches are all short, 120 -> 166 at 256^3.
constexpr int kRefill = 12;
constexpr int kPatience = 32, kPatience2 = 384;
constexpr int kPerTurn = 1024;  // samples in flight for one evaluation of patience more
constexpr int kGroup = 16;

// counters of a call, ahead of the two lists in memory
struct RefCounters {
  unsigned long long next_sample;
  unsigned long long count[2];  // entries of the lists
  unsigned long long taken[2];
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

// LIST: the searches of list 0 instead of the samples
template <bool LIST>
__global__ void __launch_bounds__(REF_THREADS, REF_CTAS) refine_kernel(
    RefArgs A, RefCounters* counter, Waiting* lists, unsigned long long cap,
    unsigned long long groups, int patience) {
  unsigned long long nn = A.n;
  if (LIST) {
    nn = min(counter->count[0], cap);
    if (nn <= groups) return;
  } else if (A.n_dev) {
    const unsigned long long d = *A.n_dev;
    if (d < nn) nn = d;
  }
  unsigned long long* const next = LIST ? &counter->taken[0] : &counter->next_sample;
  Field F;
  F.psi = A.psi;
  F.n[0] = A.nx;
  F.n[1] = A.ny;
  F.n[2] = A.nz;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  RState S;
  int turns = 0;
  bool last = false;  // no sample left to take (same in all lanes)
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
          turns = 0;
          if (LIST) {
            take_up(lists[qi], S);
            active = true;
          } else if (ref_init(A, F, qi, S)) {
            active = !ref_begin(A, S);
            done = !active;
          } else {
            ref_finish(A, F, S);
          }
        } else {
          drained = true;
        }
      }
      last = __any_sync(0xffffffffu, drained);
    }
    if (!__any_sync(0xffffffffu, active || done || !drained)) break;
    if (active) {
      if (ref_try(A, F, S)) {
        active = false;
        done = true;
      } else if (++turns >= patience && last) {
        turns = INT_MIN;  // once, should the list be full
        const unsigned long long at = atomicAdd(&counter->count[LIST ? 1 : 0], 1ull);
        if (at < cap) {
          put_off(S, lists[(LIST ? cap : 0) + at]);
          active = false;
        }
      }
    }
  }
}

__global__ void __launch_bounds__(REF_THREADS, REF_CTAS) refine_long_kernel(
    RefArgs A, RefCounters* counter, const Waiting* lists, unsigned long long cap,
    unsigned long long groups) {
  constexpr unsigned full = 0xffffffffu;
  const int which = min(counter->count[0], cap) > groups ? 1 : 0;
  const Waiting* const waiting = lists + which * cap;
  const unsigned long long nw = min(counter->count[which], cap);
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
      if (!active && !drained && j == 0) w = atomicAdd(&counter->taken[which], 1ull);
      w = __shfl_sync(full, w, lead);
      if (!active && !drained) {
        if (w < nw) {
          take_up(waiting[w], S);
          active = true;
        } else {
          drained = true;
        }
      }
    }
    if (!__any_sync(full, active)) break;
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
  static int per_sm = 0;
  if (per_sm == 0) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, refine_kernel<false>, REF_THREADS, 0) !=
            cudaSuccess ||
        b < 1)
      b = 1;
    per_sm = b;
  }
  long long blocks = ((long long)n + REF_THREADS - 1) / REF_THREADS;
  const long long maxb = (long long)h->num_sms * per_sm;
  if (blocks > maxb) blocks = maxb;
  const unsigned long long cap = (unsigned long long)maxb * REF_THREADS;
  const bool twice = n > 4 * cap;
  // lists longer than this are taken by the second launch
  const unsigned long long groups = twice ? cap / kGroup : cap;
  const int patience = kPatience + (twice ? 0 : (int)((n < cap ? n : cap) / kPerTurn));
  // counters and lists of one size for every call, so that a captured call keeps its
  // pointers
  if (!h->refine_counter) {
    const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&h->refine_counter),
                                     kRefHead + 2 * cap * sizeof(Waiting));
    if (e != cudaSuccess) {
      h->refine_counter = nullptr;
      return check_cuda(e, "cudaMalloc(refine counter)");
    }
  }
  RefCounters* const counter = reinterpret_cast<RefCounters*>(h->refine_counter);
  Waiting* const lists =
      reinterpret_cast<Waiting*>(reinterpret_cast<char*>(h->refine_counter) + kRefHead);
  TraceScope ts(h, K_REFINE, st);
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(RefCounters), st);
  if (e != cudaSuccess) return check_cuda(e, "cudaMemsetAsync(refine counter)");
  refine_kernel<false><<<(int)blocks, REF_THREADS, 0, st>>>(a, counter, lists, cap, groups, patience);
  if (twice)
    refine_kernel<true><<<(int)blocks, REF_THREADS, 0, st>>>(a, counter, lists, cap, groups, kPatience2);
  blocks = ((long long)(n < cap ? n : cap) * kGroup + REF_THREADS - 1) / REF_THREADS;
  if (blocks > maxb) blocks = maxb;
  refine_long_kernel<<<(int)blocks, REF_THREADS, 0, st>>>(a, counter, lists, cap, groups);
  e = cudaGetLastError();
  return check_cuda(e, "refine_kernel launch");
}

}  // namespace qtv
