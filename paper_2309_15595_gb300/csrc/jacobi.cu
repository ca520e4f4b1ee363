// Two-sided cyclic Jacobi eigensolver for the small Hermitian Rayleigh-Ritz
// problem (the paper's HEEVD step, Alg. 2) and the Lanczos tridiagonals.
//
// Rotation for a pair (p, q) with a = G_pp, d = G_qq (real), b = G_pq = |b| phi:
//   tau = (d - a) / (2|b|), t = sign(tau) / (|tau| + sqrt(1 + tau^2)),
//   c = 1/sqrt(1 + t^2), s = t c,
//   J = [[c, s phi], [-s conj(phi), c]]  (identity elsewhere),
// so that J^H G J has a zero (p, q) entry, new G_pp = a - t|b|, G_qq = d + t|b|.
// Pairs follow the round-robin (tournament) order: index 0 stays, the others
// rotate, so each round holds n/2 disjoint pairs that are rotated in parallel
// and n - 1 rounds visit every pair once (one sweep).
#include <algorithm>
#include <cstdio>
#include <vector>

#include "common.cuh"

namespace chase {
namespace {

#define RC_(call)                   \
  do {                              \
    const int _rc = (call);         \
    if (_rc != CHASE_OK) return _rc; \
  } while (0)
#define RC_NEG(call)                  \
  do {                                \
    const int _rc = (call);           \
    if (_rc != CHASE_OK) return -_rc; \
  } while (0)

constexpr int kMaxSweeps = 40;
constexpr int kCoopMaxGrid = 2048;  // reduction scratch holds 2 * kCoopMaxGrid partials

__device__ __forceinline__ void rr_pair(int m, int round, int k, int& p, int& q) {
  auto pos = [&](int i) { return i == 0 ? 0 : 1 + (i - 1 + round) % (m - 1); };
  p = pos(k);
  q = pos(m - 1 - k);
  if (p > q) { const int tmp = p; p = q; q = tmp; }
}

__device__ bool converged_rule(double off, double fro, double off_prev) {
  if (off == 0.0 || off <= 1e-15 * fro) return true;
  return off <= 1e-12 * fro && off > 0.25 * off_prev;
}

// ------------------------------------------------- single-CTA batched version
constexpr int SJ_MAX = 64, SJ_T = 256;
// Eigenproblems of order up to kSmallFp64 run in FP64 in one CTA; its time grows
// like n^3 (one SM has two DFMA a clock), so larger ones start in FP32 in one CTA and
// refine in FP64 on many SMs. A Rayleigh-Ritz call with N = 300, FP64 against FP32 and
// refinement, in us: n = 16 773 / 784, 20 914 / 894, 24 1184 / 913, 32 1600 / 1043, 64
// 8270 / 1430. They cross at 16 to 20; 24 is where the line was drawn for a slower
// FP64 kernel.
constexpr int64_t kSmallFp64 = 24;
// Largest order whose FP64 refinement multiplies on the CUDA cores: a product of
// order 64 takes 20 us there and, with the digits of both operands, 60 us on the
// tensor cores. A Rayleigh-Ritz call with N = 1000, CUDA cores against tensor cores, in
// ms: n = 65 2.21 / 2.28, 96 3.14 / 2.84, 128 2.92 / 2.90, 129 4.46 / 4.08, 256 7.63 /
// 6.26 (the orders differ in their sweeps).
constexpr int64_t kCoreRefine = 128;

// A whole FP64 Jacobi in one CTA, n <= 64 (one SM: two DFMA a clock, so FP64
// operations are what a round costs). The matrix is scaled by a power of two to
// entries of at most 1 and padded to an even order. Per round: the rotations, with
// the angle from FP32 and the cosine (and phase) made exact to FP64, so that the
// rotated entry is small and not zero (a sweep still gains seven digits at the
// least); then each 2 x 2 block where two pairs meet is rotated from both sides at
// once and mirrored, and Z by columns. REAL: a real symmetric matrix (the Lanczos
// tridiagonals), a quarter of the operations. n = 25, four matrices: 1.1 ms with FP64
// angles, separate passes over columns and rows and complex arithmetic.
template <bool REAL> struct Sj;
template <> struct Sj<true> {
  using C = double;
  static __device__ __forceinline__ C mk(double x, double) { return x; }
  static __device__ __forceinline__ double re(C a) { return a; }
  static __device__ __forceinline__ double abs2(C a) { return a * a; }
  static __device__ __forceinline__ C conj(C a) { return a; }
  // c x - w y  and  c x + w y
  static __device__ __forceinline__ C sub(double c, C x, C w, C y) { return fma(c, x, -(w * y)); }
  static __device__ __forceinline__ C add(double c, C x, C w, C y) { return fma(c, x, w * y); }
  static __device__ __forceinline__ double2 z(C a) { return make_double2(a, 0.0); }
};
template <> struct Sj<false> {
  using C = double2;
  static __device__ __forceinline__ C mk(double x, double y) { return make_double2(x, y); }
  static __device__ __forceinline__ double re(C a) { return a.x; }
  static __device__ __forceinline__ double abs2(C a) { return cabs2(a); }
  static __device__ __forceinline__ C conj(C a) { return conjz(a); }
  static __device__ __forceinline__ C sub(double c, C x, C w, C y) {
    return make_double2(fma(c, x.x, fma(-w.x, y.x, w.y * y.y)),
                        fma(c, x.y, -fma(w.x, y.y, w.y * y.x)));
  }
  static __device__ __forceinline__ C add(double c, C x, C w, C y) {
    return make_double2(fma(c, x.x, fma(w.x, y.x, -(w.y * y.y))),
                        fma(c, x.y, fma(w.x, y.y, w.y * y.x)));
  }
  static __device__ __forceinline__ double2 z(C a) { return a; }
};
// 1 / sqrt(w) for w in FP32's normal range: an FP32 seed and two Newton steps
__device__ __forceinline__ double rsqrt_seeded(double w, float wf) {
  double y = (double)rsqrtf(wf);
  const double h = 0.5 * w;
#pragma unroll
  for (int i = 0; i < 2; ++i) y = fma(y, fma(-h * y, y, 0.5), y);
  return y;
}

constexpr int SJ_LD = SJ_MAX + 1;
constexpr double kSjSkip = 1e-18;  // entries this far below the largest one stay

template <bool REAL>
__global__ void __launch_bounds__(SJ_T)
    jacobi_small_kernel(int n, const double2* __restrict__ Gin, double* __restrict__ w,
                        double2* __restrict__ Zout, int* status, int max_sweeps) {
  using O = Sj<REAL>;
  using C = typename O::C;
  struct SjRot {
    double c;
    C u;  // s phi
    int p, q, on;
  };
  extern __shared__ double2 sm[];
  C* G = reinterpret_cast<C*>(sm);  // m x m, ld SJ_LD
  C* Z = G + SJ_MAX * SJ_LD;
  __shared__ SjRot rots[SJ_MAX / 2];
  __shared__ double red[SJ_T], red2[SJ_T];
  __shared__ int rank_s[SJ_MAX], s_exp;
  const int t = threadIdx.x;
  const double2* Gb = Gin + (size_t)blockIdx.x * n * n;
  const int m = n + (n & 1), npairs = m / 2, nblocks = npairs * (npairs - 1) / 2;
  if (t == 0) s_exp = 0;
  __syncthreads();
  int ex = 0;
  for (int e = t; e < n * n; e += SJ_T) {
    const double2 v = Gb[e];
    ex = max(ex, (__double2hiint(v.x) >> 20) & 0x7ff);
    if constexpr (!REAL) ex = max(ex, (__double2hiint(v.y) >> 20) & 0x7ff);
  }
  atomicMax(&s_exp, ex);
  __syncthreads();
  // 2^sh G has entries below 1; nothing is scaled where that leaves FP64's range
  const int sh = s_exp > 0 && s_exp < 2040 ? 1022 - s_exp : 0;
  for (int e = t; e < m * m; e += SJ_T) {
    const int r = e % m, c = e / m;
    // Hermitian part of the input (inputs formed as X^H (G X) are Hermitian
    // only up to rounding)
    C g = O::mk(0.0, 0.0);
    if (r < n && c < n) {
      const double2 a = Gb[r + c * n], b = Gb[c + r * n];
      g = O::mk(ldexp(0.5 * a.x + 0.5 * b.x, sh), ldexp(0.5 * a.y - 0.5 * b.y, sh));
    }
    G[r + c * SJ_LD] = g;
    Z[r + c * SJ_LD] = O::mk(r == c ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  double off_prev = 1e300;
  bool conv = false;
  for (int sweep = 0; sweep <= max_sweeps; ++sweep) {
    double so = 0.0, sf = 0.0;
    for (int e = t; e < m * m; e += SJ_T) {
      const int r = e % m, c = e / m;
      const double v = O::abs2(G[r + c * SJ_LD]);
      sf += v;
      if (r != c) so += v;
    }
    red[t] = so;
    red2[t] = sf;
    __syncthreads();
    for (int s = SJ_T / 2; s >= 1; s >>= 1) {
      if (t < s) { red[t] += red[t + s]; red2[t] += red2[t + s]; }
      __syncthreads();
    }
    const double off = sqrt(red[0]), fro = sqrt(red2[0]);
    __syncthreads();
    if (converged_rule(off, fro, off_prev)) {
      conv = true;
      break;
    }
    off_prev = off;
    if (sweep == max_sweeps) break;
    for (int round = 0; round < m - 1; ++round) {
      if (t < npairs) {
        SjRot r;
        rr_pair(m, round, t, r.p, r.q);
        C* gp = G + r.p * SJ_LD;
        C* gq = G + r.q * SJ_LD;
        const double a = O::re(gp[r.p]), d = O::re(gq[r.q]), delta = d - a;
        const C b = gq[r.p];  // G(p, q)
        const double bb = O::abs2(b);
        r.c = 1.0;
        r.u = O::mk(0.0, 0.0);
        r.on = bb > kSjSkip * kSjSkip;
        if (r.on) {
          const float bf = (float)bb, rf = rsqrtf(bf);
          const float tau = 0.5f * (float)delta * rf;
          const float tf = copysignf(
              __fdividef(1.f, fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f))), tau);
          const double tt = (double)tf, ww = fma(tt, tt, 1.0);
          r.c = rsqrt_seeded(ww, (float)ww);
          const double sn = tt * r.c, ri = REAL ? 0.0 : rsqrt_seeded(bb, bf);
          const double ab = REAL ? fabs(O::re(b)) : bb * ri;
          const double s2 = sn * sn, cs = r.c * sn;
          const double v = fma(s2, delta, -2.0 * cs * ab);
          const double no = fma(fma(r.c, r.c, -s2), ab, -cs * delta);  // what is left of |b|
          if constexpr (REAL) {
            const double sg = O::re(b) < 0.0 ? -1.0 : 1.0;
            r.u = sg * sn;
            gq[r.p] = gp[r.q] = sg * no;
          } else {
            const double2 ph = cscale(ri, b);
            r.u = cscale(sn, ph);
            gq[r.p] = cscale(no, ph);
            gp[r.q] = conjz(gq[r.p]);
          }
          gp[r.p] = O::mk(a + v, 0.0);
          gq[r.q] = O::mk(d - v, 0.0);
        }
        rots[t] = r;
      }
      __syncthreads();
      for (int e = t; e < nblocks; e += SJ_T) {  // block (k, l), k < l: number l (l-1)/2 + k
        int l = (int)((1.f + sqrtf(8.f * (float)e + 1.f)) * 0.5f);
        while (l * (l - 1) / 2 > e) --l;
        while (l * (l + 1) / 2 <= e) ++l;
        const SjRot& jk = rots[e - l * (l - 1) / 2];
        const SjRot& jl = rots[l];
        if (!(jk.on | jl.on)) continue;
        const int pk = jk.p, qk = jk.q, pl = jl.p, ql = jl.q;
        const double ck = jk.c, cl = jl.c;
        const C uk = jk.u, ul = jl.u, uck = O::conj(uk), ucl = O::conj(ul);
        const C x0 = G[pk + pl * SJ_LD], x1 = G[pk + ql * SJ_LD];
        const C x2 = G[qk + pl * SJ_LD], x3 = G[qk + ql * SJ_LD];
        // columns of pair l, then rows of pair k
        const C y0 = O::sub(cl, x0, ucl, x1), y1 = O::add(cl, x1, ul, x0);
        const C y2 = O::sub(cl, x2, ucl, x3), y3 = O::add(cl, x3, ul, x2);
        const C z0 = O::sub(ck, y0, uk, y2), z2 = O::add(ck, y2, uck, y0);
        const C z1 = O::sub(ck, y1, uk, y3), z3 = O::add(ck, y3, uck, y1);
        G[pk + pl * SJ_LD] = z0;
        G[pk + ql * SJ_LD] = z1;
        G[qk + pl * SJ_LD] = z2;
        G[qk + ql * SJ_LD] = z3;
        G[pl + pk * SJ_LD] = O::conj(z0);
        G[ql + pk * SJ_LD] = O::conj(z1);
        G[pl + qk * SJ_LD] = O::conj(z2);
        G[ql + qk * SJ_LD] = O::conj(z3);
      }
      for (int e = t; e < npairs * n; e += SJ_T) {
        const SjRot& r = rots[e / n];
        if (!r.on) continue;
        C* zp = Z + r.p * SJ_LD + e % n;
        C* zq = Z + r.q * SJ_LD + e % n;
        const C x = *zp, y = *zq;
        *zp = O::sub(r.c, x, O::conj(r.u), y);
        *zq = O::add(r.c, y, r.u, x);
      }
      __syncthreads();
    }
  }
  if (t == 0 && !conv) *status = 1;
  // rank sort of the diagonal (ties by index)
  if (t < n) {
    const double v = O::re(G[t + t * SJ_LD]);
    int rk = 0;
    for (int j = 0; j < n; ++j) {
      const double u = O::re(G[j + j * SJ_LD]);
      rk += (u < v) || (u == v && j < t);
    }
    rank_s[t] = rk;
  }
  __syncthreads();
  double* wb = w + (size_t)blockIdx.x * n;
  double2* Zb = Zout + (size_t)blockIdx.x * n * n;
  if (t < n) wb[rank_s[t]] = ldexp(O::re(G[t + t * SJ_LD]), -sh);
  for (int e = t; e < n * n; e += SJ_T) {
    const int r = e % n, c = e / n;
    Zb[r + rank_s[c] * n] = O::z(Z[r + c * SJ_LD]);
  }
}

// ------------------------------------------------------ large-n version
// Templated on the real type T (float or double): the large-n solver first
// sweeps in FP32 (the FP64 pipe of this part is 1/58 of the FP32 one), then
// re-orthonormalises the FP32 eigenvectors in FP64, forms Z^H G Z in FP64
// (nearly diagonal) and finishes with a few FP64 sweeps.
constexpr int LJ_T = 256;

template <typename T> struct Cx;
// eps: threshold of the rotation skip, |b| <= eps sqrt(|a d|) (unit round-off)
template <> struct Cx<double> {
  using C = double2;
  static __device__ __forceinline__ C mk(double x, double y) { return make_double2(x, y); }
  static constexpr double tiny = 1e-300, huge = 1e150, eps = 1.1102230246251565e-16;
};
template <> struct Cx<float> {
  using C = float2;
  static __device__ __forceinline__ C mk(float x, float y) { return make_float2(x, y); }
  static constexpr float tiny = 1e-30f, huge = 1e15f, eps = 5.9604645e-8f;
};

template <typename T>
struct RotT {
  T c, s, px, py, app, aqq;
};

template <typename T>
__device__ __forceinline__ RotT<T> make_rot_t(T a, T d, typename Cx<T>::C b) {
  RotT<T> r;
  const T ab = sqrt(b.x * b.x + b.y * b.y);
  // threshold Jacobi: an entry below eps sqrt(|a d|) changes neither the
  // eigenvalues nor the eigenvectors at working precision; skip it
  if (!(ab > Cx<T>::tiny) || ab <= Cx<T>::eps * sqrt(fabs(a) * fabs(d))) {
    r.c = T(1); r.s = T(0); r.px = T(1); r.py = T(0); r.app = a; r.aqq = d;
    return r;
  }
  r.px = b.x / ab;
  r.py = b.y / ab;
  const T tau = (d - a) / (T(2) * ab);
  T t;
  if (fabs(tau) > Cx<T>::huge) t = T(0.5) / tau;
  else t = (tau >= T(0) ? T(1) : T(-1)) / (fabs(tau) + sqrt(T(1) + tau * tau));
  r.c = T(1) / sqrt(T(1) + t * t);
  r.s = t * r.c;
  r.app = a - t * ab;
  r.aqq = d + t * ab;
  return r;
}

// (x_p, x_q) <- (x_p, x_q) J   with J = [[c, s phi], [-s conj(phi), c]]
template <typename T, typename C>
__device__ __forceinline__ void rot_cols_t(C& xp, C& xq, const RotT<T>& r) {
  const T sx = r.s * r.px, sy = r.s * r.py;  // s phi
  // xp' = c xp - conj(s phi) xq ; xq' = (s phi) xp + c xq
  const T npx = r.c * xp.x - (sx * xq.x + sy * xq.y);
  const T npy = r.c * xp.y - (sx * xq.y - sy * xq.x);
  const T nqx = (sx * xp.x - sy * xp.y) + r.c * xq.x;
  const T nqy = (sx * xp.y + sy * xp.x) + r.c * xq.y;
  xp.x = npx; xp.y = npy; xq.x = nqx; xq.y = nqy;
}
// (y_p; y_q) <- J^H (y_p; y_q)
template <typename T, typename C>
__device__ __forceinline__ void rot_rows_t(C& yp, C& yq, const RotT<T>& r) {
  const T sx = r.s * r.px, sy = r.s * r.py;
  // yp' = c yp - (s phi) yq ; yq' = conj(s phi) yp + c yq
  const T npx = r.c * yp.x - (sx * yq.x - sy * yq.y);
  const T npy = r.c * yp.y - (sx * yq.y + sy * yq.x);
  const T nqx = (sx * yp.x + sy * yp.y) + r.c * yq.x;
  const T nqy = (sx * yp.y - sy * yp.x) + r.c * yq.y;
  yp.x = npx; yp.y = npy; yq.x = nqx; yq.y = nqy;
}

template <typename T>
__device__ __forceinline__ RotT<T> load_rot_t(const T* __restrict__ params, int k) {
  const T* pp = params + 8 * k;
  RotT<T> r;
  r.c = pp[0]; r.s = pp[1]; r.px = pp[2]; r.py = pp[3]; r.app = pp[4]; r.aqq = pp[5];
  return r;
}

// *out = the largest exponent field of G's entries (0 before)
__global__ void max_exp_kernel(int64_t n, const double2* __restrict__ G, int64_t ldg,
                               int* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = blockIdx.y;
  int e = 0;
  if (i < n) {
    const double2 g = G[i + j * ldg];
    e = max((__double2hiint(g.x) >> 20) & 0x7ff, (__double2hiint(g.y) >> 20) & 0x7ff);
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0 && e > *(volatile int*)out) atomicMax(out, e);
}
// G32 = G times a power of two that brings its entries below 2 (the rotations square
// them, and 1.8e19 is where FP32 ends); not where *max_exp says that G is not finite.
__global__ void init32_kernel(int64_t n, const double2* G, int64_t ldg, const int* max_exp,
                              float2* G32, float2* Z32) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = blockIdx.y;
  if (i >= n) return;
  const double2 g = G[i + j * ldg];
  const int sh = *max_exp == 0x7ff ? 0 : 1023 - *max_exp;
  G32[i + j * n] = make_float2((float)ldexp(g.x, sh), (float)ldexp(g.y, sh));
  Z32[i + j * n] = make_float2(i == j ? 1.f : 0.f, 0.f);
}
__global__ void promote_kernel(int64_t n, const float2* Z32, double2* Z) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = blockIdx.y;
  if (i >= n) return;
  const float2 z = Z32[i + j * n];
  Z[i + j * n] = make_double2((double)z.x, (double)z.y);
}
__global__ void identity_kernel(int64_t n, double2* Z) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = blockIdx.y;
  if (i < n) Z[i + j * n] = make_double2(i == j ? 1.0 : 0.0, 0.0);
}

// Pair k of round `round`, G double-buffered: the owner of pair (p, q) writes
// the new columns p, q of J^H G J into Gnew, reading only the pre-round Gold,
// so owners never race. Its column rotation J_k mixes columns p and q row by
// row; then every pair's row rotation J_k'^H (computed once per round, in
// `params`) mixes rows (p', q') of these two columns. Z is updated in place:
// its columns p, q belong to this owner alone.
template <typename T>
__device__ void process_pair(int64_t n, int m, int round, int k,
                             const typename Cx<T>::C* __restrict__ Gold,
                             typename Cx<T>::C* __restrict__ Gnew, typename Cx<T>::C* __restrict__ Zw,
                             typename Cx<T>::C* colbuf, const T* __restrict__ params,
                             const T* sparams) {
  using C = typename Cx<T>::C;
  int p, q;
  rr_pair(m, round, k, p, q);
  // odd n: the pair holding the padding index n has one real column, p, which
  // still receives every other pair's row rotation
  const bool single = q >= n;
  if (single) q = p;
  C* gp = colbuf;
  C* gq = colbuf + n;
  RotT<T> r = load_rot_t(params, k);
  if (single) r.s = T(0);
  const C* Gp = Gold + (int64_t)p * n;
  const C* Gq = Gold + (int64_t)q * n;
  C* Zp = Zw + (int64_t)p * n;
  C* Zq = Zw + (int64_t)q * n;
  for (int64_t i = threadIdx.x; i < n; i += LJ_T) {
    C a = Gp[i], b = Gq[i];
    if (r.s != T(0)) rot_cols_t(a, b, r);
    gp[i] = a;
    gq[i] = b;
    if (r.s != T(0)) {
      C x = Zp[i], y = Zq[i];
      rot_cols_t(x, y, r);
      Zp[i] = x;
      Zq[i] = y;
    }
  }
  __syncthreads();
  for (int kk = threadIdx.x; kk < m / 2; kk += LJ_T) {
    int pr, qr;
    rr_pair(m, round, kk, pr, qr);
    if (qr >= n) continue;
    const RotT<T> rk = load_rot_t(sparams, kk);
    if (rk.s == T(0)) continue;
    rot_rows_t(gp[pr], gp[qr], rk);
    rot_rows_t(gq[pr], gq[qr], rk);
  }
  __syncthreads();
  if (threadIdx.x == 0 && r.s != T(0)) {  // exact 2 x 2 block of this pair
    gp[p] = Cx<T>::mk(r.app, T(0));
    gq[q] = Cx<T>::mk(r.aqq, T(0));
    gp[q] = Cx<T>::mk(T(0), T(0));
    gq[p] = Cx<T>::mk(T(0), T(0));
  }
  __syncthreads();
  C* Np_ = Gnew + (int64_t)p * n;
  C* Nq_ = Gnew + (int64_t)q * n;
  for (int64_t i = threadIdx.x; i < n; i += LJ_T) {
    Np_[i] = gp[i];
    if (!single) Nq_[i] = gq[i];
  }
  __syncthreads();  // colbuf is reused by this block's next pair
}

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid-wide barrier of a cooperative launch (all blocks are co-resident). The
// wait is bounded: after 2 s it records status[0] = 1 and returns false.
__device__ bool grid_sync(unsigned* bar, int* status) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok_s = 1;
    volatile unsigned* vgen = bar + 1;
    __threadfence();
    const unsigned gen = *vgen;
    if (atomicAdd(bar, 1u) == gridDim.x - 1) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      const unsigned long long t0 = gtimer();
      while (*vgen == gen) {
        if (*(volatile int*)status != 0) {  // another block gave up: leave at once
          ok_s = 0;
          break;
        }
        if (gtimer() - t0 > 2000000000ull) {
          atomicExch(status, 1);
          ok_s = 0;
          break;
        }
      }
    }
    __threadfence();
    if (*(volatile int*)status != 0) ok_s = 0;
  }
  __syncthreads();
  return ok_s != 0;
}

template <typename T>
struct CoopArgs {
  int64_t n;
  int m, max_sweeps;
  double tol_conv, tol_stag;  // converged: off <= tol_conv fro, or <= tol_stag fro and stalled
  typename Cx<T>::C* G0;
  typename Cx<T>::C* G1;
  typename Cx<T>::C* Z;
  T* params;        // 8 values per pair of the current round
  double* red;      // 2 * gridDim.x partial sums
  unsigned* bar;    // barrier counter and generation
  int* status;      // [0] error, [1] sweeps, [2] converged, [3] result in G1
};

// A whole cyclic Jacobi in one cooperative launch: per sweep a fixed-order
// off-norm test (identical in every block, so the decision is uniform), then
// the m - 1 rounds; per round the rotations are computed once (phase A) and
// applied by the pair owners (phase B), each phase closed by a grid barrier.
template <typename T>
__global__ void __launch_bounds__(LJ_T) jacobi_coop_kernel(CoopArgs<T> a) {
  using C = typename Cx<T>::C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* colbuf = reinterpret_cast<C*>(smem_raw);
  // this round's rotations, staged once per block (8 values per pair)
  T* sparams = reinterpret_cast<T*>(colbuf + 2 * a.n);
  __shared__ double so[LJ_T], sf[LJ_T];
  __shared__ int decide;
  const int64_t n = a.n;
  const int npairs = a.m / 2;
  C* Gcur = a.G0;
  C* Gnxt = a.G1;
  double off_prev = 1e300;
  int sweep = 0;
  bool conv = false, alive = true;
  for (; sweep <= a.max_sweeps && alive; ++sweep) {
    double o = 0.0, f = 0.0;
    const int64_t tot = n * n;
    for (int64_t e = (int64_t)blockIdx.x * LJ_T + threadIdx.x; e < tot; e += (int64_t)gridDim.x * LJ_T) {
      const C g = Gcur[e];
      const double v = (double)g.x * g.x + (double)g.y * g.y;
      f += v;
      if (e % n != e / n) o += v;
    }
    so[threadIdx.x] = o;
    sf[threadIdx.x] = f;
    __syncthreads();
    for (int w = LJ_T / 2; w >= 1; w >>= 1) {
      if (threadIdx.x < w) {
        so[threadIdx.x] += so[threadIdx.x + w];
        sf[threadIdx.x] += sf[threadIdx.x + w];
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      a.red[blockIdx.x] = so[0];
      a.red[gridDim.x + blockIdx.x] = sf[0];
    }
    if (!grid_sync(a.bar, a.status)) { alive = false; break; }
    if (threadIdx.x == 0) {
      double to = 0.0, tf = 0.0;
      for (unsigned b = 0; b < gridDim.x; ++b) {
        to += a.red[b];
        tf += a.red[gridDim.x + b];
      }
      const double off = sqrt(to), fro = sqrt(tf);
      int d = 0;
      if (off == 0.0 || off <= a.tol_conv * fro || (off <= a.tol_stag * fro && off > 0.25 * off_prev))
        d = 1;
      else if (sweep == a.max_sweeps)
        d = 2;
      off_prev = off;
      decide = d;
    }
    __syncthreads();
    // every block has read the partials before any block rewrites them
    if (!grid_sync(a.bar, a.status)) { alive = false; break; }
    if (decide == 1) { conv = true; break; }
    if (decide == 2) break;
    for (int round = 0; round < a.m - 1; ++round) {
      if constexpr (sizeof(T) == 4) {
        // FP32: every block computes all of this round's rotations itself (cheap
        // in FP32), which saves the grid barrier between computing and applying
        for (int k = threadIdx.x; k < npairs; k += LJ_T) {
          int p, q;
          rr_pair(a.m, round, k, p, q);
          const RotT<T> r = q < n ? make_rot_t<T>(Gcur[p + (int64_t)p * n].x,
                                                  Gcur[q + (int64_t)q * n].x,
                                                  Gcur[p + (int64_t)q * n])
                                  : make_rot_t<T>(T(0), T(0), Cx<T>::mk(T(0), T(0)));
          T* pp = sparams + 8 * k;
          pp[0] = r.c; pp[1] = r.s; pp[2] = r.px; pp[3] = r.py; pp[4] = r.app; pp[5] = r.aqq;
        }
        __syncthreads();
        for (int k = blockIdx.x; k < npairs; k += gridDim.x)
          process_pair<T>(n, a.m, round, k, Gcur, Gnxt, a.Z, colbuf, sparams, sparams);
      } else {
        // FP64 rotations are expensive on this part: computed once (phase A),
        // published through global memory, then applied (phase B)
        for (int k = blockIdx.x * LJ_T + threadIdx.x; k < npairs; k += gridDim.x * LJ_T) {
          int p, q;
          rr_pair(a.m, round, k, p, q);
          const RotT<T> r = q < n ? make_rot_t<T>(Gcur[p + (int64_t)p * n].x,
                                                  Gcur[q + (int64_t)q * n].x,
                                                  Gcur[p + (int64_t)q * n])
                                  : make_rot_t<T>(T(0), T(0), Cx<T>::mk(T(0), T(0)));
          T* pp = a.params + 8 * k;
          pp[0] = r.c; pp[1] = r.s; pp[2] = r.px; pp[3] = r.py; pp[4] = r.app; pp[5] = r.aqq;
        }
        if (!grid_sync(a.bar, a.status)) { alive = false; break; }
        for (int e = threadIdx.x; e < 8 * npairs; e += LJ_T) sparams[e] = a.params[e];
        __syncthreads();
        for (int k = blockIdx.x; k < npairs; k += gridDim.x)
          process_pair<T>(n, a.m, round, k, Gcur, Gnxt, a.Z, colbuf, a.params, sparams);
      }
      if (!grid_sync(a.bar, a.status)) { alive = false; break; }
      C* t = Gcur;
      Gcur = Gnxt;
      Gnxt = t;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.status[1] = sweep;
    a.status[2] = conv ? 1 : 0;
    a.status[3] = Gcur == a.G1 ? 1 : 0;
  }
}

// Runs one cooperative Jacobi on G0 (destroyed; the result may end in G1).
// Returns CHASE_OK and fills *sweeps, *conv, *in_g1; CHASE_ERR_CUDA on a
// launch failure or an expired barrier.
template <typename T>
int run_coop(cudaStream_t s, int64_t n, typename Cx<T>::C* G0, typename Cx<T>::C* G1,
             typename Cx<T>::C* Z, T* params, double* red, int max_sweeps, double tol_conv,
             double tol_stag, int* sweeps, bool* conv, bool* in_g1) {
  using C = typename Cx<T>::C;
  const int m = (int)(n + (n & 1));
  const int npairs = m / 2;
  const size_t smem = (size_t)2 * n * sizeof(C) + (size_t)8 * npairs * sizeof(T);
  // The opt-in limit covers dynamic + static shared memory (the kernel's static
  // reduction arrays add 4 KB, so sizes just under 48 KB need it too). It is a
  // process-wide property of the function that concurrent solves on other host
  // threads share, so it is set once per device to the largest size any
  // context can ask for (n <= 3500), never lowered.
  static std::once_flag attr_once[kMaxDevices];
  once_per_device(attr_once, []() {
    constexpr int64_t nmax = 3500;
    const size_t most = (size_t)2 * nmax * sizeof(C) + (size_t)8 * (nmax / 2) * sizeof(T);
    cudaFuncSetAttribute(jacobi_coop_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)most);
  });
  int dev = 0, nsm = 0, per_sm = 0, coop = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  const cudaError_t oe =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, jacobi_coop_kernel<T>, LJ_T, smem);
  if (!coop || oe != cudaSuccess || per_sm < 1) {
    fprintf(stderr,
            "[chase] Jacobi (%s) n=%lld: no cooperative residency (coop %d, occupancy %s, "
            "blocks/SM %d, dynamic smem %zu B)\n",
            sizeof(T) == 4 ? "FP32" : "FP64", (long long)n, coop, cudaGetErrorString(oe), per_sm,
            smem);
    return CHASE_CUDA_FAIL();
  }
  // one pair per block where the blocks fit, so pairs run concurrently
  const int grid = std::min(std::min(npairs, per_sm * nsm), kCoopMaxGrid);
  unsigned* bar = reinterpret_cast<unsigned*>(red + 2 * kCoopMaxGrid);
  int* st = reinterpret_cast<int*>(red + 2 * kCoopMaxGrid + 2);
  if (cudaMemsetAsync(red + 2 * kCoopMaxGrid, 0, 8 * sizeof(double), s) != cudaSuccess)
    return CHASE_CUDA_FAIL();
  CoopArgs<T> args;
  args.n = n;
  args.m = m;
  args.max_sweeps = max_sweeps;
  args.tol_conv = tol_conv;
  args.tol_stag = tol_stag;
  args.G0 = G0;
  args.G1 = G1;
  args.Z = Z;
  args.params = params;
  args.red = red;
  args.bar = bar;
  args.status = st;
  void* kargs[] = {&args};
  if (cudaLaunchCooperativeKernel((const void*)jacobi_coop_kernel<T>, dim3(grid), dim3(LJ_T), kargs,
                                  smem, s) != cudaSuccess)
    return CHASE_CUDA_FAIL();
  count_launch();
  int hst[4] = {0, 0, 0, 0};
  if (cudaMemcpyAsync(hst, st, sizeof(hst), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CHASE_CUDA_FAIL();
  if (hst[0] != 0) {
    fprintf(stderr, "[chase] Jacobi: grid barrier wait expired\n");
    return CHASE_CUDA_FAIL();
  }
  *sweeps = hst[1];
  *conv = hst[2] != 0;
  *in_g1 = hst[3] != 0;
  return CHASE_OK;
}

// ------------------------------------------------------ blocked FP32 Jacobi
// The FP32 stage as a block Jacobi method: the columns are cut into blocks of
// BJ_B, the blocks are paired in round-robin order (as the scalar method pairs
// columns), and per round every block pair's 2 BJ_B x 2 BJ_B principal
// submatrix S is diagonalised by one cyclic Jacobi sweep in shared memory,
// which accumulates its rotations into R (S <- R^H S R). The pair's columns of
// G and Z are then multiplied by R and its rows of G by R^H, as small GEMMs.
// Pairs of one round touch disjoint columns (and rows), so they run in
// parallel; a sweep visits every block pair once. Compared with one scalar
// rotation per column pair and round, the matrix streams through memory
// BJ_B times less often.
constexpr int BJ_B = 32;          // block width
constexpr int BJ_M = 2 * BJ_B;    // order of a block pair
constexpr int BJ_T = 256;
constexpr int BJ_ROWS = 64;       // rows (or columns) of G per CTA in the update kernels

__device__ __forceinline__ void bj_pair(int64_t n, int nb, int nbp, int round, int k, int64_t& i0,
                                        int& ni, int64_t& j0, int& nj) {
  auto pos = [&](int i) { return i == 0 ? 0 : 1 + (i - 1 + round) % (nbp - 1); };
  int p = pos(k), q = pos(nbp - 1 - k);
  if (p > q) {
    const int t = p;
    p = q;
    q = t;
  }
  i0 = (int64_t)p * BJ_B;
  j0 = (int64_t)q * BJ_B;
  ni = p < nb ? (int)min((int64_t)BJ_B, n - i0) : 0;
  nj = q < nb ? (int)min((int64_t)BJ_B, n - j0) : 0;
}
// global index of local index a of a block pair (first block, then second)
__device__ __forceinline__ int64_t bj_gidx(int a, int64_t i0, int ni, int64_t j0) {
  return a < ni ? i0 + a : j0 + (a - ni);
}

constexpr int BJ_IT = 512;           // threads of the inner kernel
constexpr int BJ_P = BJ_M / 2;       // rotations of a round
constexpr int BJ_LD = BJ_M + 1;
constexpr int BJ_INNER_SMEM = 2 * BJ_M * BJ_LD * (int)sizeof(float2);

// J = [[c, u], [-conj(u), c]] with u = s phi for the pair p < q; pq = p | q << 8,
// and bit 16 where the rotation is not the identity
struct Jrot {
  float c, ux, uy;
  int pq;
};
// The rotation of make_rot_t for a sweep, with approximate square roots and
// quotients (two units in the last place) and a Newton step on c and on 1 / |b|,
// so that J is unitary to FP32 rounding: this chain is a third of a round's
// latency, and the annihilated entry need only be small beside the FP32 rounding
// of the others.
__device__ __forceinline__ Jrot fast_rot(float a, float d, float2 b, float& app, float& aqq) {
  Jrot r;
  float bb = fmaf(b.x, b.x, b.y * b.y), back = 1.f;
  if (bb < 1e-30f) {  // squares near FP32's smallest: the rotation of 2^50 times the block
    a *= 0x1p50f;
    d *= 0x1p50f;
    b.x *= 0x1p50f;
    b.y *= 0x1p50f;
    bb = fmaf(b.x, b.x, b.y * b.y);
    back = 0x1p-50f;
  }
  if (!(bb > 1e-30f) || bb <= Cx<float>::eps * Cx<float>::eps * fabsf(a) * fabsf(d)) {
    r.c = 1.f; r.ux = 0.f; r.uy = 0.f; r.pq = 0; app = a * back; aqq = d * back;
    return r;
  }
  float ri = rsqrtf(bb);
  ri = ri * fmaf(-0.5f * bb, ri * ri, 1.5f);
  const float ab = bb * ri, tau = 0.5f * (d - a) * ri, at = fabsf(tau);
  const float q = fmaf(tau, tau, 1.f);
  const float t = copysignf(at > 1e15f ? __fdividef(0.5f, at) : __fdividef(1.f, at + q * rsqrtf(q)),
                            tau);
  const float w = fmaf(t, t, 1.f);
  float c = rsqrtf(w);
  c = c * fmaf(-0.5f * w, c * c, 1.5f);
  const float sr = t * c * ri;
  r.c = c;
  r.ux = sr * b.x;
  r.uy = sr * b.y;
  r.pq = 1 << 16;
  app = fmaf(-t, ab, a) * back;
  aqq = fmaf(t, ab, d) * back;
  return r;
}

// One cyclic sweep on S (64 x 64, Hermitian, ld BJ_LD in shared memory; a
// smaller matrix is padded with zeros, which no rotation touches), its rotations
// accumulated into R, by BJ_IT threads. It is a chain of 63 rounds, so what
// counts is a round's latency and its instructions: the 2 x 2 block of S where
// pairs k < l meet is rotated from both sides at once (one barrier instead of
// two), its mirror image is written and not computed, the pairs' own blocks are
// set exactly by the threads that compute the rotations. Warp w takes the blocks
// of pair w and of pair 31 - w, together one per lane, and rows w, w + 16, .. of
// R, a lane per pair. Bound by the 128 bytes a cycle of shared memory (8 KB of R and
// S's blocks a round, read and written).
__device__ __forceinline__ void bj_sweep(float2* S, float2* R, Jrot* rots) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  static_assert(BJ_P == 32 && BJ_IT / 32 == BJ_P / 2, "one pair per lane, two per warp");
  // the off-diagonal block of this lane: pairs k < l
  const bool lower = lane < warp;
  const int k = lower ? BJ_P - 1 - warp : warp, l = lower ? BJ_P - 1 - lane : lane;
  for (int rd = 0; rd < BJ_M - 1; ++rd) {
    __syncthreads();
    if (t < BJ_P) {
      int p, q;
      rr_pair(BJ_M, rd, t, p, q);
      float app, aqq;
      Jrot r = fast_rot(S[p * BJ_LD + p].x, S[q * BJ_LD + q].x, S[p * BJ_LD + q], app, aqq);
      if (r.pq) {  // the rotated 2 x 2 block exactly (no other thread reads it)
        S[p * BJ_LD + p] = make_float2(app, 0.f);
        S[q * BJ_LD + q] = make_float2(aqq, 0.f);
        S[p * BJ_LD + q] = make_float2(0.f, 0.f);
        S[q * BJ_LD + p] = make_float2(0.f, 0.f);
      }
      r.pq |= p | q << 8;
      rots[t] = r;
    }
    __syncthreads();
    const Jrot jm = rots[lane];
    const int2 pm = make_int2(jm.pq & 255, (jm.pq >> 8) & 255);
    if (k != l) {  // B <- J_k^H B J_l
      const Jrot jk = rots[k], jl = rots[l];
      if ((jk.pq | jl.pq) >> 16) {
        const int2 pk = make_int2(jk.pq & 255, (jk.pq >> 8) & 255);
        const int2 pl = make_int2(jl.pq & 255, (jl.pq >> 8) & 255);
        float2 b00 = S[pk.x * BJ_LD + pl.x], b01 = S[pk.x * BJ_LD + pl.y];
        float2 b10 = S[pk.y * BJ_LD + pl.x], b11 = S[pk.y * BJ_LD + pl.y];
        auto cols = [](float2& x, float2& y, const Jrot& j) {
          const float2 nx = make_float2(j.c * x.x - (j.ux * y.x + j.uy * y.y),
                                        j.c * x.y - (j.ux * y.y - j.uy * y.x));
          y = make_float2(j.ux * x.x - j.uy * x.y + j.c * y.x,
                          j.ux * x.y + j.uy * x.x + j.c * y.y);
          x = nx;
        };
        auto rows = [](float2& x, float2& y, const Jrot& j) {
          const float2 nx = make_float2(j.c * x.x - (j.ux * y.x - j.uy * y.y),
                                        j.c * x.y - (j.ux * y.y + j.uy * y.x));
          y = make_float2(j.ux * x.x + j.uy * x.y + j.c * y.x,
                          j.ux * x.y - j.uy * x.x + j.c * y.y);
          x = nx;
        };
        cols(b00, b01, jl);
        cols(b10, b11, jl);
        rows(b00, b10, jk);
        rows(b01, b11, jk);
        S[pk.x * BJ_LD + pl.x] = b00;
        S[pk.x * BJ_LD + pl.y] = b01;
        S[pk.y * BJ_LD + pl.x] = b10;
        S[pk.y * BJ_LD + pl.y] = b11;
        S[pl.x * BJ_LD + pk.x] = make_float2(b00.x, -b00.y);
        S[pl.y * BJ_LD + pk.x] = make_float2(b01.x, -b01.y);
        S[pl.x * BJ_LD + pk.y] = make_float2(b10.x, -b10.y);
        S[pl.y * BJ_LD + pk.y] = make_float2(b11.x, -b11.y);
      }
    }
    if (jm.pq >> 16) {
#pragma unroll
      for (int h = 0; h < BJ_M / (BJ_IT / 32); ++h) {
        float2* row = R + (warp + h * (BJ_IT / 32)) * BJ_LD;
        const float2 x = row[pm.x], y = row[pm.y];
        row[pm.x] = make_float2(jm.c * x.x - (jm.ux * y.x + jm.uy * y.y),
                                jm.c * x.y - (jm.ux * y.y - jm.uy * y.x));
        row[pm.y] = make_float2(jm.ux * x.x - jm.uy * x.y + jm.c * y.x,
                                jm.ux * x.y + jm.uy * x.x + jm.c * y.y);
      }
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(BJ_IT)
    bj_inner_kernel(int64_t n, int nb, int nbp, int round, const float2* __restrict__ G,
                    float2* __restrict__ Rbuf) {
  extern __shared__ float2 bj_smem[];
  float2* S = bj_smem;
  float2* R = bj_smem + BJ_M * BJ_LD;
  __shared__ Jrot rots[BJ_P];
  const int t = threadIdx.x;
  int64_t i0, j0;
  int ni, nj;
  bj_pair(n, nb, nbp, round, blockIdx.x, i0, ni, j0, nj);
  const int m = ni + nj;
  for (int e = t; e < BJ_M * BJ_M; e += BJ_IT) {
    const int a = e % BJ_M, c = e / BJ_M;
    S[a * BJ_LD + c] = (a < m && c < m)
                           ? G[bj_gidx(a, i0, ni, j0) + bj_gidx(c, i0, ni, j0) * n]
                           : make_float2(0.f, 0.f);
    R[a * BJ_LD + c] = make_float2(a == c ? 1.f : 0.f, 0.f);
  }
  bj_sweep(S, R, rots);
  float2* Rk = Rbuf + (int64_t)blockIdx.x * BJ_M * BJ_M;
  for (int e = t; e < m * m; e += BJ_IT)
    Rk[(e % m) + (e / m) * BJ_M] = R[(e % m) * BJ_LD + e / m];
}

// The FP32 stage of a matrix of order n <= 64 in one CTA: sweeps with the
// stopping rule of run_block_jacobi32, eigenvectors written in FP64 (ld n). The
// matrix is scaled by a power of two into FP32's range; info[0] = 1 when it holds an
// infinity or NaN, info[1] = sweeps.
__global__ void __launch_bounds__(BJ_IT)
    jacobi32_small_kernel(int n, const double2* __restrict__ G, int64_t ldg, int max_sweeps,
                          double tol_conv, double tol_stag, double2* __restrict__ X,
                          double* __restrict__ info) {
  extern __shared__ float2 bj_smem[];
  float2* S = bj_smem;
  float2* R = bj_smem + BJ_M * BJ_LD;
  __shared__ Jrot rots[BJ_P];
  __shared__ float red[BJ_IT / 32][2];
  __shared__ int s_exp;  // largest exponent field
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t == 0) s_exp = 0;
  __syncthreads();
  int ex = 0;
  for (int e = t; e < n * n; e += BJ_IT) {
    const double2 v = G[e % n + e / n * ldg];
    ex = max(ex, max((__double2hiint(v.x) >> 20) & 0x7ff, (__double2hiint(v.y) >> 20) & 0x7ff));
  }
  atomicMax(&s_exp, ex);
  __syncthreads();
  const int sh = 1023 - s_exp;
  if (t == 0) info[0] = s_exp == 0x7ff ? 1.0 : 0.0;
  for (int e = t; e < BJ_M * BJ_M; e += BJ_IT) {
    const int a = e % BJ_M, c = e / BJ_M;
    float2 g = make_float2(0.f, 0.f);
    if (a < n && c < n) {
      const double2 v = G[a + c * ldg];
      g = make_float2((float)ldexp(v.x, sh), (float)ldexp(v.y, sh));
    }
    S[a * BJ_LD + c] = g;
    R[a * BJ_LD + c] = make_float2(a == c ? 1.f : 0.f, 0.f);
  }
  double off_prev = 1e300;
  int sw = 0;
  for (; sw <= max_sweeps; ++sw) {
    __syncthreads();
    float o = 0.f, d = 0.f;
    for (int e = t; e < BJ_M * BJ_M; e += BJ_IT) {
      const int a = e % BJ_M, c = e / BJ_M;
      const float2 g = S[a * BJ_LD + c];
      const float v = fmaf(g.x, g.x, g.y * g.y);
      if (a == c) d += v;
      else o += v;
    }
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
      o += __shfl_xor_sync(0xffffffffu, o, w);
      d += __shfl_xor_sync(0xffffffffu, d, w);
    }
    if (lane == 0) {
      red[warp][0] = o;
      red[warp][1] = d;
    }
    __syncthreads();
    double so = 0.0, sf = 0.0;
#pragma unroll
    for (int w = 0; w < BJ_IT / 32; ++w) {
      so += red[w][0];
      sf += red[w][1];
    }
    const double off = sqrt(so), fro = sqrt(so + sf);
    if (off == 0.0 || off <= tol_conv * fro || (off <= tol_stag * fro && off > 0.25 * off_prev))
      break;
    off_prev = off;
    if (sw < max_sweeps) bj_sweep(S, R, rots);
  }
  if (t == 0) info[1] = (double)min(sw, max_sweeps);
  for (int e = t; e < n * n; e += BJ_IT) {
    const float2 r = R[(e % n) * BJ_LD + e / n];
    X[e] = make_double2((double)r.x, (double)r.y);
  }
}

// After a round's inner sweeps: G <- R^H G R and Z <- Z R with the block-diagonal R
// of all pairs, 64 x 64 tiles, one CTA each, one launch. The tile of G where pairs
// k <= l meet is multiplied from both sides and written with its conjugate
// transpose (half the tiles, and G stays Hermitian); tiles of Z take one product.
// Bound by FP32 FMAs and the shared-memory reads that feed them. n = 1072: separate
// column and row passes over all of G took 73 us a round.
constexpr int BJ_TILE = BJ_M * BJ_LD;
constexpr int BJ_UPD_SMEM = 3 * BJ_TILE * (int)sizeof(float2);

// o(r, c) = sum_a X(r, a) Y(a, c) for rows tx + 16 r and columns ty + 16 c; X is T
// row-major, or conj(R)^T for CONJT
template <bool CONJT>
__device__ __forceinline__ void bj_product(const float2* X, const float2* Y, int tx, int ty,
                                           float2 (&o)[4][4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) o[r][c] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int a = 0; a < BJ_M; ++a) {
    float2 x[4], y[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      x[r] = CONJT ? X[a * BJ_LD + tx + 16 * r] : X[(tx + 16 * r) * BJ_LD + a];
      if (CONJT) x[r].y = -x[r].y;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) y[c] = Y[a * BJ_LD + ty + 16 * c];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        o[r][c].x = fmaf(x[r].x, y[c].x, fmaf(-x[r].y, y[c].y, o[r][c].x));
        o[r][c].y = fmaf(x[r].x, y[c].y, fmaf(x[r].y, y[c].x, o[r][c].y));
      }
  }
}
// R of a pair (order m, column-major, ld 64) row-major into shared memory, zero padded
__device__ __forceinline__ void bj_load_r(float2* R, const float2* __restrict__ src, int m) {
  for (int e = threadIdx.x; e < BJ_M * BJ_M; e += BJ_T) {
    const int a = e % BJ_M, c = e / BJ_M;
    R[a * BJ_LD + c] = (a < m && c < m) ? src[a + c * BJ_M] : make_float2(0.f, 0.f);
  }
}

__global__ void __launch_bounds__(BJ_T)
    bj_update_kernel(int64_t n, int nb, int nbp, int round, int ng, float2* __restrict__ G,
                     float2* __restrict__ Z, const float2* __restrict__ Rbuf) {
  extern __shared__ float2 bj_smem[];
  float2* T = bj_smem;
  float2* Rl = bj_smem + BJ_TILE;
  float2* Rk = bj_smem + 2 * BJ_TILE;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4, npair = nbp / 2;
  const bool in_g = (int)blockIdx.x < ng;
  int k = 0, l;
  int64_t r0 = 0;
  if (in_g) {  // tile number l (l + 1) / 2 + k
    l = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
    while (l * (l + 1) / 2 > (int)blockIdx.x) --l;
    while ((l + 1) * (l + 2) / 2 <= (int)blockIdx.x) ++l;
    k = (int)blockIdx.x - l * (l + 1) / 2;
  } else {
    l = ((int)blockIdx.x - ng) % npair;
    r0 = (int64_t)(((int)blockIdx.x - ng) / npair) * BJ_ROWS;
  }
  int64_t li0, lj0, ki0 = 0, kj0 = 0;
  int lni, lnj, kni = 0, knj = 0;
  bj_pair(n, nb, nbp, round, l, li0, lni, lj0, lnj);
  const int ml = lni + lnj;
  int mk = 0;
  if (in_g) {
    bj_pair(n, nb, nbp, round, k, ki0, kni, kj0, knj);
    mk = kni + knj;
  } else {
    mk = (int)min((int64_t)BJ_ROWS, n - r0);
  }
  if (ml == 0 || mk <= 0) return;
  float2* M = in_g ? G : Z;
  auto row = [&](int a) { return in_g ? bj_gidx(a, ki0, kni, kj0) : r0 + a; };
  bj_load_r(Rl, Rbuf + (int64_t)l * BJ_M * BJ_M, ml);
  if (in_g) bj_load_r(Rk, Rbuf + (int64_t)k * BJ_M * BJ_M, mk);
  for (int e = t; e < BJ_M * BJ_M; e += BJ_T) {
    const int a = e % BJ_M, c = e / BJ_M;
    T[a * BJ_LD + c] = (a < mk && c < ml) ? M[row(a) + bj_gidx(c, li0, lni, lj0) * n]
                                          : make_float2(0.f, 0.f);
  }
  __syncthreads();
  float2 o[4][4];
  bj_product<false>(T, Rl, tx, ty, o);
  if (!in_g) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int cc = ty + 16 * c;
      if (cc >= ml) continue;
      const int64_t col = bj_gidx(cc, li0, lni, lj0);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (tx + 16 * r < mk) M[r0 + tx + 16 * r + col * n] = o[r][c];
    }
    return;
  }
  auto keep = [&]() {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) T[(tx + 16 * r) * BJ_LD + ty + 16 * c] = o[r][c];
    __syncthreads();
  };
  keep();
  bj_product<true>(Rk, T, tx, ty, o);
  keep();
  for (int e = t; e < BJ_M * BJ_M; e += BJ_T) {
    const int a = e % BJ_M, c = e / BJ_M;
    if (a < mk && c < ml) G[row(a) + bj_gidx(c, li0, lni, lj0) * n] = T[a * BJ_LD + c];
    if (k != l && a < ml && c < mk) {  // the mirror image
      const float2 v = T[c * BJ_LD + a];
      G[bj_gidx(a, li0, lni, lj0) + row(c) * n] = make_float2(v.x, -v.y);
    }
  }
}

__global__ void bj_norms_kernel(int64_t n, const float2* __restrict__ G, double* __restrict__ part) {
  __shared__ double so[256], sf[256];
  double o = 0.0, f = 0.0;
  const int64_t tot = n * n;
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < tot; e += (int64_t)gridDim.x * 256) {
    const float2 g = G[e];
    const double v = (double)g.x * g.x + (double)g.y * g.y;
    f += v;
    if (e % n != e / n) o += v;
  }
  so[threadIdx.x] = o;
  sf[threadIdx.x] = f;
  __syncthreads();
  for (int w = 128; w >= 1; w >>= 1) {
    if (threadIdx.x < w) {
      so[threadIdx.x] += so[threadIdx.x + w];
      sf[threadIdx.x] += sf[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = so[0];
    part[2 * blockIdx.x + 1] = sf[0];
  }
}

std::once_flag g_bj_attr[kMaxDevices];
void set_bj_attrs() {
  once_per_device(g_bj_attr, []() {
    cudaFuncSetAttribute(bj_inner_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         BJ_INNER_SMEM);
    cudaFuncSetAttribute(jacobi32_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         BJ_INNER_SMEM);
    cudaFuncSetAttribute(bj_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         BJ_UPD_SMEM);
  });
}

// Blocked FP32 Jacobi on G (n x n, destroyed) with eigenvectors into Z (starts
// as I): sweeps until off(G) <= tol_conv ||G||_F, or <= tol_stag ||G||_F with
// less than a 4x decrease in the last sweep, or max_sweeps. part: 512 doubles
// of device scratch, host_part: 512 doubles of host memory.
int run_block_jacobi32(cudaStream_t s, int64_t n, float2* G, float2* Z, float2* Rbuf,
                       double* part, double* host_part, int max_sweeps, double tol_conv,
                       double tol_stag, int* sweeps, bool* conv) {
  set_bj_attrs();
  const int nb = (int)cdiv(n, BJ_B);
  const int nbp = nb + (nb & 1);
  const int npair = nbp / 2;
  const unsigned gt = (unsigned)cdiv(n, BJ_ROWS);
  const int ng = npair * (npair + 1) / 2;  // tiles of G on and above the diagonal
  constexpr int kNormBlocks = 256;
  double off_prev = 1e300;
  *conv = false;
  int sw = 0;
  for (; sw <= max_sweeps; ++sw) {
    bj_norms_kernel<<<kNormBlocks, 256, 0, s>>>(n, G, part);
    count_launch();
    if (cudaMemcpyAsync(host_part, part, 2 * kNormBlocks * sizeof(double), cudaMemcpyDeviceToHost,
                        s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return CHASE_CUDA_FAIL();
    double o = 0.0, f = 0.0;
    for (int b = 0; b < kNormBlocks; ++b) {
      o += host_part[2 * b];
      f += host_part[2 * b + 1];
    }
    const double off = std::sqrt(o), fro = std::sqrt(f);
    if (off == 0.0 || off <= tol_conv * fro || (off <= tol_stag * fro && off > 0.25 * off_prev)) {
      *conv = true;
      break;
    }
    off_prev = off;
    if (sw == max_sweeps) break;
    for (int rd = 0; rd < nbp - 1; ++rd) {
      bj_inner_kernel<<<npair, BJ_IT, BJ_INNER_SMEM, s>>>(n, nb, nbp, rd, G, Rbuf);
      bj_update_kernel<<<(unsigned)(ng + npair * (int)gt), BJ_T, BJ_UPD_SMEM, s>>>(n, nb, nbp, rd,
                                                                                ng, G, Z, Rbuf);
      count_launch();
      count_launch();
    }
    if (cudaGetLastError() != cudaSuccess) return CHASE_CUDA_FAIL();
  }
  *sweeps = sw;
  return CHASE_OK;
}

__global__ void rank_kernel(int64_t n, const double2* Gw, double* w, int* rank) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = Gw[i + i * n].x;
  int64_t rk = 0;
  for (int64_t j = 0; j < n; ++j) {
    const double u = Gw[j + j * n].x;
    rk += (u < v) || (u == v && j < i);
  }
  rank[i] = (int)rk;
  w[rk] = v;
}
__global__ void permute_cols_kernel(int64_t n, const double2* Zw, const int* rank, double2* Z,
                                    int64_t ldz) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t c = blockIdx.y;
  if (i >= n) return;
  Z[i + (int64_t)rank[c] * ldz] = Zw[i + c * n];
}

// ------------------------------------------ FP64 refinement of the FP32 pairs
// One step of the iterative refinement of Ogita and Aishima (2018) for an
// approximate eigenvector matrix X of Hermitian G, with S = X^H G X and
// R = I - X^H X: lambda_i = Re s_ii / (1 - Re r_ii) and
// E_ij = (s_ij + lambda_j r_ij) / (lambda_j - lambda_i) (i != j), E_ii = r_ii / 2,
// then X <- X (I + E). Quadratic convergence from the FP32 Jacobi vectors. A
// pair whose first-order correction would exceed 1e-3 (eigenvalues too close
// to separate at this accuracy; larger corrections made near-degenerate pairs
// oscillate in tests) is only orthogonalised (E_ij = r_ij / 2); the largest
// |s_ij| of such pairs is reported so that FP64 Jacobi sweeps can finish them.
__global__ void oa_lambda_kernel(int64_t n, const double2* __restrict__ S,
                                 const double2* __restrict__ XX, double* __restrict__ lam) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  lam[i] = S[i + i * n].x / XX[i + i * n].x;  // 1 - r_ii = (X^H X)_ii
}
__global__ void oa_e_kernel(int64_t n, const double2* __restrict__ S,
                            const double2* __restrict__ XX, const double* __restrict__ lam,
                            double2* __restrict__ E, double* __restrict__ partial,
                            int* __restrict__ pairs, int* __restrict__ npairs) {
  __shared__ double me[256], mc[256];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // row
  const int64_t j = blockIdx.y;                                        // column
  double emax = 0.0, cmax = 0.0;
  if (i < n) {
    const double2 x = XX[i + j * n];
    const double2 r = make_double2((i == j ? 1.0 : 0.0) - x.x, -x.y);
    double2 e;
    if (i == j) {
      e = make_double2(0.5 * r.x, 0.5 * r.y);
      emax = 0.5 * sqrt(r.x * r.x + r.y * r.y);
    } else {
      const double2 sv = S[i + j * n];
      const double lj = lam[j], d = lj - lam[i];
      const double2 num = make_double2(fma(lj, r.x, sv.x), fma(lj, r.y, sv.y));
      const double an = sqrt(num.x * num.x + num.y * num.y);
      if (an == 0.0 && d == 0.0) {  // equal values without coupling: no pair to finish
        e = make_double2(0.5 * r.x, 0.5 * r.y);
        emax = 0.5 * sqrt(r.x * r.x + r.y * r.y);
      } else if (an <= 1e-3 * fabs(d)) {
        e = make_double2(num.x / d, num.y / d);
        emax = an / fabs(d);
      } else {
        e = make_double2(0.5 * r.x, 0.5 * r.y);
        emax = 0.5 * sqrt(r.x * r.x + r.y * r.y);
        cmax = sqrt(sv.x * sv.x + sv.y * sv.y);
        // a pair left to the FP64 finish: recorded (capacity permitting; the
        // host takes the full FP64 sweeps when the list overflows)
        const int k = atomicAdd(npairs, 1);
        if (k < kMaxClusterPairs) {
          pairs[2 * k] = (int)i;
          pairs[2 * k + 1] = (int)j;
        }
      }
    }
    E[i + j * n] = e;
  }
  me[threadIdx.x] = emax;
  mc[threadIdx.x] = cmax;
  __syncthreads();
  for (int w = 128; w >= 1; w >>= 1) {
    if (threadIdx.x < w) {
      me[threadIdx.x] = fmax(me[threadIdx.x], me[threadIdx.x + w]);
      mc[threadIdx.x] = fmax(mc[threadIdx.x], mc[threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int64_t b = blockIdx.x + (int64_t)blockIdx.y * gridDim.x;
    partial[2 * b] = me[0];
    partial[2 * b + 1] = mc[0];
  }
}
// E = (I - XX) / 2: one orthogonalisation step X <- X (I + E)
__global__ void half_residual_kernel(int64_t n, const double2* __restrict__ XX,
                                     double2* __restrict__ E) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= n) return;
  const double2 x = XX[i + j * n];
  E[i + j * n] = make_double2(0.5 * ((i == j ? 1.0 : 0.0) - x.x), -0.5 * x.y);
}
__global__ void max2_kernel(int64_t nb, const double* __restrict__ partial, double* __restrict__ out) {
  __shared__ double a[256], c[256];
  double x = 0.0, y = 0.0;
  for (int64_t b = threadIdx.x; b < nb; b += 256) {
    x = fmax(x, partial[2 * b]);
    y = fmax(y, partial[2 * b + 1]);
  }
  a[threadIdx.x] = x;
  c[threadIdx.x] = y;
  __syncthreads();
  for (int w = 128; w >= 1; w >>= 1) {
    if (threadIdx.x < w) {
      a[threadIdx.x] = fmax(a[threadIdx.x], a[threadIdx.x + w]);
      c[threadIdx.x] = fmax(c[threadIdx.x], c[threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = a[0];
    out[1] = c[0];
  }
}
// Block S_c = X_c^H (G X_c) of each cluster c of size k (clusters of one size,
// consecutive in XI / TI): CTAs (x: cluster, y: share of its entries) of 8 warps, one
// warp per output entry at a time, lanes over rows, fixed-order reduction. Output
// k x k column-major. (A CTA per cluster left it to a few SMs' FP64 pipes: 0.4 ms for
// clusters of 20 columns of 1072.)
__global__ void cluster_gram_kernel(int64_t n, int k, const double2* __restrict__ XI,
                                    const double2* __restrict__ TI, int64_t ld,
                                    double2* __restrict__ Sout) {
  const int c = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double2* X = XI + (int64_t)c * k * ld;
  const double2* T = TI + (int64_t)c * k * ld;
  for (int e = warp + 8 * blockIdx.y; e < k * k; e += 8 * gridDim.y) {
    const int a = e % k, b = e / k;
    double2 acc = make_double2(0.0, 0.0);
    for (int64_t r = lane; r < n; r += 32) acc = cadd(acc, cmulc(X[r + a * ld], T[r + b * ld]));
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
    }
    if (lane == 0) Sout[(int64_t)c * k * k + a + b * k] = acc;
  }
}
// X(:, idx_c) = XI_c Z_c for each cluster (its FP64 eigenvectors), and the
// cluster's eigenvalues into lam at the same column indices.
__global__ void cluster_apply_kernel(int64_t n, int k, const double2* __restrict__ XI, int64_t ld,
                                     const double2* __restrict__ Z, const double* __restrict__ wz,
                                     const int* __restrict__ idx, double2* __restrict__ X,
                                     double* __restrict__ lam) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int c = blockIdx.y;
  const double2* Xc = XI + (int64_t)c * k * ld;
  const double2* Zc = Z + (int64_t)c * k * k;
  const int* ic = idx + (int64_t)c * k;
  if (blockIdx.x == 0 && threadIdx.x < k) lam[ic[threadIdx.x]] = wz[(int64_t)c * k + threadIdx.x];
  if (r >= n) return;
  for (int b = 0; b < k; ++b) {
    double2 acc = make_double2(0.0, 0.0);
    for (int a = 0; a < k; ++a) acc = cadd(acc, cmul(Xc[r + a * ld], Zc[a + b * k]));
    X[r + (int64_t)ic[b] * n] = acc;
  }
}

// X(:, idx[j]) = P(:, j) and lam[idx[j]] = Re S(j, j) for a large cluster's
// eigenvectors P (n x m, ld n) and its diagonalised block S (m x m, ld m).
__global__ void scatter_cluster_kernel(int64_t n, int64_t m, const double2* __restrict__ P,
                                       const int* __restrict__ idx, const double2* __restrict__ S,
                                       double2* __restrict__ X, double* __restrict__ lam) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = blockIdx.y;
  if (blockIdx.x == 0 && threadIdx.x == 0) lam[idx[j]] = S[j + j * m].x;
  if (r < n) X[r + (int64_t)idx[j] * n] = P[r + j * n];
}

__global__ void rank_vec_kernel(int64_t n, const double* __restrict__ lam, double* w, int* rank) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = lam[i];
  int64_t rk = 0;
  for (int64_t j = 0; j < n; ++j) {
    const double u = lam[j];
    rk += (u < v) || (u == v && j < i);
  }
  rank[i] = (int)rk;
  w[rk] = v;
}
__global__ void frob2_kernel(int64_t n, const double2* __restrict__ G, int64_t ldg,
                             double* __restrict__ partial) {
  __shared__ double a[256];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  double v = 0.0;
  if (i < n) {
    const double2 g = G[i + j * ldg];
    v = g.x * g.x + g.y * g.y;
  }
  a[threadIdx.x] = v;
  __syncthreads();
  for (int w = 128; w >= 1; w >>= 1) {
    if (threadIdx.x < w) a[threadIdx.x] += a[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int64_t b = blockIdx.x + (int64_t)blockIdx.y * gridDim.x;
    partial[2 * b] = sqrt(a[0]);  // max of column-block norms: a cheap scale of ||G||
    partial[2 * b + 1] = 0.0;
  }
}

std::once_flag g_small_attr[kMaxDevices];

}  // namespace

size_t jacobi_red_elems() { return (size_t)2 * kCoopMaxGrid + 16; }

namespace {
// refinement products: P = A B (n x n) or P = X^H Y, on the tensor cores when
// the context supplied a product, else with the CUDA-core kernels
cudaError_t heev_nn(cudaStream_t s, const JacobiWork& wk, bool tc, int64_t n, const double2* A,
                    int64_t lda, const double2* B, const Epilogue& ep, bool extended = false) {
  if (tc && wk.gemm) return wk.gemm(wk.gemm_ctx, n, n, A, lda, false, n, B, n, ep, extended);
  return zgemm_nn(s, n, n, n, A, lda, B, n, ep);
}
cudaError_t heev_cn(cudaStream_t s, const JacobiWork& wk, bool tc, int64_t n, const double2* X,
                    const double2* Y, double2* P, bool hermitian, bool extended = false) {
  if (tc && wk.gemm) {
    Epilogue ep{};
    ep.mode = EPI_STORE;
    ep.Y = P;
    ep.ldy = n;
    cudaError_t e = wk.gemm(wk.gemm_ctx, n, n, X, n, true, n, Y, n, ep, extended);
    if (e != cudaSuccess || !hermitian) return e;
    return hermitian_part(s, n, P, n);
  }
  return zgram(s, n, n, n, X, n, Y, n, P, n, hermitian, wk.gram_ws, wk.gram_ws_elems);
}
}  // namespace

size_t jacobi_rot_elems(int64_t n) {
  const int64_t nb = cdiv(n, BJ_B);
  return (size_t)((nb + 1) / 2) * BJ_M * BJ_M;
}

size_t jacobi_params_elems(int64_t n) { return (size_t)8 * (n / 2 + 2) + 8 + n; }

cudaError_t jacobi_small_batched(cudaStream_t s, int n, int batch, const double2* G, double* w,
                                 double2* Z, int* status, int max_sweeps, bool real) {
  if (n > SJ_MAX || n < 1) return cudaErrorInvalidValue;
  constexpr size_t elems = 2 * SJ_MAX * SJ_LD;
  once_per_device(g_small_attr, []() {
    cudaFuncSetAttribute(jacobi_small_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(elems * sizeof(double2)));
    cudaFuncSetAttribute(jacobi_small_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(elems * sizeof(double)));
  });
  const int cap = max_sweeps > 0 ? std::min(max_sweeps, kMaxSweeps) : kMaxSweeps;
  if (real)
    jacobi_small_kernel<true><<<batch, SJ_T, elems * sizeof(double), s>>>(n, G, w, Z, status, cap);
  else
    jacobi_small_kernel<false><<<batch, SJ_T, elems * sizeof(double2), s>>>(n, G, w, Z, status, cap);
  count_launch();
  return cudaGetLastError();
}

namespace {
// FP64 finish restricted to the clusters of pairs the refinement left coupled
// (connected components of the recorded pairs, union-find on the host). For
// each cluster I: S_I = X_I^H G X_I in FP64, its eigenvectors Z_I by Jacobi
// (clusters of up to 64 batched in the single-CTA kernel, larger ones one by
// one in the cooperative kernel on their m x m block), X_I <- X_I Z_I, and its
// eigenvalues into lam. A cluster's coupling to every other vector is already
// at FP64 rounding level after the refinement, so the blocks are independent.
// Returns 1 when done, 0 when not applicable (pair list overflowed, or a
// cluster above 0.7 n, where the full FP64 sweeps cost about the same),
// -status on an error. *sweeps64 receives the FP64 sweeps of the large clusters.
int cluster_finish(cudaStream_t s, int64_t n, const double2* G, int64_t ldg, double2* X,
                   double2* XI, double* lam, JacobiWork& wk, int* status, int* info,
                   int max_sweeps, int* sweeps64) {
  info[0] = info[1] = 0;
  *sweeps64 = 0;
  int np = 0;
  if (cudaMemcpyAsync(&np, wk.npairs, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return -CHASE_CUDA_FAIL();
  info[1] = np;
  if (np <= 0 || np > kMaxClusterPairs) return 0;
  std::vector<int> pr(2 * (size_t)np);
  if (cudaMemcpy(pr.data(), wk.pairs, pr.size() * sizeof(int), cudaMemcpyDeviceToHost) !=
      cudaSuccess)
    return -CHASE_CUDA_FAIL();
  std::vector<int> parent((size_t)n);
  for (int64_t i = 0; i < n; ++i) parent[i] = (int)i;
  auto find = [&](int x) {
    while (parent[x] != x) x = parent[x] = parent[parent[x]];
    return x;
  };
  for (int k = 0; k < np; ++k) {
    const int a = find(pr[2 * k]), b = find(pr[2 * k + 1]);
    if (a != b) parent[std::max(a, b)] = std::min(a, b);
  }
  // members of each component in ascending index order, components by size
  std::vector<std::vector<int>> comp((size_t)n);
  for (int64_t i = 0; i < n; ++i) comp[find((int)i)].push_back((int)i);
  std::vector<int> roots;
  for (int64_t i = 0; i < n; ++i)
    if (comp[i].size() >= 2) {
      info[0] = std::max(info[0], (int)comp[i].size());
      roots.push_back((int)i);
    }
  // a large cluster's Jacobi rotations (m x m, ld m) live in G32a viewed as FP64
  if ((double)info[0] > 0.7 * (double)n) return 0;
  if (roots.empty()) return 0;
  std::stable_sort(roots.begin(), roots.end(),
                   [&](int a, int b) { return comp[a].size() < comp[b].size(); });
  std::vector<int> idx;
  struct Group { int k, count; int64_t off; };
  std::vector<Group> groups;
  for (int r : roots) {
    const int k = (int)comp[r].size();
    if (groups.empty() || groups.back().k != k) groups.push_back({k, 0, (int64_t)idx.size()});
    groups.back().count++;
    idx.insert(idx.end(), comp[r].begin(), comp[r].end());
  }
  const int64_t ktot = (int64_t)idx.size();
  if (cudaMemcpyAsync(wk.cl_idx, idx.data(), ktot * sizeof(int), cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaMemsetAsync(status, 0, sizeof(int), s) != cudaSuccess)
    return -CHASE_CUDA_FAIL();
  // XI = X(:, idx), TI = G XI (FP64)
  if (gather_cols(s, n, ktot, X, n, wk.cl_idx, XI, n) != cudaSuccess) return -CHASE_CUDA_FAIL();
  Epilogue ep{};
  ep.mode = EPI_STORE;
  ep.Y = wk.T;
  ep.ldy = n;
  if (zgemm_nn(s, n, ktot, n, G, ldg, XI, n, ep) != cudaSuccess) return -CHASE_CUDA_FAIL();
  double* wz = reinterpret_cast<double*>(wk.G32b);  // ktot eigenvalues
  for (const Group& g : groups) {
    const int64_t off = g.off;
    if (g.k > SJ_MAX) {  // one large cluster at a time, FP64 cooperative Jacobi
      for (int q = 0; q < g.count; ++q) {
        const int64_t m = g.k, o = off + (int64_t)q * m;
        if (zgram(s, n, m, m, XI + o * n, n, wk.T + o * n, n, wk.Gw, m, false, wk.gram_ws,
                  wk.gram_ws_elems) != cudaSuccess ||
            hermitian_part(s, m, wk.Gw, m) != cudaSuccess)
          return -CHASE_CUDA_FAIL();
        double2* Zr = reinterpret_cast<double2*>(wk.G32a);
        identity_kernel<<<dim3((unsigned)cdiv(m, 128), (unsigned)m, 1), 128, 0, s>>>(m, Zr);
        count_launch();
        int sw = 0;
        bool conv = false, in_g1 = false;
        RC_NEG(run_coop<double>(s, m, wk.Gw, wk.Gw2, Zr, wz + n, wk.red, max_sweeps, 1e-15, 1e-12,
                                &sw, &conv, &in_g1));
        *sweeps64 += sw;
        if (!conv) return -CHASE_ERR_HEEV_NOCONV;
        Epilogue ez{};
        ez.mode = EPI_STORE;  // P = X_I Z into the cluster's (now free) columns of T
        ez.Y = wk.T + o * n;
        ez.ldy = n;
        if (zgemm_nn(s, n, m, m, XI + o * n, n, Zr, m, ez) != cudaSuccess) return -CHASE_CUDA_FAIL();
        scatter_cluster_kernel<<<dim3((unsigned)cdiv(n, 128), (unsigned)m, 1), 128, 0, s>>>(
            n, m, wk.T + o * n, wk.cl_idx + o, in_g1 ? wk.Gw2 : wk.Gw, X, lam);
        count_launch();
      }
      continue;
    }
    cluster_gram_kernel<<<dim3((unsigned)g.count, (unsigned)std::min<int64_t>(64, cdiv(g.k * g.k, 8)), 1),
                          256, 0, s>>>(n, g.k, XI + off * n, wk.T + off * n, n, wk.Gw);
    count_launch();
    if (jacobi_small_batched(s, g.k, g.count, wk.Gw, wz + off, wk.Gw2, status, wk.max_sweeps) !=
        cudaSuccess)
      return -CHASE_CUDA_FAIL();
    cluster_apply_kernel<<<dim3((unsigned)cdiv(n, 128), (unsigned)g.count, 1), 128, 0, s>>>(
        n, g.k, XI + off * n, n, wk.Gw2, wz + off, wk.cl_idx + off, X, lam);
    count_launch();
  }
  int hs = 0;
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(&hs, status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return -CHASE_CUDA_FAIL();
  info[1] = (int)roots.size();
  return hs ? -CHASE_ERR_HEEV_NOCONV : 1;
}
}  // namespace

int jacobi_heev(cudaStream_t s, int64_t n, const double2* G, int64_t ldg, double* w, double2* Z,
                int64_t ldz, JacobiWork& wk, int* sweeps_out, int* fp64_sweeps_out,
                int* cluster_out) {
  if (cluster_out) cluster_out[0] = cluster_out[1] = cluster_out[2] = 0;
  if (n <= 0) return CHASE_OK;
  int* status = reinterpret_cast<int*>(wk.red + 2 * kCoopMaxGrid + 8);
  // FP64 in one CTA: G (ld n) into Gw, the single-CTA kernel into Zw, copied to Z
  auto small_fp64 = [&]() -> int {
    cudaError_t e = cudaMemsetAsync(status, 0, sizeof(int), s);
    if (e != cudaSuccess) return CHASE_CUDA_FAIL();
    e = cudaMemcpy2DAsync(wk.Gw, n * sizeof(double2), G, ldg * sizeof(double2),
                          n * sizeof(double2), n, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return CHASE_CUDA_FAIL();
    e = jacobi_small_batched(s, (int)n, 1, wk.Gw, w, wk.Zw, status, wk.max_sweeps);
    if (e != cudaSuccess) return CHASE_CUDA_FAIL();
    e = cudaMemcpy2DAsync(Z, ldz * sizeof(double2), wk.Zw, n * sizeof(double2),
                          n * sizeof(double2), n, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return CHASE_CUDA_FAIL();
    int hs = 0;
    e = cudaMemcpyAsync(&hs, status, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return CHASE_CUDA_FAIL();
    if (cudaStreamSynchronize(s) != cudaSuccess) return CHASE_CUDA_FAIL();
    if (sweeps_out) *sweeps_out = 0;
    return hs ? CHASE_ERR_HEEV_NOCONV : CHASE_OK;
  };
  if (n <= kSmallFp64) return small_fp64();
  // --- FP32 sweeps on the converted matrix
  const dim3 g2((unsigned)cdiv(n, 128), (unsigned)n, 1);
  int sw32 = 0;
  bool conv32 = false;
  // stage caps: 30 FP32 sweeps, 8 refinement steps, kMaxSweeps FP64 sweeps, each
  // lowered to the caller's cap when one is set
  auto cap = [&](int def) { return wk.max_sweeps > 0 ? std::min(def, wk.max_sweeps) : def; };
  constexpr double kTol32 = 4e-6, kStag32 = 1e-4;
  double* out2 = wk.red + 2 * kCoopMaxGrid + 12;  // two maxima; [2]: non-finite input, [3]: FP32 sweeps
  if (n <= BJ_M) {
    set_bj_attrs();
    jacobi32_small_kernel<<<1, BJ_IT, BJ_INNER_SMEM, s>>>((int)n, G, ldg, cap(30), kTol32, kStag32,
                                                          wk.Zw, out2 + 2);
    count_launch();
  } else {
    int* max_exp = reinterpret_cast<int*>(out2 + 2);
    if (cudaMemsetAsync(max_exp, 0, sizeof(int), s) != cudaSuccess) return CHASE_CUDA_FAIL();
    max_exp_kernel<<<g2, 128, 0, s>>>(n, G, ldg, max_exp); count_launch();
    init32_kernel<<<g2, 128, 0, s>>>(n, G, ldg, max_exp, wk.G32a, wk.Z32); count_launch();
    // blocked FP32 Jacobi: G32a is G (in place), Rb the block rotations
    if (jacobi_rot_elems(n) > wk.rb_elems) return CHASE_ERR_INVALID_ARG;
    RC_(run_block_jacobi32(s, n, wk.G32a, wk.Z32, wk.Rb, wk.red, wk.host_part, cap(30), kTol32,
                           kStag32, &sw32, &conv32));
    promote_kernel<<<g2, 128, 0, s>>>(n, wk.Z32, wk.Zw); count_launch();
  }
  // --- FP64: refine the FP32 eigenvectors (Ogita-Aishima steps, FP64 GEMMs)
  const unsigned gb = (unsigned)cdiv(n, 256);
  const int64_t nb = (int64_t)gb * n;  // partial slots (2 doubles each) of the E kernel
  double* lam = wk.params;             // n eigenvalue estimates (params is free here)
  double2* X = wk.Zw;
  double2* Xn = wk.Zw2;
  // scale of G for the cluster test
  frob2_kernel<<<dim3(gb, (unsigned)n, 1), 256, 0, s>>>(n, G, ldg, reinterpret_cast<double*>(wk.T));
  count_launch();
  max2_kernel<<<1, 256, 0, s>>>(nb, reinterpret_cast<double*>(wk.T), out2); count_launch();
  if (cudaMemcpyAsync(wk.host_red, out2, 4 * sizeof(double), cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CHASE_CUDA_FAIL();
  if (n <= BJ_M) {
    if (wk.host_red[2] != 0.0) return CHASE_ERR_HEEV_NOCONV;
    sw32 = (int)wk.host_red[3];
  }
  // sqrt(n) times the largest norm of a 256-row column segment: within a factor
  // sqrt(n) of ||G||_2 either way, enough for the 1e-14 cluster test below
  const double gscale = wk.host_red[0] * std::sqrt((double)n);
  int refine = 0;
  double emax = 1.0, cmax = 0.0;
  // With the digit-sliced tensor-core products (when the context supplies them)
  // the first, coarse steps use the 21-pair products, whose error (about
  // sqrt(n) 2^-50 of max|G_i.| max|X_.j| per entry) is far above what the Ritz
  // values need. Once the corrections fall below 1e-6 the steps are fine ones:
  // G X, X^H (G X) and X^H X, whose off-diagonal parts cancel to the size of
  // the corrections, keep the level-8 digit pairs too (error near the digit
  // rounding of the operands, a few 2^-48 of ||G||, like the CUDA-core FP64
  // products' sqrt(n) 2^-53), and so does the final orthogonalisation. Without
  // them, all products are the CUDA-core FP64 ones.
  // Up to order kCoreRefine those are the faster ones too.
  const bool tc = wk.gemm != nullptr && n > kCoreRefine;
  bool fine = false;
  const int max_refine = cap(8);
  for (; refine < max_refine; ++refine) {  // 2-4 steps from FP32 accuracy; a slow start gets more
    Epilogue ep{};
    ep.mode = EPI_STORE;
    ep.Y = wk.T;
    ep.ldy = n;
    if (heev_nn(s, wk, tc, n, G, ldg, X, ep, fine) != cudaSuccess ||         // T = G X
        heev_cn(s, wk, tc, n, X, wk.T, wk.Gw, false, fine) != cudaSuccess ||   // S = X^H T
        heev_cn(s, wk, tc, n, X, X, wk.Gw2, true, fine) != cudaSuccess)        // X^H X
      return CHASE_CUDA_FAIL();
    oa_lambda_kernel<<<(unsigned)cdiv(n, 128), 128, 0, s>>>(n, wk.Gw, wk.Gw2, lam); count_launch();
    // E into T (T is free once S is formed)
    if (cudaMemsetAsync(wk.npairs, 0, sizeof(int), s) != cudaSuccess) return CHASE_CUDA_FAIL();
    oa_e_kernel<<<dim3(gb, (unsigned)n, 1), 256, 0, s>>>(n, wk.Gw, wk.Gw2, lam, wk.T,
                                                        reinterpret_cast<double*>(wk.G32a),
                                                        wk.pairs, wk.npairs);
    count_launch();
    max2_kernel<<<1, 256, 0, s>>>(nb, reinterpret_cast<double*>(wk.G32a), out2); count_launch();
    // Xn = X + X E
    if (cudaMemcpyAsync(Xn, X, (size_t)n * n * sizeof(double2), cudaMemcpyDeviceToDevice, s) !=
        cudaSuccess)
      return CHASE_CUDA_FAIL();
    Epilogue eu{};
    eu.mode = EPI_FILTER;
    eu.alpha = 1.0;
    eu.beta = 1.0;
    eu.gamma = 0.0;
    eu.X = Xn;
    eu.ldx = n;
    eu.Y = Xn;
    eu.ldy = n;
    if (heev_nn(s, wk, tc, n, X, n, wk.T, eu) != cudaSuccess) return CHASE_CUDA_FAIL();
    std::swap(X, Xn);
    if (cudaMemcpyAsync(wk.host_red, out2, 2 * sizeof(double), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return CHASE_CUDA_FAIL();
    emax = wk.host_red[0];
    cmax = wk.host_red[1];
    // the applied correction was ~emax; the error left is ~emax^2 (plus the
    // products' own error, hence the last step with the accurate products)
    if (emax <= 1e-8 && (!tc || fine)) {
      ++refine;
      break;
    }
    if (emax <= 1e-6) fine = true;
  }
  {
    // the corrections of close pairs carry rounding of order u / gap; one more
    // orthogonalisation step brings X^H X back to I at working precision
    if (heev_cn(s, wk, tc, n, X, X, wk.Gw2, true, true) != cudaSuccess) return CHASE_CUDA_FAIL();
    half_residual_kernel<<<g2, 128, 0, s>>>(n, wk.Gw2, wk.T); count_launch();
    if (cudaMemcpyAsync(Xn, X, (size_t)n * n * sizeof(double2), cudaMemcpyDeviceToDevice, s) !=
        cudaSuccess)
      return CHASE_CUDA_FAIL();
    Epilogue eo{};
    eo.mode = EPI_FILTER;
    eo.alpha = 1.0;
    eo.beta = 1.0;
    eo.gamma = 0.0;
    eo.X = Xn;
    eo.ldx = n;
    eo.Y = Xn;
    eo.ldy = n;
    if (heev_nn(s, wk, tc, n, X, n, wk.T, eo) != cudaSuccess) return CHASE_CUDA_FAIL();
    std::swap(X, Xn);
  }
  int sw64 = 0;
  bool conv = emax <= 1e-8 && (!tc || fine);
  double2* Zfinal = X;
  double* wsrc = lam;
  bool clustered = false;
  // couplings of pairs left together that are finished: below 64 columns the
  // clusters cost little, and those of a close spectrum add up
  const double cfinish = (n <= BJ_M ? 1e-16 : 1e-14) * gscale;
  if (conv && cmax > cfinish) {
    // pairs the refinement could not separate: FP64 Jacobi on each cluster of
    // them alone (their couplings to every other vector are already at FP64
    // level); falls through to full FP64 sweeps when the clusters are too many
    // or too large for the single-CTA kernel
    int cinfo[2];
    const int rc = cluster_finish(s, n, G, ldg, X, Xn, lam, wk, status, cinfo, cap(kMaxSweeps),
                                  &sw64);
    if (rc < 0) return -rc;
    clustered = rc == 1;
    if (cluster_out) {
      cluster_out[0] = clustered ? 1 : 0;  // finished by the cluster path
      cluster_out[1] = cinfo[0];           // largest cluster
      cluster_out[2] = cinfo[1];           // clusters (or recorded pairs if not used)
    }
  }
  if (!conv || (cmax > cfinish && !clustered)) {
    if (n <= SJ_MAX) {
      const int rc = small_fp64();
      if (sweeps_out) *sweeps_out = sw32 + refine;
      return rc;
    }
    // pairs the refinement could not separate (or no convergence): FP64 Jacobi
    // sweeps on G' = X^H G X finish them; eigenvectors X Z'
    Epilogue ep{};
    ep.mode = EPI_STORE;
    ep.Y = wk.T;
    ep.ldy = n;
    if (zgemm_nn(s, n, n, n, G, ldg, X, n, ep) != cudaSuccess ||
        zgram(s, n, n, n, X, n, wk.T, n, wk.Gw, n, false, wk.gram_ws, wk.gram_ws_elems) !=
            cudaSuccess ||
        hermitian_part(s, n, wk.Gw, n) != cudaSuccess)
      return CHASE_CUDA_FAIL();
    double2* Zrot = Xn;  // the buffer X does not use
    identity_kernel<<<g2, 128, 0, s>>>(n, Zrot); count_launch();
    bool in_g1_64 = false;
    RC_(run_coop<double>(s, n, wk.Gw, wk.Gw2, Zrot, wk.params, wk.red, cap(kMaxSweeps), 1e-15,
                         1e-12, &sw64, &conv, &in_g1_64));
    double2* Gcur = in_g1_64 ? wk.Gw2 : wk.Gw;
    Epilogue ez{};
    ez.mode = EPI_STORE;
    ez.Y = wk.T;
    ez.ldy = n;
    if (zgemm_nn(s, n, n, n, X, n, Zrot, n, ez) != cudaSuccess) return CHASE_CUDA_FAIL();
    Zfinal = wk.T;
    int* rank = reinterpret_cast<int*>(wk.params + 8 * (n / 2 + 2));
    rank_kernel<<<(unsigned)cdiv(n, 128), 128, 0, s>>>(n, Gcur, w, rank); count_launch();
    permute_cols_kernel<<<dim3((unsigned)cdiv(n, 128), (unsigned)n, 1), 128, 0, s>>>(
        n, Zfinal, rank, Z, ldz); count_launch();
    wsrc = nullptr;
  }
  if (wsrc) {
    int* rank = reinterpret_cast<int*>(wk.params + 8 * (n / 2 + 2));
    rank_vec_kernel<<<(unsigned)cdiv(n, 128), 128, 0, s>>>(n, lam, w, rank); count_launch();
    permute_cols_kernel<<<dim3((unsigned)cdiv(n, 128), (unsigned)n, 1), 128, 0, s>>>(
        n, Zfinal, rank, Z, ldz); count_launch();
  }
  if (cudaGetLastError() != cudaSuccess) return CHASE_CUDA_FAIL();
  if (sweeps_out) *sweeps_out = sw32 + sw64 + refine;
  if (fp64_sweeps_out) *fp64_sweeps_out = sw64;
  return conv ? CHASE_OK : CHASE_ERR_HEEV_NOCONV;
}

}  // namespace chase
