// CholeskyQR building blocks (Alg. 3 / Alg. 4): blocked right-looking upper
// Cholesky G = U^H U with the first failing pivot reported like LAPACK POTRF's
// info, and the triangular solve X <- X U^{-1} done per row panel (rows of
// X U^{-1} are independent, so each CTA solves its own rows left to right and
// needs no grid-wide ordering).
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace chase {
namespace {

constexpr int NB = kNB;  // 64
constexpr int FT = 256;  // threads

// Unblocked Cholesky of the kb x kb diagonal block at (k0, k0) and the inverse
// of the resulting upper-triangular block, in the registers of a cluster.
//
// The elimination that turns G into U turns an identity beside it into
// V = U^-H, and the two fit one 64 x 64 array: U on and above the diagonal, V
// below it. Step j subtracts conj(M(j, r)) M(j, c) / p_j from M(r, c) for all
// r > j and c >= r (U) or c <= j (V); rows are divided by their sqrt(p) at the
// end. One SM's FP64 pipe (2 DFMA a clock) takes 85 us for the 87 thousand complex
// multiply-adds (208 us measured with the patches' idle lanes), so the columns go
// to the four CTAs of a cluster, 4 of every 16 each; a thread owns one row of its
// CTA's columns, four entries. The owners of the next row write it into every CTA's
// shared memory, the owner of the next pivot its reciprocal root, and a step ends
// with one cluster barrier (the row buffer alternates): 98 us.
constexpr int PF_C = 4;
__device__ __forceinline__ uint32_t remote_smem(const void* p, unsigned rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a)
               : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

__global__ void __cluster_dims__(PF_C, 1, 1) __launch_bounds__(FT)
    potf2_kernel(double2* G, int64_t ldg, int64_t k0, int kb, double2* dinv_blk, int* info) {
  __shared__ double2 row_s[2][NB];  // raw row j of M, 1 at column j
  __shared__ double rd_s[NB];       // 1 / sqrt(p_j), 0 if p_j is not positive
  if (*info != 0) return;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, rank = blockIdx.x;
  static_assert(FT / 32 * 8 == NB && PF_C * 4 * 4 == NB, "rows by warps, columns by CTAs");
  const int r = warp * 8 + (lane & 7), c0 = 4 * rank + (lane >> 3);
  double2 m[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int c = 16 * b + c0;
    m[b] = (r <= c && c < kb) ? G[(k0 + r) + (k0 + c) * ldg] : make_double2(0.0, 0.0);
  }
  auto publish = [&](int j) {
    if (r != j) return;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int c = 16 * b + c0;
      const double2 v = c == j ? make_double2(1.0, 0.0) : m[b];
      for (unsigned q = 0; q < PF_C; ++q)
        asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(
                         remote_smem(&row_s[j & 1][c], q)),
                     "d"(v.x), "d"(v.y)
                     : "memory");
      if (c == j) {
        const double p = m[b].x, rd = p > 0.0 ? rsqrt(p) : 0.0;  // 0 for NaN too
        for (unsigned q = 0; q < PF_C; ++q)
          asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote_smem(&rd_s[j], q)), "d"(rd)
                       : "memory");
      }
    }
  };
  // 1 / p is no finite number for the smallest subnormal pivots. Blocks with a diagonal
  // that small divide by one root at a time; the others are spared the test, which
  // costs a step 5 % (0.2 ms of a QR with 34 blocks), and keep their rounding.
  const bool tiny = __syncthreads_or(t < kb && G[(k0 + t) * (ldg + 1)].x < 0x1p-900);
  auto eliminate = [&](auto tiny_c) -> bool {
    for (int j = 0; j < kb; ++j) {
      const double rd = rd_s[j];
      if (rd == 0.0) {  // the same in every CTA
        if (rank == 0 && t == 0) *info = (int)(k0 + j + 1);
        return false;
      }
      if (r > j) {
        const double2* w = row_s[j & 1];
        const double2 f = decltype(tiny_c)::value ? cscale(-rd, cscale(rd, conjz(w[r])))
                                                  : cscale(-(rd * rd), conjz(w[r]));
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c = 16 * b + c0;
          if (c >= r || c <= j) cfma(m[b], f, w[c]);
        }
      }
      if (j + 1 < kb) {
        publish(j + 1);
        cluster_sync();
      }
    }
    return true;
  };
  cluster_sync();  // every CTA has started
  publish(0);
  cluster_sync();
  if (!(tiny ? eliminate(std::true_type{}) : eliminate(std::false_type{}))) return;
  const double rd = r < kb ? rd_s[r] : 0.0;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int c = 16 * b + c0;
    const bool in = r < kb && c < kb;
    double2 u = make_double2(0.0, 0.0);  // U(r, c)
    double2 v = make_double2(0.0, 0.0);  // V(r, c) = conj(U^-1(c, r))
    if (in && r == c) {
      u.x = sqrt(m[b].x);
      v.x = rd;
    } else if (in && r < c) {
      u = cscale(rd, m[b]);
    } else if (in) {
      v = cscale(rd, m[b]);
    }
    if (in) G[(k0 + r) + (k0 + c) * ldg] = u;
    dinv_blk[c + r * NB] = conjz(v);
  }
}

// Panel: U(k-block, j) = W^H G(k-block, j), PC columns per CTA (a 64 x 64 block
// per CTA kept at most n / 64 SMs busy), one row and column per thread. 16 blocks of a
// 1072-column Gram: 375 -> 26 us each on average.
constexpr int PC = FT / NB;  // 4
constexpr int PANEL_SMEM = (NB * (NB + 1) + PC * NB) * (int)sizeof(double2);
__global__ void __launch_bounds__(FT)
    panel_kernel(int64_t n, double2* G, int64_t ldg, int64_t k0, int kb, const double2* dinv_blk,
                 const int* info) {
  extern __shared__ double2 sm[];
  double2* Wt = sm;                    // W(l, r) at l (NB + 1) + r
  double2* P = sm + NB * (NB + 1);     // G block, ld NB
  if (*info != 0) return;
  const int t = threadIdx.x, r = t % NB;
  const int64_t c = k0 + kb + (int64_t)blockIdx.x * PC + t / NB;
  const bool in = r < kb && c < n;
  for (int e = t; e < NB * NB; e += FT) Wt[(e % NB) * (NB + 1) + e / NB] = dinv_blk[e];
  P[t] = in ? G[(k0 + r) + c * ldg] : make_double2(0.0, 0.0);
  __syncthreads();
  if (!in) return;
  double2 acc = make_double2(0.0, 0.0);
  const double2* p = P + (t / NB) * NB;
  for (int l = 0; l <= r; ++l) cfma(acc, conjz(Wt[l * (NB + 1) + r]), p[l]);
  G[(k0 + r) + c * ldg] = acc;
}

// Trailing update of upper tiles: G(i, j) -= sum_l conj(U(l, i)) U(l, j),
// l over the k-block rows, k0 + kb <= i <= j (tile-wise upper). 16 x 16 tiles of
// two warps: FP64-bound like the GEMM, and even at n = 128 on many SMs. n = 1072: 333 ->
// 110 us a step on average against 64 x 64 tiles.
constexpr int TB = 16, TT = 64;
__global__ void __launch_bounds__(TT)
    trailing_kernel(int64_t n, double2* G, int64_t ldg, int64_t k0, int kb, const int* info) {
  if (*info != 0) return;
  if (blockIdx.x > blockIdx.y) return;
  __shared__ double2 Ui[TB][NB + 1];
  __shared__ double2 Uj[TB][NB + 1];
  const int t = threadIdx.x, tx = t & 7, ty = t >> 3;
  const int64_t s0 = k0 + kb;
  const int64_t i0 = s0 + (int64_t)blockIdx.x * TB, j0 = s0 + (int64_t)blockIdx.y * TB;
  for (int c = 0; c < TB; ++c) {  // thread t: row t of the k-block
    const bool okl = t < kb;
    Ui[c][t] = (okl && i0 + c < n) ? G[(k0 + t) + (i0 + c) * ldg] : make_double2(0.0, 0.0);
    Uj[c][t] = (okl && j0 + c < n) ? G[(k0 + t) + (j0 + c) * ldg] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  double2 acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b] = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int l = 0; l < kb; ++l) {
    double2 a[2], b[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      a[q] = conjz(Ui[tx + 8 * q][l]);
      b[q] = Uj[ty + 8 * q][l];
    }
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q) cfma(acc[p][q], a[p], b[q]);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int64_t j = j0 + ty + 8 * q;
    if (j >= n) continue;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int64_t i = i0 + tx + 8 * p;
      if (i < n && i <= j) G[i + j * ldg] = csub(G[i + j * ldg], acc[p][q]);
    }
  }
}

// Row-panel triangular solve X <- X U^{-1}. Each CTA owns 64 rows of X and
// walks the 64-column blocks left to right:
//   T = X(rows, jb) - X(rows, 0:jb) U(0:jb, jb);  X(rows, jb) = T W_jb
constexpr int RP = 64, TK = 8;
__global__ void __launch_bounds__(FT)
    trsm_kernel(int64_t m, int64_t n, double2* X, int64_t ldx, const double2* U, int64_t ldu,
                const double2* dinv, const int* info) {
  if (*info != 0) return;
  extern __shared__ double2 sm[];
  double2* Ts = sm;                 // [c'][r]  NB x RP
  double2* Ws = sm + NB * RP;       // [c'][c]  NB x NB
  double2* Xs = Ws + NB * NB;       // [k][r]   TK x RP
  double2* Us = Xs + TK * RP;       // [k][c]   TK x NB
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int64_t r0 = (int64_t)blockIdx.x * RP;
  const int64_t nblk = cdiv(n, NB);
  for (int64_t jb = 0; jb < nblk; ++jb) {
    const int64_t c0 = jb * NB;
    const int cb = (int)min((int64_t)NB, n - c0);
    double2 acc[4][4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t r = r0 + tx + 16 * p, c = ty + 16 * q;
        acc[p][q] = (r < m && c < cb) ? X[r + (c0 + c) * ldx] : make_double2(0.0, 0.0);
      }
    for (int64_t l0 = 0; l0 < c0; l0 += TK) {
      __syncthreads();
      for (int e = t; e < TK * RP; e += FT) {
        const int r = e % RP, k = e / RP;
        const int64_t row = r0 + r;
        Xs[k * RP + r] = (row < m) ? X[row + (l0 + k) * ldx] : make_double2(0.0, 0.0);
      }
      for (int e = t; e < TK * NB; e += FT) {
        const int k = e % TK, c = e / TK;
        Us[k * NB + c] = (c < cb) ? U[(l0 + k) + (c0 + c) * ldu] : make_double2(0.0, 0.0);
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < TK; ++k) {
        double2 a[4], b[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) a[p] = Xs[k * RP + tx + 16 * p];
#pragma unroll
        for (int q = 0; q < 4; ++q) b[q] = Us[k * NB + ty + 16 * q];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            double2& o = acc[p][q];
            o.x = fma(-a[p].x, b[q].x, o.x);
            o.x = fma(a[p].y, b[q].y, o.x);
            o.y = fma(-a[p].x, b[q].y, o.y);
            o.y = fma(-a[p].y, b[q].x, o.y);
          }
      }
    }
    __syncthreads();
    // T -> shared, W_jb -> shared
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) Ts[(ty + 16 * q) * RP + tx + 16 * p] = acc[p][q];
    const double2* Wb = dinv + jb * NB * NB;
    for (int e = t; e < NB * NB; e += FT) {
      const int cp = e % NB, c = e / NB;
      Ws[cp * NB + c] = Wb[cp + c * NB];
    }
    __syncthreads();
    double2 out[4][4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) out[p][q] = make_double2(0.0, 0.0);
    for (int cp = 0; cp < cb; ++cp) {
      double2 a[4], b[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) a[p] = Ts[cp * RP + tx + 16 * p];
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] = Ws[cp * NB + ty + 16 * q];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) cfma(out[p][q], a[p], b[q]);
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t r = r0 + tx + 16 * p;
        const int c = ty + 16 * q;
        if (r < m && c < cb) X[r + (c0 + c) * ldx] = out[p][q];
      }
  }
}

__global__ void trace_shift_kernel(int64_t n, double2* G, int64_t ldg, double factor,
                                   double* scratch) {
  __shared__ double red[256];
  const int t = threadIdx.x;
  double s = 0.0;
  for (int64_t i = t; i < n; i += 256) s += G[i + i * ldg].x;
  red[t] = s;
  __syncthreads();
  for (int w = 128; w >= 1; w >>= 1) {
    if (t < w) red[t] += red[t + w];
    __syncthreads();
  }
  const double shift = factor * red[0];
  if (t == 0) scratch[0] = shift;
  for (int64_t i = t; i < n; i += 256) G[i + i * ldg].x += shift;
}

// Largest of non-negative doubles (NaN counted as +inf) into *out, which holds
// the bit pattern of a non-negative double (monotone in unsigned order): the
// result does not depend on the order of the atomics.
__device__ __forceinline__ void atomic_max_nonneg(double* out, double v) {
  if (!(v <= 1.7976931348623157e308)) v = __longlong_as_double(0x7ff0000000000000ll);
  atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)__double_as_longlong(v));
}

__device__ __forceinline__ double block_max256(double m, double* red) {
  red[threadIdx.x] = m;
  __syncthreads();
  for (int w = 128; w >= 1; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  return red[0];
}

// max over the upper triangle of |U_ij - delta_ij|: one CTA per column
__global__ void __launch_bounds__(256)
    dev_identity_kernel(int64_t n, const double2* __restrict__ U, int64_t ldu,
                        double* __restrict__ out) {
  __shared__ double red[256];
  const int64_t j = blockIdx.x;
  double m = 0.0;
  for (int64_t i = threadIdx.x; i <= j; i += 256) {
    double2 u = U[i + j * ldu];
    if (i == j) u.x -= 1.0;
    m = fmax(m, sqrt(u.x * u.x + u.y * u.y));
  }
  m = block_max256(m, red);
  if (threadIdx.x == 0) atomic_max_nonneg(out, m);
}

// max_j (max_i |R_ij|) / (max_i |X_ij|), |z| = max(|Re z|, |Im z|): one CTA per column
__global__ void __launch_bounds__(256)
    col_ratio_kernel(int64_t m, const double2* __restrict__ R, int64_t ldr,
                     const double2* __restrict__ X, int64_t ldx, double* __restrict__ out) {
  __shared__ double red[256];
  const int64_t j = blockIdx.x;
  double mr = 0.0, mx = 0.0;
  for (int64_t i = threadIdx.x; i < m; i += 256) {
    const double2 r = R[i + j * ldr], x = X[i + j * ldx];
    mr = fmax(mr, fmax(fabs(r.x), fabs(r.y)));
    mx = fmax(mx, fmax(fabs(x.x), fabs(x.y)));
  }
  mr = block_max256(mr, red);
  __syncthreads();
  mx = block_max256(mx, red);
  if (threadIdx.x == 0) atomic_max_nonneg(out, mx > 0.0 ? mr / mx : (mr > 0.0 ? __longlong_as_double(0x7ff0000000000000ll) : 0.0));
}

// strict lower triangle of the n x n M set to zero
__global__ void zero_lower_kernel(int64_t n, double2* __restrict__ M, int64_t ldm) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = blockIdx.y;
  if (i < n && i > j) M[i + j * ldm] = make_double2(0.0, 0.0);
}

// M = I (set) or M -= I (subtract), n x n, ld ldm
__global__ void identity_kernel(int64_t n, double2* __restrict__ M, int64_t ldm, bool subtract) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = blockIdx.y;
  if (i >= n) return;
  if (subtract) {
    if (i == j) M[i + j * ldm].x -= 1.0;
  } else {
    M[i + j * ldm] = make_double2(i == j ? 1.0 : 0.0, 0.0);
  }
}

// kb x kb diagonal-block inverse (ld NB) into the diagonal block of Y (ld ldy)
__global__ void copy_dinv_kernel(int kb, const double2* __restrict__ W, double2* __restrict__ Y,
                                 int64_t ldy) {
  const int r = threadIdx.x, c = blockIdx.x;
  if (r < kb && c < kb) Y[r + (int64_t)c * ldy] = r <= c ? W[r + c * NB] : make_double2(0.0, 0.0);
}

// Y = U^{-1} for the leading n x n block of U (upper triangular, diagonal-block
// inverses in dinv, block b at dinv + b NB^2), recursively:
// inv([[U11, U12], [0, U22]]) = [[Y11, -Y11 U12 Y22], [0, Y22]], split at a
// multiple of NB so the leaves are the stored diagonal-block inverses.
cudaError_t trinv_rec(cudaStream_t s, int64_t n, const double2* U, int64_t ldu,
                      const double2* dinv, double2* Y, int64_t ldy, double2* T) {
  if (n <= NB) {
    copy_dinv_kernel<<<(unsigned)n, NB, 0, s>>>((int)n, dinv, Y, ldy); count_launch();
    return cudaGetLastError();
  }
  const int64_t n1 = cdiv(cdiv(n, 2), NB) * NB, n2 = n - n1;
  cudaError_t e = trinv_rec(s, n1, U, ldu, dinv, Y, ldy, T);
  if (e != cudaSuccess) return e;
  e = trinv_rec(s, n2, U + n1 + n1 * ldu, ldu, dinv + (n1 / NB) * NB * NB, Y + n1 + n1 * ldy,
                ldy, T);
  if (e != cudaSuccess) return e;
  Epilogue ep{};
  ep.mode = EPI_STORE;  // T = U12 Y22 (n1 x n2, ld n1)
  ep.Y = T;
  ep.ldy = n1;
  e = zgemm_nn(s, n1, n2, n2, U + n1 * ldu, ldu, Y + n1 + n1 * ldy, ldy, ep, TRI_B);
  if (e != cudaSuccess) return e;
  Epilogue e2{};
  e2.mode = EPI_FILTER;  // Y12 = -(Y11 T) (beta = 0: the old Y12 is not read)
  e2.alpha = -1.0;
  e2.beta = 0.0;
  e2.gamma = 0.0;
  e2.X = Y + n1 * ldy;
  e2.ldx = ldy;
  e2.Y = Y + n1 * ldy;
  e2.ldy = ldy;
  return zgemm_nn(s, n1, n2, n1, Y, ldy, T, n1, e2, TRI_A);
}

std::once_flag g_attr_once[kMaxDevices];
void set_attrs() {
  once_per_device(g_attr_once, []() {
    cudaFuncSetAttribute(panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PANEL_SMEM);
    cudaFuncSetAttribute(trsm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (NB * RP + NB * NB + TK * RP + TK * NB) * (int)sizeof(double2));
  });
}

}  // namespace

cudaError_t potrf_upper(cudaStream_t s, int64_t n, double2* G, int64_t ldg, double2* dinv,
                        int* info) {
  set_attrs();
  cudaError_t e = cudaMemsetAsync(info, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  for (int64_t k0 = 0, b = 0; k0 < n; k0 += NB, ++b) {
    const int kb = (int)std::min<int64_t>(NB, n - k0);
    potf2_kernel<<<PF_C, FT, 0, s>>>(G, ldg, k0, kb, dinv + b * NB * NB, info); count_launch();
    const int64_t rest = n - k0 - kb;
    if (rest > 0) {
      panel_kernel<<<(unsigned)cdiv(rest, PC), FT, PANEL_SMEM, s>>>(n, G, ldg, k0, kb,
                                                                    dinv + b * NB * NB, info);
      count_launch();
      const unsigned tt = (unsigned)cdiv(rest, TB);
      trailing_kernel<<<dim3(tt, tt, 1), TT, 0, s>>>(n, G, ldg, k0, kb, info); count_launch();
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t trsm_right_upper(cudaStream_t s, int64_t m, int64_t n, double2* X, int64_t ldx,
                             const double2* U, int64_t ldu, const double2* dinv, const int* info) {
  set_attrs();
  if (m <= 0 || n <= 0) return cudaSuccess;
  const size_t smem = (NB * RP + NB * NB + TK * RP + TK * NB) * sizeof(double2);
  trsm_kernel<<<(unsigned)cdiv(m, RP), FT, smem, s>>>(m, n, X, ldx, U, ldu, dinv, info); count_launch();
  return cudaGetLastError();
}

cudaError_t triangular_inverse(cudaStream_t s, int64_t n, const double2* U, int64_t ldu,
                               const double2* dinv, double2* Y, int64_t ldy, double2* T) {
  if (n <= 0) return cudaSuccess;
  cudaError_t e = cudaMemset2DAsync(Y, ldy * sizeof(double2), 0, n * sizeof(double2), n, s);
  if (e != cudaSuccess) return e;
  return trinv_rec(s, n, U, ldu, dinv, Y, ldy, T);
}

cudaError_t max_dev_identity(cudaStream_t s, int64_t n, const double2* U, int64_t ldu,
                             double* out) {
  if (n <= 0) return cudaMemsetAsync(out, 0, sizeof(double), s);
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), s);
  if (e != cudaSuccess) return e;
  dev_identity_kernel<<<(unsigned)n, 256, 0, s>>>(n, U, ldu, out); count_launch();
  return cudaGetLastError();
}

cudaError_t max_col_ratio(cudaStream_t s, int64_t m, int64_t n, const double2* R, int64_t ldr,
                          const double2* X, int64_t ldx, double* out) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), s);
  if (e != cudaSuccess || m <= 0 || n <= 0) return e;
  col_ratio_kernel<<<(unsigned)n, 256, 0, s>>>(m, R, ldr, X, ldx, out); count_launch();
  return cudaGetLastError();
}

cudaError_t zero_lower(cudaStream_t s, int64_t n, double2* M, int64_t ldm) {
  if (n <= 1) return cudaSuccess;
  zero_lower_kernel<<<dim3((unsigned)cdiv(n, 128), (unsigned)n, 1), 128, 0, s>>>(n, M, ldm);
  count_launch();
  return cudaGetLastError();
}

cudaError_t set_identity(cudaStream_t s, int64_t n, double2* M, int64_t ldm, bool subtract) {
  identity_kernel<<<dim3((unsigned)cdiv(n, 128), (unsigned)n, 1), 128, 0, s>>>(n, M, ldm, subtract);
  count_launch();
  return cudaGetLastError();
}

cudaError_t add_trace_shift(cudaStream_t s, int64_t n, double2* G, int64_t ldg, double factor,
                            double* scratch) {
  trace_shift_kernel<<<1, 256, 0, s>>>(n, G, ldg, factor, scratch); count_launch();
  return cudaGetLastError();
}

}  // namespace chase
