// Birkhoff products B v and B^T v on the CGL grid (FastBV and its transpose).
//
// Paper: "Fast Computation of Birkhoff Matrix-Vector Products" (Eqs. vi=sumT .. chatk=,
// algorithms Fasta2v / FastBV) and Appendix B (Fastv2a).
//
// Formulation used by the kernels. Let R be the unnormalised type-I DCT of length N+1,
//   R(x)_k = x_0 + (-1)^k x_N + 2 sum_{m=1}^{N-1} x_m cos(pi k m / N),
// which is twice the paper's DCT-I (Eq. vm=DCT-1). Write Y = R(v). The Chebyshev coefficients
// of Fastv2a are a_k = (-1)^k h_k Y_k / N (h = 1/2 at k = 0, N), and the sign (-1)^k that the
// reversal steps of Fastv2a / Fasta2v introduce cancels inside the integration stencil of
// Eq. c_k=bydef, so with chat'_k = (-1)^k chat_k:
//   chat'_1     = (Y_2 - Y_0) / (2N)
//   chat'_k     = (Y_{k+1} - Y_{k-1}) / (2kN),                 2 <= k <= N-2
//   chat'_{N-1} = (Y_N/2 - Y_{N-2}) / (2(N-1)N) - (Y_N/2) / (2(N+1)N)   (aliasing fold, Eq. chatk=)
//   chat'_N     = -Y_{N-1} / (2N^2)
// and the nodal values are y'_i = sum_k chat'_k cos(pi k i / N) = R(g)_i with g_0 = 0,
// g_k = chat'_k / 2 (0 < k < N), g_N = chat'_N. The constant coefficient c_0 is not formed:
// row 0 of B^a is zero (B^a_j(tau^a) = 0, Eq. birk-conditions), and c_0 multiplies T_0 = 1,
// so B^a v = y' - y'_0. With the time scale s = (tf - t0)/2:  B v = s (y' - y'_0 1).
// Transpose: B = s (I - 1 e_0^T) R G R / N with R = C W (C symmetric, W = diag(1,2,..,2,1)),
// so B^T u = (s/N) W R W^{-1} G^T W R W^{-1} (I - e_0 1^T) u, and R W^{-1} (I - e_0 1^T) u =
// R(W^{-1} u) - (sum u) 1 because column 0 of R is all ones and sum_m (W^{-1}u)_ext = sum u.
//
// The DCT-I is computed by a complex FFT of length N of z_j = x_ext[2j] + i x_ext[2j+1]
// (x_ext the even 2N-periodic extension of x) and the standard real-FFT split:
//   Y_k = P + Q,  Y_{N-k} = P - Q,  P = Re(Z_k + Z_{N-k}) / 2,
//   Q = [cos(pi k/N) Im(Z_k + Z_{N-k}) - sin(pi k/N) Re(Z_k - Z_{N-k})] / 2.
// N <= NSMALL: one CTA per vector does the whole chain in shared memory (one HBM read and one
// write) with that FFT. Larger powers of two: the real-even four-step DFT of bk_dct.cuh in two
// passes per DCT, the integration stencil fused into the load of the second DCT.
#include <math.h>
#include <stdarg.h>
#include <stdlib.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>
#include <string>
#include <vector>

#include "bk_common.cuh"
#include "bk_fft.cuh"
#include "bk_plan.cuh"

namespace bk {

// The kernels compute in T and keep their internal real vectors (the stage buffers between the
// two DCTs) in T; the caller's vectors are User<T> (binary64 for double-float arithmetic, whose
// products convert the input in the first pass's loads and the output in the last pass's stores).
template <typename T> using Us = typename User<T>::t;
// Conversion of a stored element S to the arithmetic type T and back (identity when S == T).
template <typename T, typename S> struct Cv;
template <typename T> struct Cv<T, T> {
  static __device__ __forceinline__ T in(T x) { return x; }
  static __device__ __forceinline__ T out(T x) { return x; }
};
template <> struct Cv<dfl, double> {
  static __device__ __forceinline__ dfl in(double x) { return d2df(x); }
  static __device__ __forceinline__ double out(dfl x) { return df2d(x); }
};
template <typename T, typename S> __device__ __forceinline__ T rdv(const S* __restrict__ p, int64_t i) {
  return Cv<T, S>::in(p[i]);
}

#ifndef BK_TRANSFORM_KERNEL_UNIT  // one definition of the library's globals, in the main unit
// (bk_birkhoff_f64.cu and bk_birkhoff_f32.cu include this file for the transform kernels only)
static thread_local std::string g_last_error = "no error";
static std::atomic<unsigned long long> g_launches{0};
// When set (by the creating thread), dmalloc adds every allocation's size to it: plans and
// problems report their device footprint this way.
static thread_local size_t* g_alloc_acc = nullptr;

AllocCounter::AllocCounter(size_t* acc) : prev(g_alloc_acc) { g_alloc_acc = acc; }
AllocCounter::~AllocCounter() { g_alloc_acc = prev; }

static thread_local unsigned long long t_launches = 0;
void note_launch() {
  g_launches.fetch_add(1, std::memory_order_relaxed);
  ++t_launches;
}
unsigned long long thread_launches() { return t_launches; }
void note_launches(long long n) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }

void set_error(const char* fmt, ...) {
  char buf[1024];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_last_error = buf;
}

bk_status dmalloc(void** p, size_t bytes) {
  *p = nullptr;
  if (bytes == 0) return BK_OK;
  if (g_alloc_acc) *g_alloc_acc += bytes;
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    *p = nullptr;
    set_error("cudaMalloc(%zu bytes): %s", bytes, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? BK_ERR_OOM : BK_ERR_CUDA;
  }
  return BK_OK;
}

void dfree(void* p) {
  if (p) cudaFree(p);
}

#endif  // BK_TRANSFORM_KERNEL_UNIT

// ---------------------------------------------------------------------------------------------
// Table construction (device, FP64 sincospi; FP32 tables are rounded copies)
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void k_tw_table(typename V2<T>::t* tw, int64_t n, double denom_half_turns) {
  // tw[i] = (cos(2 pi i / n), -sin(2 pi i / n)) computed as sincospi(2 i / n)
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s, c;
    sincospi((double)(2 * i) / denom_half_turns, &s, &c);
    tw[i] = mk2<T>((T)c, (T)(-s));
  }
}

// tw[i] = omega_n^{i * stride}, i < count (sincospi of 2 i stride / n)
template <typename T>
__global__ void k_tw_table_strided(typename V2<T>::t* tw, int64_t count, int64_t stride, double n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    double s, c;
    sincospi((double)(2 * i * stride) / n, &s, &c);
    tw[i] = mk2<T>((T)c, (T)(-s));
  }
}

template <typename T>
__global__ void k_post_table(typename V2<T>::t* tp, int64_t N) {
  // tp[k] = (cos(pi k / N), sin(pi k / N)), k = 0..N/2
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k <= N / 2;
       k += (int64_t)gridDim.x * blockDim.x) {
    double s, c;
    sincospi((double)k / (double)N, &s, &c);
    tp[k] = mk2<T>((T)c, (T)s);
  }
}

// Stage twiddle table of a length-2^log2n FFT of radix R = 2^e (see bk_fft.cuh): entry
// off + (r-1) Ns + k of the block of the stage with Ns = 2^l is omega_{R Ns}^{r k}, from
// sincospi(2 r k / (R Ns)).
template <typename T>
__global__ void k_stage_tw(typename V2<T>::t* stw, int log2n, int e, int len) {
  const int R1 = (1 << e) - 1;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < len; idx += gridDim.x * blockDim.x) {
    int l = log2n % e ? log2n % e : e, off = 0;
    while (idx >= off + (R1 << l)) { off += R1 << l; l += e; }
    const int i = idx - off;
    const int r = (i >> l) + 1, k = i & ((1 << l) - 1);
    double sn, cs;
    sincospi((double)(2 * r * k) / (double)(1 << (l + e)), &sn, &cs);
    stw[idx] = mk2<T>((T)cs, (T)(-sn));
  }
}

// Twiddles of one mixed-radix stage: stw[(r - 1) Ns + k] = omega_{R Ns}^{r k}.
template <typename T>
__global__ void k_mix_tw(typename V2<T>::t* stw, int Ns, int R) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < (R - 1) * Ns; i += gridDim.x * blockDim.x) {
    const int r = i / Ns + 1, k = i % Ns;
    double sn, cs;
    sincospi((double)(2 * r * k) / (double)(R * Ns), &sn, &cs);
    stw[i] = mk2<T>((T)cs, (T)(-sn));
  }
}

// Inter-pass twiddles of the real-even passes, [N1/2 + 1][N2/2 + 2] (2N = N1 N2; see bk_dct.cuh):
// omega_2N^{n2 k} / 2 for a pair's first column (even positions; position 0 is column 0), times -i
// for its second (odd positions; position 1 is column N2/2).
template <typename T>
__global__ void k_re_tw(typename V2<T>::t* tw, int N1, int N2) {
  const int RS = N2 / 2 + 2;
  const int64_t len = (int64_t)(N1 / 2 + 1) * RS;
  const double N = 0.5 * (double)N1 * (double)N2;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = i / RS;
    const int pos = (int)(i - k * RS);
    const int64_t n2 = pos == 0 ? 0 : (pos == 1 ? N2 / 2 : pos - 1);
    double sn, cs;
    sincospi((double)(n2 * k) / N, &sn, &cs);
    tw[i] = (pos & 1) ? mk2<T>((T)(-0.5 * sn), (T)(-0.5 * cs)) : mk2<T>((T)(0.5 * cs), (T)(-0.5 * sn));
  }
}

// rk[k] = 1 / (4k), k >= 1 (rk[0] = 0), rounded once from FP64.
template <typename T>
__global__ void k_rk_table(T* rk, int64_t n) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    rk[k] = k == 0 ? T(0) : (T)(1.0 / (4.0 * (double)k));
}

// Bluestein chirp w_j = exp(-i pi j^2 / N) = (cos, -sin)(pi r / N), r = j^2 mod 2N in integers.
template <typename T>
__global__ void k_chirp(typename V2<T>::t* w, int64_t N) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = (j * j) % (2 * N);
    double sn, cs;
    sincospi((double)r / (double)N, &sn, &cs);
    w[j] = mk2<T>((T)cs, (T)(-sn));
  }
}

// The convolution kernel b of Bluestein's identity, scaled by 1/M, as M complex values (real
// pairs): b_m = conj(w_m) for m < N, b_{M-m} = conj(w_m) for 0 < m < N, zero between.
template <typename T>
__global__ void k_bs_kernel(T* b, int64_t N, int64_t M) {
  for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M; m += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = m < N ? m : (m > M - N ? M - m : -1);
    double sn = 0.0, cs = 0.0;
    if (j >= 0) sincospi((double)((j * j) % (2 * N)) / (double)N, &sn, &cs);
    b[2 * m] = (T)(cs / (double)M);
    b[2 * m + 1] = (T)(sn / (double)M);
  }
}

#ifndef BK_TRANSFORM_KERNEL_UNIT
__global__ void k_grid_tables(double* t_nodes, int64_t N, double t0, double s) {
  // tau_j = -cos(j pi / N) = sin(pi (2j - N) / (2N)) (Eq. CGLpts), t_j = t0 + s (tau_j + 1)
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j <= N;
       j += (int64_t)gridDim.x * blockDim.x) {
    double tau = sinpi((double)(2 * j - N) / (double)(2 * N));
    if (j == 0) tau = -1.0;
    if (j == N) tau = 1.0;
    t_nodes[j] = t0 + s * (tau + 1.0);
  }
}
#endif  // BK_TRANSFORM_KERNEL_UNIT

// ---------------------------------------------------------------------------------------------
// Element accessors of the transform inputs
// ---------------------------------------------------------------------------------------------
// Kinds of the first-DCT input x:
//   IN_PLAIN : x_m = v_m                  (forward product)
//   IN_WINV  : x_m = v_m / W_m            (transpose product; W = 1 at the ends, 2 inside)
// Kinds of the second-DCT input (from Y = output of the first DCT):
//   ST_FWD   : x_m = g_m = G(Y)_m                          (forward stencil, includes 1/N)
//   ST_TRN   : x_m = W_m^{-1} G^T(W (Y - Y_0))_m          (transposed stencil)
enum { IN_PLAIN = 0, IN_WINV = 1, ST_FWD = 2, ST_TRN = 3 };

// rk[k] = 1 / (4k) for 1 <= k <= N + 1 (plan table): the stencils multiply instead of divide.
template <typename T, typename S>
__device__ __forceinline__ T stencil_fwd(const S* __restrict__ Y, int m, int N, T invN, const T* __restrict__ rk) {
  // g_m = chat'_m / 2 for 0 < m < N, g_N = chat'_N, g_0 = 0 (see the file comment). invN is 1/N,
  // or 1 where Y was stored already divided by N.
  if (m == 0) return T(0);
  if (m == N) return -rdv<T>(Y, N - 1) * (invN * T(2) * rk[N]);
  if (m == 1) return (rdv<T>(Y, 2) - rdv<T>(Y, 0)) * (invN * T(0.25));
  if (m == N - 1) {
    const T yN = rdv<T>(Y, N);
    return (T(0.5) * yN - rdv<T>(Y, N - 2)) * (invN * rk[N - 1]) - yN * (invN * T(0.5) * rk[N + 1]);
  }
  return (rdv<T>(Y, m + 1) - rdv<T>(Y, m - 1)) * (invN * rk[m]);
}

template <typename T, typename S>
__device__ __forceinline__ T stencil_trn(const S* __restrict__ Qs, int m, int N, T Y0, const T* __restrict__ rk,
                                         T cN) {
  auto Q = [&](int i) { return rdv<T>(Qs, i); };
  // r = W (Y - Y0); t = G^T r; return t_m / W_m. G^T rows:
  //   t_0 = -r_1/4, t_1 = -r_2/8, t_j = r_{j-1}/(4(j-1)) - r_{j+1}/(4(j+1)) (2<=j<=N-2),
  //   t_{N-1} = r_{N-2}/(4(N-2)) - r_N/(2N), t_N = r_{N-1}/(4(N^2-1)).
  // r_k = 2 (Y_k - Y0) for 0 < k < N, r_0 = Y_0 - Y0 = 0, r_N = Y_N - Y0.
  // cN = 1 / (4 (N^2 - 1))
  if (m == 0) return -(T(2) * (Q(1) - Y0)) * T(0.25);
  if (m == N) return (T(2) * (Q(N - 1) - Y0)) * cN;
  T t;
  if (m == 1) {
    t = -(T(2) * (Q(2) - Y0)) * T(0.125);
  } else if (m == N - 1) {
    t = (T(2) * (Q(N - 2) - Y0)) * rk[N - 2] - (Q(N) - Y0) * (T(2) * rk[N]);
  } else {
    t = (Q(m - 1) - Y0) * rk[m - 1] - (Q(m + 1) - Y0) * rk[m + 1];
    return t;
  }
  return T(0.5) * t;
}

// Value x_m of the transform input of kind K. `src` is the vector (first DCT) or the stage
// buffer Y (second DCT). Y0 is used by ST_TRN only.
// Stencil constants passed to the transform kernels.
template <typename T> struct StencilTab {
  const T* rk;  // rk[k] = 1/(4k), k = 1..N+1
  T cN;         // 1/(4(N^2 - 1))
};

template <typename T, int K, typename S>
__device__ __forceinline__ T load_x(const S* __restrict__ src, int m, int N, T invN, T Y0, StencilTab<T> tb) {
  if (K == IN_PLAIN) return rdv<T>(src, m);
  if (K == IN_WINV) return (m == 0 || m == N) ? rdv<T>(src, m) : T(0.5) * rdv<T>(src, m);
  if (K == ST_FWD) return stencil_fwd<T>(src, m, N, invN, tb.rk);
  return stencil_trn<T>(src, m, N, Y0, tb.rk, tb.cN);
}

// z_j = x_ext[2j] + i x_ext[2j+1]
template <typename T, int K, typename S>
__device__ __forceinline__ typename V2<T>::t load_z(const S* __restrict__ src, int j, int N, T invN,
                                                    T Y0, StencilTab<T> tb) {
  const int m1 = 2 * j, m2 = 2 * j + 1;
  const int i1 = m1 <= N ? m1 : 2 * N - m1;
  const int i2 = m2 <= N ? m2 : 2 * N - m2;
  return mk2<T>(load_x<T, K>(src, i1, N, invN, Y0, tb), load_x<T, K>(src, i2, N, invN, Y0, tb));
}

// Real-FFT split: from Z_k, Z_{N-k} and (cos, sin)(pi kk / N), kk = min(k, N - k).
template <typename T>
__device__ __forceinline__ void split_pair(typename V2<T>::t zk, typename V2<T>::t zc,
                                           typename V2<T>::t cs, T& yk, T& ynk) {
  const T P = T(0.5) * (zk.x + zc.x);
  const T Q = T(0.5) * (cs.x * (zk.y + zc.y) - cs.y * (zk.x - zc.x));
  yk = P + Q;
  ynk = P - Q;
}

// ---------------------------------------------------------------------------------------------
// Single-CTA fused kernel: the whole chain for one vector in shared memory.
// ---------------------------------------------------------------------------------------------
template <typename T>
__device__ void dct1_block(const T* __restrict__ X, int kind, T* __restrict__ Y,
                           typename V2<T>::t* buf, int N, int log2N,
                           const typename V2<T>::t* __restrict__ tw, const typename V2<T>::t* __restrict__ stw,
                           const typename V2<T>::t* __restrict__ tpost, T invN, T Y0, StencilTab<T> tb) {
  typedef typename V2<T>::t C;
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    C z;
    switch (kind) {
      case IN_PLAIN: z = load_z<T, IN_PLAIN>(X, j, N, invN, Y0, tb); break;
      case IN_WINV: z = load_z<T, IN_WINV>(X, j, N, invN, Y0, tb); break;
      case ST_FWD: z = load_z<T, ST_FWD>(X, j, N, invN, Y0, tb); break;
      default: z = load_z<T, ST_TRN>(X, j, N, invN, Y0, tb); break;
    }
    buf[padi(j)] = z;
  }
  __syncthreads();
  if (N >= 16) {
    fft_any<T, SmallFft<T>::E, SmallFft<T>::EPT, 4, sizeof(T) == 8 ? 9 : 12>(buf, log2N, 1, pad_stride(N), stw);
  } else {
    // N = 4 or 8: direct DFT (tw holds omega_N^i, n_tab = N)
    C zk = mk2<T>(T(0), T(0));
    const int k = threadIdx.x;
    if (k < N) {
      for (int j = 0; j < N; ++j) zk = cadd(zk, cmul(buf[padi(j)], tw[(j * k) & (N - 1)]));
    }
    __syncthreads();
    if (k < N) buf[padi(k)] = zk;
    __syncthreads();
  }
  for (int k = threadIdx.x; k <= N / 2; k += blockDim.x) {
    const C zk = buf[padi(k)];
    const C zc = buf[padi((N - k) & (N - 1))];
    T yk, ynk;
    split_pair<T>(zk, zc, tpost[k], yk, ynk);
    Y[k] = yk;
    if (k != N / 2) Y[N - k] = ynk;
  }
  __syncthreads();
}

// Element loads each thread keeps in flight in the pass kernels' load phases.
// FP32: 8 (latency-bound passes; 16 spilled under the 64-register cap of two 512-thread CTAs
// per SM), FP64: 4 (FP64-pipe-bound, register-heavy).
template <typename T> struct InFlight { static constexpr int v = sizeof(T) == 8 ? 4 : 8; };

// Whole chain for vector vec in one CTA (every value independent of the CTA's thread count, so
// a batched launch with more threads gives the same results).
template <typename T, bool TRANS>
__device__ __forceinline__ void small_body(int vec, const Us<T>* __restrict__ in, Us<T>* __restrict__ out, int N,
                                           int log2N, int64_t pitch, T s, const typename V2<T>::t* __restrict__ tw,
                                           const typename V2<T>::t* __restrict__ stw,
                                           const typename V2<T>::t* __restrict__ tpost, StencilTab<T> tb) {
  typedef typename V2<T>::t C;
  extern __shared__ __align__(16) unsigned char smem[];
  const int L = N + 1;
  const int Lp = (L + 3) & ~3;
  T* X = reinterpret_cast<T*>(smem);
  T* Y = X + Lp;
  C* buf = reinterpret_cast<C*>(Y + Lp);
  const int64_t base = (int64_t)vec * pitch;
  const Us<T>* src = in + base;
  Us<T>* dst = out + base;
  typedef Cv<T, Us<T>> CV;
  const T invN = T(1.0 / (double)N);
  for (int m = threadIdx.x; m < L; m += blockDim.x) X[m] = CV::in(src[m]);
  __syncthreads();
  if (!TRANS) {
    dct1_block<T>(X, IN_PLAIN, Y, buf, N, log2N, tw, stw, tpost, invN, T(0), tb);
    dct1_block<T>(Y, ST_FWD, X, buf, N, log2N, tw, stw, tpost, invN, T(0), tb);
    const T y0 = X[0];
    for (int m = threadIdx.x; m < L; m += blockDim.x) dst[m] = CV::out(s * (X[m] - y0));
  } else {
    dct1_block<T>(X, IN_WINV, Y, buf, N, log2N, tw, stw, tpost, invN, T(0), tb);
    const T y0 = Y[0];
    dct1_block<T>(Y, ST_TRN, X, buf, N, log2N, tw, stw, tpost, invN, y0, tb);
    const T sN = s * invN;
    for (int m = threadIdx.x; m < L; m += blockDim.x)
      dst[m] = CV::out((m == 0 || m == N) ? sN * X[m] : T(2) * sN * X[m]);
  }
  for (int m = L + threadIdx.x; m < pitch; m += blockDim.x) dst[m] = Us<T>(0);
}

template <typename T, bool TRANS>
__global__ void __launch_bounds__(sizeof(T) == 8 ? 256 : 1024)
    k_birkhoff_small(const Us<T>* __restrict__ in, Us<T>* __restrict__ out, int N, int log2N, int64_t pitch,
                     T s, const typename V2<T>::t* __restrict__ tw, const typename V2<T>::t* __restrict__ stw,
                     const typename V2<T>::t* __restrict__ tpost, StencilTab<T> tb) {
  pdl_wait();
  small_body<T, TRANS>(blockIdx.x, in, out, N, log2N, pitch, s, tw, stw, tpost, tb);
}

// ---------------------------------------------------------------------------------------------
// Four-step passes of a plain complex FFT of length n = N1 N2 (Bluestein's convolution; j = N2 j1 +
// j2, k = k1 + N1 k2). Pass A: per CTA, NB columns j2; FFT over j1 (length N1), twiddle
// omega_n^{j2 k1}; writes A[k1][j2]. Pass B: per CTA, 2P rows k1; FFT over j2 (length N2); writes
// the outputs in natural order.
// ---------------------------------------------------------------------------------------------
template <typename T, typename F>
__global__ void __launch_bounds__(F::MT, F::MINB)
    k_passA(const T* __restrict__ src, int64_t src_stride, typename V2<T>::t* __restrict__ Aout, int N, int N1,
            int log2N1, int N2, int NB, int bs, const typename V2<T>::t* __restrict__ stw,
            const typename V2<T>::t* __restrict__ twN, const typename V2<T>::t* __restrict__ twLo,
            const typename V2<T>::t* __restrict__ twHi, int tw_h) {
  pdl_wait();
  typedef typename V2<T>::t C;
  extern __shared__ __align__(16) unsigned char smem[];
  C* buf = reinterpret_cast<C*>(smem);
  // FP32: sub-FFT twiddles in shared memory after the tile (FP64 reads the global table)
  C* tws = buf + (size_t)NB * bs;
  const bool smem_tw = sizeof(T) == 4;
  if (smem_tw) load_tw_smem<T>(tws, stw, stage_tw_len(log2N1, F::E));
  const int vec = blockIdx.y;
  const C* x = reinterpret_cast<const C*>(src + (int64_t)vec * src_stride);
  const int c0 = blockIdx.x * NB;
  const int log2NB = __ffs(NB) - 1, log2N2 = __ffs(N2) - 1;  // NB, N2 are powers of two
  const int total = NB * N1;
  // independent element loads in flight per thread before the shared-memory stores
  constexpr int LD = InFlight<T>::v;
  for (int idx0 = threadIdx.x; idx0 < total; idx0 += LD * blockDim.x) {
    C z[LD];
#pragma unroll
    for (int u = 0; u < LD; ++u) {
      const int idx = idx0 + u * blockDim.x;
      if (idx < total) z[u] = x[((idx >> log2NB) << log2N2) + c0 + (idx & (NB - 1))];
    }
#pragma unroll
    for (int u = 0; u < LD; ++u) {
      const int idx = idx0 + u * blockDim.x;
      if (idx < total) buf[(idx & (NB - 1)) * bs + padi(idx >> log2NB)] = z[u];
    }
  }
  __syncthreads();
  fft_any<T, F::E, F::EPT>(buf, log2N1, NB, bs, smem_tw ? tws : stw);
  C* A = Aout + (int64_t)vec * N;
  // inter-pass twiddles omega_N^{j2 k1}, 4 independent table loads in flight per thread.
  // FP64: one table of omega_N^m (the FP64 pipe, not memory, bounds these kernels).
  // FP32: omega_N^m = omega_N^{(m >> h) 2^h} omega_N^{m mod 2^h} from two tables of ~sqrt N.
  for (int idx0 = threadIdx.x; idx0 < total; idx0 += 4 * blockDim.x) {
    C w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = idx0 + u * blockDim.x;
      if (idx < total) {
        const int m = (c0 + (idx & (NB - 1))) * (idx >> log2NB);  // < N
        w[u] = sizeof(T) == 8 ? ldg(&twN[m]) : cmul(ldg(&twHi[m >> tw_h]), ldg(&twLo[m & ((1 << tw_h) - 1)]));
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = idx0 + u * blockDim.x;
      if (idx < total) {
        const int b = idx & (NB - 1);
        const int k1 = idx >> log2NB;
        A[(int64_t)k1 * N2 + c0 + b] = cmul(buf[b * bs + padi(k1)], w[u]);
      }
    }
  }
}

// Second-DCT input of a Bluestein product as its own elementwise pass: x_m of kind K (ST_FWD with
// scale sc, or ST_TRN with Y0 = 0) for every m <= N, written to G.
template <typename T, int K>
__global__ void __launch_bounds__(256) k_stencil(const T* __restrict__ stage, int64_t Ls, T* __restrict__ G, int N, T sc,
                                                 StencilTab<T> tb) {
  pdl_wait();
  const T* Y = stage + (int64_t)blockIdx.y * Ls;
  T* g = G + (int64_t)blockIdx.y * Ls;
  // interior nodes 2..N-2 by the plain three-point formulas (the boundary cases, if-converted
  // into the same loop, tripled its FP64 instructions); the four boundary nodes by one thread
  const T* __restrict__ rk = tb.rk;
  for (int m = 2 + blockIdx.x * blockDim.x + threadIdx.x; m <= N - 2; m += gridDim.x * blockDim.x) {
    const T ym = Y[m - 1], yp = Y[m + 1];
    g[m] = K == ST_FWD ? (yp - ym) * (sc * rk[m]) : ym * rk[m - 1] - yp * rk[m + 1];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int mb[4] = {0, 1, N - 1, N};
    for (int i = 0; i < 4; ++i) g[mb[i]] = load_x<T, K>(Y, mb[i], N, sc, T(0), tb);
  }
}

// Epilogue kinds of a DCT-I's outputs R_k:
//   EP_STORE     : stage[k] = R_k / N                      (after the first DCT, forward)
//   EP_STORE_TRN : stage of the transposed product         (after the first DCT, transpose)
//   EP_FWD_OUT   : out[k] = s (R_k - R_0)                  (after the second DCT, forward)
//   EP_TRN_OUT   : out[k] = (s/N) W_k R_k                  (after the second DCT, transpose)
// and of the plain complex FFT's pass B:
//   EP_CPLX      : dst[k] = Z_k
//   EP_CPLX_MC   : dst[k] = conj(Z_k tab[k])             (spectral product, conjugated)
enum { EP_STORE = 0, EP_STORE_TRN = 1, EP_FWD_OUT = 2, EP_TRN_OUT = 3, EP_CPLX = 4, EP_CPLX_MC = 5 };

template <typename T, int E, typename S>
__device__ __forceinline__ void ep_write(S* __restrict__ dst, int k, T yk, int N, T s, T Y0, T invN) {
  typedef Cv<T, S> CV;
  if (E == EP_STORE) dst[k] = CV::out(yk * invN);
  else if (E == EP_STORE_TRN) dst[k] = CV::out(yk - Y0);
  else if (E == EP_FWD_OUT) dst[k] = CV::out(s * (yk - Y0));
  else dst[k] = CV::out((k == 0 || k == N) ? s * invN * yk : T(2) * s * invN * yk);
}

}  // namespace bk

#include "bk_dct.cuh"

namespace bk {

// ---------------------------------------------------------------------------------------------
// N that is not a power of two (N > 1024): Bluestein's identity j k = (j^2 + k^2 - (k - j)^2)/2
// turns the length-N complex DFT Z = DFT_N(z) of the DCT-I into a circular convolution of
// length M (a power of two, M >= 2N - 1), run by the four-step FFT passes above in their plain
// complex modes:
//   a_j = z_j w_j (j < N, 0 up to M),  w_j = e^{-i pi j^2 / N} (j^2 reduced mod 2N in integers),
//   c = IFFT_M(FFT_M(a) . Bh),  Bh = FFT_M(b) / M,  b_m = conj(w_m) = b_{M-m} (|m| < N, else 0),
//   Z_k = w_k c_k.
// The inverse FFT runs as conj(FFT(conj .)): the first FFT's pass B stores conj(A . Bh), the
// second FFT is a forward one, and the post kernel takes conj of its output. Then the real-FFT
// split gives the DCT-I outputs Y_k (k = 0..N) as for powers of two, with Y_0 = Re Z_0 + Im Z_0.
// ---------------------------------------------------------------------------------------------
// a = z w zero-padded to M (one complex per element), z_j from the input kind K (IN_PLAIN / IN_WINV).
template <typename T, int K>
__global__ void __launch_bounds__(256) k_bs_pre(const T* __restrict__ src, int64_t sstride, int N, int64_t M,
                                                const typename V2<T>::t* __restrict__ w, T* __restrict__ a) {
  pdl_wait();
  typedef typename V2<T>::t C;
  const T* x = src + (int64_t)blockIdx.y * sstride;
  T* dst = a + (int64_t)blockIdx.y * 2 * M;
  StencilTab<T> tb;
  tb.rk = nullptr;
  tb.cN = T(0);
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < M; j += (int64_t)gridDim.x * blockDim.x) {
    C r = mk2<T>(T(0), T(0));
    if (j < N) r = cmul(load_z<T, K>(x, (int)j, N, T(1), T(0), tb), w[j]);
    dst[2 * j] = r.x;
    dst[2 * j + 1] = r.y;
  }
}

// DCT-I outputs from the second FFT's output y (M complex per vector): Z_k = w_k conj(y_k), the
// real-FFT split of (Z_k, Z_{N-k}) for k <= N/2, and the epilogue E (Y0 = Y_0 = Re Z_0 + Im Z_0).
template <typename T, int E>
__global__ void __launch_bounds__(256) k_bs_post(const T* __restrict__ y, int64_t M, int N,
                                                 const typename V2<T>::t* __restrict__ w,
                                                 const typename V2<T>::t* __restrict__ tpost,
                                                 T* __restrict__ dst, int64_t dstride,
                                                 int64_t zero_to, T s, T invN) {
  pdl_wait();
  typedef typename V2<T>::t C;
  const T* yv = y + (int64_t)blockIdx.y * 2 * M;
  T* out = dst + (int64_t)blockIdx.y * dstride;
  auto Z = [&](int k) {  // w_k conj(y_k)
    const C yk = mk2<T>(yv[2 * (int64_t)k], -yv[2 * (int64_t)k + 1]);
    return cmul(w[k], yk);
  };
  const C z0 = Z(0);
  const T Y0 = z0.x + z0.y;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= N / 2; k += gridDim.x * blockDim.x) {
    const int kc = k == 0 ? 0 : N - k;
    T yk, ynk;
    split_pair<T>(Z(k), Z(kc), tpost[k], yk, ynk);
    ep_write<T, E>(out, k, yk, N, s, Y0, invN);
    if (N - k != k) ep_write<T, E>(out, N - k, ynk, N, s, Y0, invN);
  }
  if ((E == EP_FWD_OUT || E == EP_TRN_OUT) && blockIdx.x == 0) {
    for (int64_t m = N + 1 + threadIdx.x; m < zero_to; m += blockDim.x) out[m] = T(0);
  }
}

// Pass B of the plain complex FFT: outputs as complex pairs in natural order; EP_CPLX_MC multiplies
// by the spectral table and conjugates.
template <typename T, int E, typename F>
__global__ void __launch_bounds__(F::MT, F::MINB)
    k_passB(const typename V2<T>::t* __restrict__ Ain, T* __restrict__ dst, int64_t dst_stride, int N, int N1, int N2,
            int log2N2, int P, const typename V2<T>::t* __restrict__ stw, const typename V2<T>::t* __restrict__ tab) {
  pdl_wait();
  typedef typename V2<T>::t C;
  extern __shared__ __align__(16) unsigned char smem[];
  const int bs = pad_stride(N2);
  C* buf = reinterpret_cast<C*>(smem);
  C* tws = buf + (size_t)2 * P * bs;
  const bool smem_tw = sizeof(T) == 4;
  if (smem_tw) load_tw_smem<T>(tws, stw, stage_tw_len(log2N2, F::E));
  const C* A = Ain + (int64_t)blockIdx.y * N;
  C* out = reinterpret_cast<C*>(dst + (int64_t)blockIdx.y * dst_stride);
  const int p0 = blockIdx.x * P;
  const int total = 2 * P * N2;
  constexpr int LD = InFlight<T>::v;
  for (int idx0 = threadIdx.x; idx0 < total; idx0 += LD * blockDim.x) {
    C z[LD];
#pragma unroll
    for (int u = 0; u < LD; ++u) {
      const int idx = idx0 + u * blockDim.x;
      if (idx < total) z[u] = A[((int64_t)(2 * p0 + (idx >> log2N2)) << log2N2) + (idx & (N2 - 1))];
    }
#pragma unroll
    for (int u = 0; u < LD; ++u) {
      const int idx = idx0 + u * blockDim.x;
      if (idx < total) buf[(idx >> log2N2) * bs + padi(idx & (N2 - 1))] = z[u];
    }
  }
  __syncthreads();
  fft_any<T, F::E, F::EPT>(buf, log2N2, 2 * P, bs, smem_tw ? tws : stw);
  // lanes take consecutive rows, so each store run covers 2P consecutive outputs
  const int log2R = __ffs(2 * P) - 1;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int q = idx & (2 * P - 1);
    const int k2 = idx >> log2R;
    C R = buf[q * bs + padi(k2)];
    const int64_t k = (int64_t)(2 * p0 + q) + (int64_t)N1 * k2;
    if (E == EP_CPLX_MC) {
      const C t = cmul(R, tab[k]);
      R.x = t.x;
      R.y = -t.y;
    }
    out[k] = R;
  }
}

// ---------------------------------------------------------------------------------------------
// Batched launches over plans of different N (birkhoff_apply_batch): one launch covers up to
// BATCH_MAX plans. A job is one plan's part of a launch (its vectors and shapes); CTA (or cluster)
// b of the launch belongs to the job q with start[q] <= b < start[q + 1] and runs that job's body,
// whose results do not depend on the launch's thread count or cluster size. The descriptors travel
// as __grid_constant__ kernel parameters.
// ---------------------------------------------------------------------------------------------
constexpr int BATCH_MAX = 16;

template <typename T> struct SmallJob {
  const T* in;
  T* out;
  int64_t pitch;
  const typename V2<T>::t* tw;
  const typename V2<T>::t* stw;
  const typename V2<T>::t* tpost;
  StencilTab<T> tb;
  T s;
  int N, log2N, nblk;
};

template <typename J> struct Batch {
  int njob;
  int start[BATCH_MAX + 1];   // first CTA of each job; start[njob] = the launch's CTAs
  J j[BATCH_MAX];
};

template <typename J>
__device__ __forceinline__ int batch_job(const Batch<J>& b, int cta) {
  int q = 0;
  while (q + 1 < b.njob && cta >= b.start[q + 1]) ++q;
  return q;
}

template <typename T, bool TRANS>
__global__ void __launch_bounds__(sizeof(T) == 8 ? 256 : 1024) k_small_batch(const __grid_constant__ Batch<SmallJob<T>> b) {
  pdl_wait();
  const int q = batch_job(b, blockIdx.x);
  const SmallJob<T>& J = b.j[q];
  small_body<T, TRANS>((int)blockIdx.x - b.start[q], J.in, J.out, J.N, J.log2N, J.pitch, J.s, J.tw, J.stw, J.tpost,
                       J.tb);
}

// Launch-per-pass plans of one radix F: CTA b of a job runs vector b % nvec of tile b / nvec.
template <typename T, bool TRANS, bool SECOND, typename F>
__global__ void __launch_bounds__(F::MT, F::MINB) k_re_passA_batch(const __grid_constant__ Batch<ReJob<T>> b) {
  pdl_wait();
  const int q = batch_job(b, blockIdx.x);
  const ReJob<T>& J = b.j[q];
  const int l = (int)blockIdx.x - b.start[q];
  if constexpr (SECOND)
    re_passA_cta<T, TRANS ? ST_TRN : ST_FWD, F, T>(J.g, l % J.nvec, l / J.nvec, J.NB, J.bsA, J.Y, J.ystride, J.A, J.astride,
                                                   J.part);
  else
    re_passA_cta<T, TRANS ? IN_WINV : IN_PLAIN, F, T>(J.g, l % J.nvec, l / J.nvec, J.NB, J.bsA, J.in, J.pitch, J.A,
                                                      J.astride, J.part);
}
template <typename T, bool TRANS, bool SECOND, typename F>
__global__ void __launch_bounds__(F::MT, F::MINB) k_re_passB_batch(const __grid_constant__ Batch<ReJob<T>> b) {
  pdl_wait();
  const int q = batch_job(b, blockIdx.x);
  const ReJob<T>& J = b.j[q];
  const int l = (int)blockIdx.x - b.start[q];
  if constexpr (SECOND)
    re_passB_cta<T, TRANS ? EP_TRN_OUT : EP_FWD_OUT, F, T>(J.g, l % J.nvec, l / J.nvec, J.P, J.bsB, J.A, J.astride, J.out,
                                                           J.pitch, J.pitch, J.part, J.s, J.invN);
  else
    re_passB_cta<T, TRANS ? EP_STORE_TRN : EP_STORE, F, T>(J.g, l % J.nvec, l / J.nvec, J.P, J.bsB, J.A, J.astride, J.Y,
                                                           J.ystride, 0, J.part, J.s, J.invN);
}

template <typename T, bool TRANS>
__global__ void __launch_bounds__(512, sizeof(T) == 8 ? 1 : 2) k_re_cluster_batch(const __grid_constant__ Batch<ReJob<T>> b, int csize) {
  pdl_wait();
  const int cl = blockIdx.x / csize;
  const int q = batch_job(b, cl);
  re_cluster_body<T, TRANS>(b.j[q], cl - b.start[q], blockIdx.x % csize, csize);
}

// ---------------------------------------------------------------------------------------------
// Plan creation / destruction and the apply entry points
// ---------------------------------------------------------------------------------------------
template <typename T>
static bk_status build_stage_table(void** dst, int64_t n, int e, cudaStream_t st) {
  typedef typename V2<T>::t C;
  const int len = stage_tw_len(ilog2(n), e);
  if (len == 0) return BK_OK;
  BK_TRY(dmalloc(dst, sizeof(C) * len));
  k_stage_tw<T><<<(len + 255) / 256, 256, 0, st>>>((C*)*dst, ilog2(n), e, len);
  BK_CHECK_LAUNCH();
  return BK_OK;
}

template <typename T>
static bk_status build_mix_table(void** dst, const unsigned char* rad, int nst, cudaStream_t st) {
  typedef typename V2<T>::t C;
  int len = 0, Ns = 1;
  for (int s = 0; s < nst; Ns *= rad[s++])
    if (Ns > 1) len += (rad[s] - 1) * Ns;
  if (len == 0) return BK_OK;
  BK_TRY(dmalloc(dst, sizeof(C) * len));
  C* p = (C*)*dst;
  Ns = 1;
  for (int s = 0; s < nst; Ns *= rad[s++]) {
    if (Ns == 1) continue;
    const int n = (rad[s] - 1) * Ns;
    k_mix_tw<T><<<(n + 255) / 256, 256, 0, st>>>(p, Ns, rad[s]);
    BK_CHECK_LAUNCH();
    p += n;
  }
  return BK_OK;
}

// Tables of the plain complex layout: stage tables and the inter-pass twiddles.
template <typename T>
static bk_status build_fs_tables(FourStep& f, int e, cudaStream_t st) {
  typedef typename V2<T>::t C;
  BK_TRY(build_stage_table<T>(&f.stw1, f.N1, e, st));
  BK_TRY(build_stage_table<T>(&f.stw2, f.N2, e, st));
  const int64_t n = f.n;
  if (sizeof(T) == 8) {
    BK_TRY(dmalloc(&f.twN, sizeof(C) * n));
    k_tw_table<T><<<(int)std::min<int64_t>((n + 255) / 256, 8192), 256, 0, st>>>((C*)f.twN, n, (double)n);
    BK_CHECK_LAUNCH();
  } else {
    const int log2n = ilog2(n);
    f.tw_h = (log2n + 1) / 2;
    const int64_t nlo = int64_t(1) << f.tw_h, nhi = n >> f.tw_h;
    BK_TRY(dmalloc(&f.twLo, sizeof(C) * nlo));
    BK_TRY(dmalloc(&f.twHi, sizeof(C) * nhi));
    k_tw_table<T><<<(int)((nlo + 255) / 256), 256, 0, st>>>((C*)f.twLo, nlo, (double)n);
    BK_CHECK_LAUNCH();
    k_tw_table_strided<T><<<(int)((nhi + 255) / 256), 256, 0, st>>>((C*)f.twHi, nhi, nlo, (double)n);
    BK_CHECK_LAUNCH();
  }
  return BK_OK;
}

static void free_fs(FourStep& f) {
  dfree(f.stw1);
  dfree(f.stw2);
  dfree(f.twN);
  dfree(f.twLo);
  dfree(f.twHi);
  f = FourStep();
}

static int re_tw_blocks(const FourStep& f) { return (int)std::min<int64_t>((f.a_len() + 255) / 256, 8192); }

template <typename T>
static bk_status build_tables(Plan* p, cudaStream_t st) {
  typedef typename V2<T>::t C;
  const int64_t N = p->N;
  // FFT twiddles: single-CTA plans keep omega_N^i (direct DFT for N < 16) and the stage table of
  // N; four-step plans the stage tables of N1 and N2 and the inter-pass table.
  if (p->blue) {
    BK_TRY(build_fs_tables<T>(p->fsM, p->fe, st));
    BK_TRY(dmalloc(&p->chirp, sizeof(C) * N));
    k_chirp<T><<<(int)std::min<int64_t>((N + 255) / 256, 4096), 256, 0, st>>>((C*)p->chirp, N);
    BK_CHECK_LAUNCH();
    BK_TRY(dmalloc(&p->bh, sizeof(C) * p->M));   // filled by blue_spectrum once the kernels are set up
  } else if (p->small) {
    BK_TRY(dmalloc(&p->tw, sizeof(C) * N));
    k_tw_table<T><<<(int)std::min<int64_t>((N + 255) / 256, 4096), 256, 0, st>>>((C*)p->tw, N, (double)N);
    BK_CHECK_LAUNCH();
    if (N >= 16) BK_TRY(build_stage_table<T>(&p->stwS, N, SmallFft<T>::E, st));
  } else {
    const int e = p->split ? p->fe : SmallFft<T>::E;
    if (p->mix) {
      BK_TRY(build_mix_table<T>(&p->fs.stw1, p->rad1, p->nst1, st));
      BK_TRY(build_mix_table<T>(&p->fs.stw2, p->rad2, p->nst2, st));
    } else {
      BK_TRY(build_stage_table<T>(&p->fs.stw1, p->fs.N1, e, st));
      BK_TRY(build_stage_table<T>(&p->fs.stw2, p->fs.N2, e, st));
    }
    BK_TRY(dmalloc(&p->fs.twN, sizeof(C) * p->fs.a_len()));
    k_re_tw<T><<<re_tw_blocks(p->fs), 256, 0, st>>>((C*)p->fs.twN, p->fs.N1, p->fs.N2);
    BK_CHECK_LAUNCH();
  }
  BK_TRY(dmalloc(&p->rk, sizeof(T) * (N + 2)));
  k_rk_table<T><<<(int)std::min<int64_t>((N + 2 + 255) / 256, 4096), 256, 0, st>>>((T*)p->rk, N + 2);
  BK_CHECK_LAUNCH();
  if (p->blue || p->small) {
    BK_TRY(dmalloc(&p->tpost, sizeof(C) * (N / 2 + 1)));
    k_post_table<T><<<(int)std::min<int64_t>((N / 2 + 256) / 256, 4096), 256, 0, st>>>((C*)p->tpost, N);
    BK_CHECK_LAUNCH();
  }
  return BK_OK;
}

#ifndef BK_TRANSFORM_KERNEL_UNIT
// Clenshaw-Curtis weights (the last row of B^a) in closed form, each to its own relative accuracy. With
// theta = pi k / N, w_k = (c / N) [1 - sum_{j <= N/2}'' 2 cos(2 j theta) / (4 j^2 - 1)] (c = 1 at the ends,
// 2 inside). The series taken to infinity is (pi/2) sin theta, and its remainder, with 2 / (4 j^2 - 1) =
// int_0^1 x^{2j-2} (1 - x^2) dx summed as a geometric series under the integral and x = e^{-t/N}, is
//   T = (1/N) int_0^inf e^{-t} e^{t/N} u^2 (1 + r) / (2 (u^2 + 4 r sin^2 theta)) dt       (N even),
//   T = (1/N) int_0^inf e^{-t} cos theta u^2 / (u^2 + 4 r sin^2 theta) dt                  (N odd),
// u = 1 - r, r = e^{-2t/N}, so that N w_k / c = (pi/2) sin theta + (-1)^k T. The integrand's poles lie near
// t = +- i pi k: from k = 32 on five Gauss-Laguerre nodes give T to 3e-18 of the weight, from k = 1024 on its
// leading term in 1 / sin^2 theta does (past 1.6e5 T is below 1e-17 of it); below, the trapezoidal rule in
// y, t = exp(y - e^{-y}), at 96 points (one warp per weight). The ends are 1 / (N^2 - 1) and 1 / N^2.
// (The transposed product with e_N, used before, has its absolute rounding in every weight: the weights next to
// the ends, which the KKT preconditioner's control block divides by, were off by some N ulp. It also needed a
// binary64 plan, 0.6 ms of the 1.1 for a plan of N = 2^20, which FP32 lengths above 2^22 do not have.)
__device__ __forceinline__ void put_weight(double v, int64_t k, int64_t N, double* w, float* wT) {
  w[k] = w[N - k] = v;
  if (wT) wT[k] = wT[N - k] = (float)v;
}

__global__ void __launch_bounds__(256) k_weights(double* __restrict__ w, float* __restrict__ wT, int64_t N, int64_t pitch) {
  // nodes and weights of the Gauss-Laguerre rule (zeros t of L_5, t / (36 L_6(t)^2))
  const double gt[5] = {0.26356031971814091020, 1.4134030591065167922, 3.5964257710407220812, 7.0858100058588375569,
                        12.640800844275782659};
  const double gw[5] = {0.52175561058280865248, 0.39866681108317592745, 0.075942449681707595388,
                        0.0036117586799220484545, 0.000023369972385776227891};
  __shared__ double su[5], sr[5], sc[5], lead;   // u^2, 4 r, and the numerator of each node
  const bool odd = N & 1;
  if (threadIdx.x < 5) {
    const int i = threadIdx.x;
    const double u = -expm1(-2.0 * gt[i] / (double)N), r = 1.0 - u;
    su[i] = u * u;
    sr[i] = 4.0 * r;
    sc[i] = gw[i] * u * u * (odd ? 1.0 : 0.5 * (1.0 + r) * exp(gt[i] / (double)N));
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0;
    for (int i = 0; i < 5; ++i) a += sc[i] / sr[i];
    lead = a;
  }
  __syncthreads();
  const double iN = 1.0 / (double)N;
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = 32 + id; k <= N / 2; k += nt) {
    const double x = (double)k / (double)N;
    const double s = sinpi(x);
    double v = 1.5707963267948966192 * s;
    if (k < 163840) {
      const double s2 = s * s;
      double T = 0.0;
      if (k >= 1024) {
        T = lead / s2;
      } else {
        for (int i = 0; i < 5; ++i) T += sc[i] / fma(sr[i], s2, su[i]);
      }
      T *= odd ? iN * cospi(x) : iN;
      v = (k & 1) ? v - T : v + T;
    }
    put_weight(2.0 * v / (double)N, k, N, w, wT);
  }
  for (int64_t k = N + 1 + id; k < pitch; k += nt) w[k] = 0.0;
}

// Weights k = blockIdx.x < 32 from either end; one warp.
__global__ void __launch_bounds__(32) k_weight_ends(double* __restrict__ w, float* __restrict__ wT, int64_t N) {
  const int64_t k = blockIdx.x;
  if (k > N / 2) return;
  const double n = (double)N;
  const bool odd = N & 1;
  if (k == 0) {
    if (threadIdx.x == 0) put_weight(odd ? 1.0 / (n * n) : 1.0 / ((n - 1.0) * (n + 1.0)), 0, N, w, wT);
    return;
  }
  double s, c;
  sincospi((double)k / n, &s, &c);
  const double h = 0.125;
  double T = 0.0;
  for (int i = threadIdx.x; i < 96; i += 32) {
    const double y = -4.5 + h * i, ey = exp(-y), t = exp(y - ey);
    const double u = -expm1(-2.0 * t / n), r = 1.0 - u;
    const double q = odd ? c : 0.5 * (1.0 + r);
    const double e = exp(odd ? -t : -t * (n - 1.0) / n);
    T += h * t * (1.0 + ey) * e * q * u * u / fma(4.0 * r, s * s, u * u);
  }
  for (int o = 16; o > 0; o >>= 1) T += __shfl_xor_sync(0xffffffffu, T, o);
  T /= n;
  const double v = 1.5707963267948966192 * s;
  if (threadIdx.x == 0) put_weight(2.0 * ((k & 1) ? v - T : v + T) / n, k, N, w, wT);
}

static bk_status compute_weights(Plan* p, cudaStream_t st) {
  BK_TRY(dmalloc((void**)&p->w64, sizeof(double) * p->pitch));
  if (p->dtype == BK_F32) BK_TRY(dmalloc(&p->wT, sizeof(float) * p->L));
  k_weights<<<(int)std::min<int64_t>((p->N / 2 + 256) / 256, 4096), 256, 0, st>>>(p->w64, (float*)p->wT, p->N, p->pitch);
  BK_CHECK_LAUNCH();
  k_weight_ends<<<32, 32, 0, st>>>(p->w64, (float*)p->wT, p->N);
  BK_CHECK_LAUNCH();
  return BK_OK;
}
#endif  // BK_TRANSFORM_KERNEL_UNIT

// Largest N run by the single-CTA kernel (one CTA per vector): 256 in FP64, whose single CTA runs
// on one SM's FP64 pipe, 2048 in FP32. Measured (4 components, us per product, one CTA / cluster): FP64
// 2^8 12.0 / 18.1, 2^9 19.8 / 18.2; FP32 2^11 10.2 / 11.6, 2^12 14.3 / 13.8 (transposed 14.6 / 13.9). BK_SMALL_MAX_LOG2
// overrides it for tuning (at least 2^4; at most 512 in FP64, 4096 in FP32). The four-step kernels
// need N >= 128.
static int small_default(int dtype) { return dtype == BK_F64 ? 256 : 2048; }
static int small_limit(int dtype) {
  const int cap = dtype == BK_F64 ? 512 : 4096;
  const char* e = getenv("BK_SMALL_MAX_LOG2");
  if (e) {
    const long v = atol(e);
    if (v >= 4 && v <= 13) return std::min(cap, 1 << (int)v);
  }
  return small_default(dtype);
}

template <typename T>
static size_t smem_small(int64_t N) {
  const int64_t L = N + 1;
  const int64_t Lp = (L + 3) & ~3;
  return sizeof(T) * 2 * Lp + sizeof(typename V2<T>::t) * (size_t)pad_stride((int)N);
}

static int round_threads(int64_t t) {  // whole warps
  t = (t + 31) / 32 * 32;
  return (int)std::min<int64_t>(1024, std::max<int64_t>(32, t));
}

static constexpr size_t FOURSTEP_SMEM_BUDGET = 192 * 1024;
static size_t align256(size_t b) { return (b + 255) / 256 * 256; }

static int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
      n = 152;
  }
  return n;
}

// Complex elements per CTA of a pass: enough CTAs for two per SM over the plan's
// vectors, at least one column of N1 and one row pair of 2 N2, at most the thread cap. Small
// transforms thus run many one-warp CTAs instead of a few full ones (at 2^14 x 4 components the
// full-size tiles gave 16 CTAs per pass). BK_FOURSTEP_ELEMS fixes it (tuning).
static int fourstep_elems(int dtype, int64_t n, int nvec, int N1, int N2, int Eforce = 0) {
  const int cap = dtype == BK_F64 ? 4096 : 8192;  // values per thread x the thread cap
  if (Eforce > 0) return std::min(cap, std::max(Eforce, std::max(N1, 2 * N2)));
  const char* e = getenv("BK_FOURSTEP_ELEMS");
  if (e) {
    long v = atol(e);
    if (v >= 16 && v <= cap && is_pow2(v)) return std::max<int>((int)v, std::max(N1, 2 * N2));
  }
  int64_t target = n * (int64_t)std::max(1, nvec) / (2 * sm_count());
  int64_t E = 1;
  while (E * 2 <= target) E *= 2;
  E = std::max<int64_t>(E, std::max(N1, 2 * N2));
  return (int)std::min<int64_t>(E, cap);
}

// Whether the four passes run as a launch each instead of as one cluster launch: from 2^13 on, and in FP64
// from 2^12 with more than 8 vectors, whose sixteen CTAs per vector then share FP64 pipes. Measured
// (us per product, cluster / launch per pass): FP64, 4 components, 2^11 20.5 / 24.5, 2^12 23.8 / 31.1, 2^13 31.7 /
// 32.1, 2^14 47.0 / 34.2; 16 components 2^10 21.6 / 25.2, 2^12 36.4 / 30.8; FP32 2^12 13.8 / 15.5,
// 2^13 17.1 / 15.5, 2^14 20.5 / 16.5 (2^13 and 2^14 with the exchange in global memory, where 2^12 took 12.9). BK_SPLIT_MIN_LOG2 sets the border for tuning.
static bool split_passes(int dtype, int64_t N, int nvec) {
  const char* e = getenv("BK_SPLIT_MIN_LOG2");
  if (e) {
    const long v = atol(e);
    // FP32 one-launch plans keep their exchange area in shared memory: N <= 2^13
    if (v >= 7 && v <= 30) return ilog2(N) >= std::min((int)v, dtype == BK_F32 ? 14 : 2 * CL_MAXLOG2);
  }
  return N >= 8192 || (dtype == BK_F64 && N >= 4096 && nvec > 8);
}

// log2 radix of the plain complex passes of length n: 4 in FP32; in FP64 2 while few warps share the
// FP64 pipes and 4 from 2^18 on, where its fewer shared-memory round trips count (products of 4
// components, radix 4 / radix 16, us: N = 3001 61 / 127, N = 140001 1512 / 1344, N = 393217 2853 / 2433).
static int cplx_radix(int dtype, int64_t n) { return dtype == BK_F64 && n < (int64_t(1) << 18) ? 2 : 4; }

static bk_status configure_fourstep(FourStep& f, int64_t n, int dtype, int fe, int nvec, int Eforce = 0) {
  const int ept = 1 << fe;
  const int log2n = ilog2(n);
  f.n = n;
  // balanced factors, with the rows short enough for one row pair per CTA (2 N2 / EPT threads)
  // and the columns for one column per CTA (N1 / EPT threads) under the thread cap
  const int maxthr = (dtype == BK_F64 ? 4096 : 8192) / ept;
  int l2 = log2n - log2n / 2;
  while (l2 > 0 && (2 << l2) / ept > maxthr) --l2;
  f.N2 = 1 << l2;
  f.N1 = 1 << (log2n - l2);
  if (f.N1 / ept > maxthr) {
    set_error("four-step configuration failed for n=%lld (transform too long for this precision)", (long long)n);
    return BK_ERR_UNSUPPORTED;
  }
  const size_t csz = 2 * dtype_size(dtype);
  const int E = fourstep_elems(dtype, n, nvec, f.N1, f.N2, Eforce);
  // pass A: NB columns of N1; pass B: P row pairs (2P rows) of N2
  int NB = std::max(1, E / f.N1);
  if (NB > f.N2) NB = f.N2;
  int P = std::max(1, E / (2 * f.N2));
  if (P > f.N1 / 2) P = f.N1 / 2;
  f.NB = NB;
  f.P = P;
  // Pass-A batch stride: when a warp's FFT stays inside one batch (N1 / 16 >= 32 threads), the
  // column-major tile accesses of the load and store phases (lane -> column idx mod NB, row
  // idx / NB) hit distinct banks if the stride is = W / NB modulo the W complex elements of a
  // 128-byte wavefront.
  const int W = (int)(128 / csz);
  const int padA = (f.N1 / 16 >= 32 && NB < W) ? W / NB : 1;
  f.bsA = f.N1 + f.N1 / 16 + padA;
  f.smemA = csz * ((size_t)NB * f.bsA + (dtype == BK_F32 ? f.N1 : 0));
  f.smemB = csz * ((size_t)2 * P * pad_stride(f.N2) + (dtype == BK_F32 ? f.N2 : 0));
  f.thrA = round_threads((int64_t)NB * f.N1 / ept);
  f.thrB = round_threads((int64_t)2 * P * f.N2 / ept);
  if ((int64_t)NB * f.N1 / ept > maxthr || (int64_t)2 * P * f.N2 / ept > maxthr || f.smemA > FOURSTEP_SMEM_BUDGET ||
      f.smemB > FOURSTEP_SMEM_BUDGET) {
    set_error("four-step configuration failed for n=%lld", (long long)n);
    return BK_ERR_UNSUPPORTED;
  }
  return BK_OK;
}

// Batch stride of a tile of nb transforms of length n in shared memory: when a warp's FFT stays
// inside one transform (n / 16 >= 32 threads), the accesses with the transform as the fastest lane
// index hit distinct banks if the stride is = W / nb modulo the W complex elements of a 128-byte
// wavefront.
static int re_stride(int dtype, int n, int nb) {
  const int W = dtype == BK_F64 ? 8 : 16;
  return n + n / 16 + (n / 16 >= 32 && nb < W ? W / nb : 1);
}

// Factors of the real-even passes, 2N = N1 N2 (both >= 16 for N >= 128). At N = 2^24 the FP64 rows
// have 8192 points (the BIG instances of pass B).
static void re_factors(FourStep& f, int64_t N) {
  const int l = ilog2(N) + 1;
  f.n = 2 * N;
  f.N1 = 1 << (l / 2);
  f.N2 = 1 << (l - l / 2);
}

// Scratch of the passes of nvec FP32 vectors: A, the stage buffer and the shares of R_0. A launch-per-pass
// plan of radix 4 keeps that of up to GUEST_VECTORS vectors of N = 4096 for the one-launch plans that
// join its launches in a batch; its own scratch serves one call at a time anyway.
static constexpr int GUEST_VECTORS = 64;
static size_t re_scratch_f32(int64_t N, int64_t nvec) {
  FourStep f;
  re_factors(f, N);
  return align256(2 * sizeof(float) * (size_t)f.a_len() * nvec) + align256(sizeof(float) * (size_t)(N + 2) * nvec) +
         align256(sizeof(float) * (size_t)f.pairs() * nvec);
}

static bool re_big(const FourStep& f, int dtype) { return dtype == BK_F64 && f.N2 > 4096; }

// log2 radix of the launch-per-pass kernels (the reasons and figures are in bk_fft.cuh), and the
// complex elements per CTA their thread cap admits.
static int re_radix(int64_t N, int dtype, bool df) {
  if (dtype == BK_F64) return df ? 3 : 2;
  return N <= (int64_t(1) << 18) ? 2 : 4;
}
static int re_elems_max(const FourStep& f, int dtype, int fe) {
  if (dtype == BK_F32) return fe == 4 ? FftShape<float, 4>::MT * FftShape<float, 4>::EPT : FftShape<float, 2>::MT * FftShape<float, 2>::EPT;
  return std::max(4096, f.N2);   // 1024 threads of 4 or 512 of 8; one longer row takes BigFft
}

// Tiles of the launch-per-pass form for E complex elements per CTA (0: enough CTAs for two per SM
// over the plan's vectors).
static bk_status configure_re(FourStep& f, int64_t N, int dtype, int fe, int nvec, int Eforce = 0) {
  re_factors(f, N);
  const int E = std::min(re_elems_max(f, dtype, fe), fourstep_elems(dtype, N / 2, nvec, f.N1, f.N2 / 2, Eforce));
  f.NB = std::max(1, E / f.N1);
  f.P = std::max(1, E / f.N2);
  const size_t csz = 2 * dtype_size(dtype);
  f.bsA = re_stride(dtype, f.N1, f.NB);
  f.bsB = re_stride(dtype, f.N2, f.P);
  f.smemA = csz * ((size_t)f.NB * f.bsA + (dtype == BK_F32 ? stage_tw_len(ilog2(f.N1), fe) : 0));
  f.smemB = csz * ((size_t)f.P * f.bsB + (dtype == BK_F32 ? stage_tw_len(ilog2(f.N2), fe) : 0));
  const int64_t tA = (int64_t)f.NB * f.N1 >> fe, tB = re_big(f, dtype) ? 512 : (int64_t)f.P * f.N2 >> fe;
  f.thrA = round_threads(tA);
  f.thrB = round_threads(tB);
  if (f.smemA > FOURSTEP_SMEM_BUDGET || f.smemB > FOURSTEP_SMEM_BUDGET || f.thrA < tA || f.thrB < tB) {
    set_error("four-step configuration failed for N=%lld", (long long)N);
    return BK_ERR_UNSUPPORTED;
  }
  return BK_OK;
}

// Mixed-radix lengths: n as radices, the odd ones first (their stage without twiddles), 0 stages when
// n has another prime factor.
static int mix_radices(int n, unsigned char* rad) {
  int k = 0;
  unsigned char r4[12];
  int k4 = 0;
  while (n % 5 == 0 && k < 12) { rad[k++] = 5; n /= 5; }
  while (n % 3 == 0 && k < 12) { rad[k++] = 3; n /= 3; }
  while (n % 4 == 0 && k4 < 12) { r4[k4++] = 4; n /= 4; }
  if (n == 2 && k < 12) { rad[k++] = 2; n = 1; }
  if (n != 1 || k + k4 > 12) return 0;
  for (int i = 0; i < k4; ++i) rad[k++] = r4[i];
  return k;
}

// Longest mixed-radix transform: two buffers of one transform in shared memory.
static int mix_max(int dtype) { return dtype == BK_F64 ? 5120 : 10240; }

// Factors 2N = N1 N2 of a mixed-radix plan: multiples of 4, N1 <= N2 as near as they come. False when N
// has no such form (N must be 16 times a product of 2, 3 and 5: then both halves of the passes' pairing are
// whole) or a factor is too long; Bluestein's convolution serves those, at 4 to 8 times the cost
// (products of 4 components, convolution / mixed radix, us: FP64 N = 100000 690 / 106, FP32 122 / 25).
static bool mix_factors(int64_t N, int dtype, int* N1, int* N2) {
  if (N % 16 != 0 || is_pow2(N)) return false;
  int64_t m = N / 16;
  for (int f : {2, 3, 5})
    while (m % f == 0) m /= f;
  if (m != 1) return false;
  int64_t best = 0;
  for (int64_t a = 16; a * a <= 2 * N; a += 4)
    if ((2 * N) % a == 0 && (2 * N / a) % 4 == 0) best = a;
  if (best == 0 || 2 * N / best > mix_max(dtype)) return false;
  unsigned char r[12];
  if (mix_radices((int)best, r) == 0 || mix_radices((int)(2 * N / best), r) == 0) return false;
  *N1 = (int)best;
  *N2 = (int)(2 * N / best);
  return true;
}

// Tiles of a mixed-radix plan for E complex elements per CTA (0: enough CTAs for two per SM).
static bk_status configure_mix(Plan* p, int nvec, int Eforce) {
  FourStep& f = p->fs;
  if (!mix_factors(p->N, p->dtype, &f.N1, &f.N2)) {
    set_error("mixed-radix configuration failed for N=%lld", (long long)p->N);
    return BK_ERR_UNSUPPORTED;
  }
  f.n = 2 * p->N;
  p->nst1 = mix_radices(f.N1, p->rad1);
  p->nst2 = mix_radices(f.N2, p->rad2);
  const int E = std::min(p->dtype == BK_F64 ? 4096 : 8192, fourstep_elems(p->dtype, p->N / 2, nvec, f.N1, f.N2 / 2, Eforce));
  f.NB = std::max(1, std::min(E / f.N1, f.N2 / 4 + 1));
  f.P = std::max(1, std::min(E / f.N2, f.N1 / 4 + 1));
  f.bsA = f.N1 + f.N1 / 16 + 1;
  f.bsB = f.N2 + f.N2 / 16 + 1;
  const size_t csz = 2 * dtype_size(p->dtype);
  f.smemA = csz * 2 * (size_t)f.NB * f.bsA;
  f.smemB = csz * 2 * (size_t)f.P * f.bsB;
  f.thrA = f.thrB = MixFft::MT;
  if (f.smemA > FOURSTEP_SMEM_BUDGET || f.smemB > FOURSTEP_SMEM_BUDGET) {
    set_error("mixed-radix tiles too large for N=%lld", (long long)p->N);
    return BK_ERR_UNSUPPORTED;
  }
  return BK_OK;
}

// Tiles of the one-launch form: a cluster of at most 16 CTAs per vector, its column and row pairs
// spread over all of them.
static bk_status configure_cluster(Plan* p) {
  FourStep& f = p->fs;
  re_factors(f, p->N);
  p->csize = std::min(16, f.N2 / 4);
  const int maxthr = 512;
  const int ept = p->dtype == BK_F64 ? SmallFft<double>::EPT : SmallFft<float>::EPT;
  const int e = p->dtype == BK_F64 ? SmallFft<double>::E : SmallFft<float>::E;
  auto per = [&](int pairs, int n) {   // pairs per CTA, in as few equal rounds as the thread cap allows
    const int each = (pairs + p->csize - 1) / p->csize;
    const int rounds = (int)(((int64_t)each * n / ept + maxthr - 1) / maxthr);
    return (each + rounds - 1) / rounds;
  };
  f.NB = per(f.N2 / 4 + 1, f.N1);
  f.P = per(f.N1 / 4 + 1, f.N2);
  f.bsA = re_stride(p->dtype, f.N1, f.NB);
  f.bsB = re_stride(p->dtype, f.N2, f.P);
  const size_t csz = 2 * dtype_size(p->dtype);
  p->csmem = csz * (size_t)(std::max(f.NB * f.bsA, f.P * f.bsB) + stage_tw_len(ilog2(f.N1), e) + stage_tw_len(ilog2(f.N2), e));
  if (p->dtype == BK_F32) {   // the exchange area: rows of A that this CTA's pass B reads, stage block, shares
    const int tiles = ((f.N1 / 4 + f.P) / f.P + p->csize - 1) / p->csize;
    p->cex = (int)align256(p->csmem);
    p->cexY = p->cex + (int)align256(csz * (size_t)tiles * f.P * 2 * f.RS());
    p->cexP = p->cexY + (int)align256(sizeof(float) * (size_t)(p->N / p->csize + 2));
    p->csmem = p->cexP + align256(sizeof(float) * (size_t)f.pairs());
  }
  p->cthr = std::max(128, round_threads(std::max(f.NB * f.N1, f.P * f.N2) / ept));
  if (p->csmem > FOURSTEP_SMEM_BUDGET || p->cthr > maxthr) {
    set_error("cluster configuration failed for N=%lld", (long long)p->N);
    return BK_ERR_UNSUPPORTED;
  }
  return BK_OK;
}

// The dynamic shared-memory cap is a per-function setting shared by every plan, so it is set to
// the largest size any plan of the type can request (never to one plan's own size, which would
// lower the cap under plans created earlier).
// No carveout is preferred: the L1 that the resident CTAs' tiles leave free holds the stage twiddles
// of the FP64 kernels (with all of the array as shared memory, 4 components, us: double-float 2^20 246,
// 2^22 1041, FP32 2^22 339; without 225, 908, 304).
template <typename K>
static bk_status smem_attr(K* fn, int cap) {
  BK_TRY_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  return BK_OK;
}

template <typename T, typename F>
static bk_status re_attrs_B(int cap) {
  BK_TRY(smem_attr(k_re_passB<T, EP_STORE, F, T>, cap));
  BK_TRY(smem_attr(k_re_passB<T, EP_STORE_TRN, F, T>, cap));
  BK_TRY(smem_attr(k_re_passB<T, EP_FWD_OUT, F, Us<T>>, cap));
  BK_TRY(smem_attr(k_re_passB<T, EP_TRN_OUT, F, Us<T>>, cap));
  return BK_OK;
}

template <typename T, typename F>
static bk_status re_attrs_AB(int cap) {
  BK_TRY(smem_attr(k_re_passA<T, IN_PLAIN, F, Us<T>>, cap));
  BK_TRY(smem_attr(k_re_passA<T, IN_WINV, F, Us<T>>, cap));
  BK_TRY(smem_attr(k_re_passA<T, ST_FWD, F, T>, cap));
  BK_TRY(smem_attr(k_re_passA<T, ST_TRN, F, T>, cap));
  return re_attrs_B<T, F>(cap);
}

template <typename T, typename F>
static bk_status cplx_attrs(int cap) {
  BK_TRY(smem_attr(k_passA<T, F>, cap));
  BK_TRY(smem_attr(k_passB<T, EP_CPLX, F>, cap));
  BK_TRY(smem_attr(k_passB<T, EP_CPLX_MC, F>, cap));
  return BK_OK;
}

template <typename F>
static bk_status cluster_attr(F* fn, int cap) {
  BK_TRY(smem_attr(fn, cap));
  BK_TRY_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  return BK_OK;
}

template <typename T>
static bk_status cluster_attrs(int cap) {
  BK_TRY(cluster_attr(k_re_cluster<T, false>, cap));
  BK_TRY(cluster_attr(k_re_cluster<T, true>, cap));
  BK_TRY(cluster_attr(k_re_cluster_batch<T, false>, cap));
  BK_TRY(cluster_attr(k_re_cluster_batch<T, true>, cap));
  return BK_OK;
}

// Whether the device (or the partition of it that the context has) holds a cluster of csize CTAs of
// every one-launch kernel, at the largest thread count a batch may launch them with.
template <typename T>
bool clusters_held(int csize, size_t smem) {
  if (cluster_attrs<T>((int)FOURSTEP_SMEM_BUDGET) != BK_OK) return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(csize);
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)csize;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  auto held = [&](auto* k) {
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      n = 0;
    }
    return n > 0;
  };
  return held(k_re_cluster<T, false>) && held(k_re_cluster<T, true>) && held(k_re_cluster_batch<T, false>) &&
         held(k_re_cluster_batch<T, true>);
}

template <typename T>
bk_status re_attrs() {
  const int cap = (int)FOURSTEP_SMEM_BUDGET;
  if constexpr (!std::is_same<T, dfl>::value) BK_TRY((re_attrs_AB<T, MixFft>(cap)));
  if constexpr (sizeof(T) == 4) {
    BK_TRY((re_attrs_AB<T, FftShape<T, 2>>(cap)));
    BK_TRY((re_attrs_AB<T, FftShape<T, 4>>(cap)));
  } else {
    BK_TRY((re_attrs_AB<T, FftShape<T, std::is_same<T, dfl>::value ? 3 : 2>>(cap)));
    BK_TRY((re_attrs_B<T, BigFft<T>>(cap)));
  }
  if constexpr (!std::is_same<T, dfl>::value) {
    BK_TRY(cluster_attrs<T>(cap));
    typedef FftShape<T, 2> F;
    BK_TRY(smem_attr(k_re_passA_batch<T, false, false, F>, cap));
    BK_TRY(smem_attr(k_re_passA_batch<T, false, true, F>, cap));
    BK_TRY(smem_attr(k_re_passA_batch<T, true, false, F>, cap));
    BK_TRY(smem_attr(k_re_passA_batch<T, true, true, F>, cap));
    BK_TRY(smem_attr(k_re_passB_batch<T, false, false, F>, cap));
    BK_TRY(smem_attr(k_re_passB_batch<T, false, true, F>, cap));
    BK_TRY(smem_attr(k_re_passB_batch<T, true, false, F>, cap));
    BK_TRY(smem_attr(k_re_passB_batch<T, true, true, F>, cap));
  }
  return BK_OK;
}

template <typename T>
bk_status set_smem_attrs(const Plan* p) {
  if (p->small) {
    if constexpr (!std::is_same<T, dfl>::value) {
      const int cap = (int)smem_small<T>(p->dtype == BK_F64 ? 512 : 4096);
      BK_TRY(smem_attr(k_birkhoff_small<T, false>, cap));
      BK_TRY(smem_attr(k_birkhoff_small<T, true>, cap));
      BK_TRY(smem_attr(k_small_batch<T, false>, cap));
      BK_TRY(smem_attr(k_small_batch<T, true>, cap));
    }
  } else if (p->blue) {
    if constexpr (!std::is_same<T, dfl>::value) {
      const int cap = (int)FOURSTEP_SMEM_BUDGET;
      BK_TRY((cplx_attrs<T, FftShape<T, 4>>(cap)));
      if constexpr (sizeof(T) == 8) BK_TRY((cplx_attrs<T, FftShape<T, 2>>(cap)));
    }
  } else {
    BK_TRY(re_attrs<T>());
  }
  return BK_OK;
}
// Largest N that is not a power of two (Bluestein, above the dense range): the length-M FFT
// (M >= 2N - 1) must fit the four-step shapes of the precision.
static int64_t blue_max(int dtype) { return dtype == BK_F64 ? (int64_t(1) << 22) : (int64_t(1) << 23); }

#ifndef BK_TRANSFORM_KERNEL_UNIT
// The instances of set_smem_attrs and apply_impl (and with them every transform kernel) are
// compiled in bk_birkhoff_f64.cu and bk_birkhoff_f32.cu, in parallel with this unit.
extern template bk_status set_smem_attrs<double>(const Plan* p);
extern template bk_status re_attrs<double>();
extern template bool clusters_held<double>(int, size_t);
extern template bool clusters_held<float>(int, size_t);
extern template bk_status set_smem_attrs<float>(const Plan* p);
extern template bk_status set_smem_attrs<dfl>(const Plan* p);
template <typename T> bk_status blue_spectrum(Plan* p, cudaStream_t st);
extern template bk_status blue_spectrum<double>(Plan* p, cudaStream_t st);
extern template bk_status blue_spectrum<float>(Plan* p, cudaStream_t st);
#endif

// Power-of-two plans take the FFT chain unless BK_DENSE=1 (read at plan creation; then every
// plan with N <= 1024 and at most 16 vectors per product starts on the dense product): building the
// dense tables (an O(N^3) FP64 formation of B^a per plan) in concurrent serving, where slots of
// other sizes are created and evicted, cut throughput from 191 to 152 solves/s on one GPU.
// BK_DENSE=0 is the default; N that is not a power of two is always dense.
// FP64 plans of N >= 2^18 compute their transforms in double-float arithmetic (bk_df.cuh) unless
// switched off: bk_set_f64_transform(0) for plans created afterwards, or the environment variable
// BK_F64_DF=0 (read at plan creation); bk_set_f64_transform(1) extends it to every FP64 plan with
// N >= 256. Measured products (4 components, warm, us, FP64 / double-float): 2^17 103 / 54, 2^18 195 /
// 79, 2^20 705 / 225. Below 2^18 the plans keep binary64's accuracy (relative errors 4e-16 against 8e-15).
#ifndef BK_TRANSFORM_KERNEL_UNIT
static std::atomic<int> g_f64_df{-1};
static bool f64_df_default(int64_t N) {
  const int m = g_f64_df.load();
  if (m >= 0) return m == 1;
  const char* e = getenv("BK_F64_DF");
  if (e && e[0] == '0') return false;
  return N >= (int64_t(1) << 18);
}
#endif

static bool dense_default(int dtype, int64_t N, int nvec) {
  (void)dtype;
  if (!dense_supported(N)) return false;
  const char* e = getenv("BK_DENSE");
  return e && e[0] == '1' && nvec <= 16;
}

// Four-step shapes of a plan for E complex elements per CTA (0: the occupancy heuristic).
static bk_status fourstep_shapes(Plan* p, int E) {
  const int nvec = p->n_comp * p->max_batch;
  if (p->mix) return configure_mix(p, nvec, E);
  return p->split ? configure_re(p->fs, p->N, p->dtype, p->fe, nvec, E) : configure_cluster(p);
}

// Tile autotuner of the four-step transforms. The elements per CTA E (powers of two from one
// column and one row pair up to the thread cap) set the CTA count, shared memory per CTA and how
// many CTAs share an SM; the best E depends on N, the vector count and the GPU. For each
// candidate the plan is re-shaped and timed (CUDA events, one B and one B^T, three times after a warm-up
// pair, on zero vectors: the kernels have no data-dependent paths); the fastest stays. Results
// are cached per (N, dtype, vectors, SM count, device) for the process, so plans of one size
// share one shape (and bitwise the same results). BK_AUTOTUNE=0 keeps the heuristic shape;
// BK_FOURSTEP_ELEMS, a fixed shape, also skips tuning.
static bool autotune_enabled() {
  const char* e = getenv("BK_AUTOTUNE");
  if (e && e[0] == '0') return false;
  return getenv("BK_FOURSTEP_ELEMS") == nullptr;
}

static std::mutex g_tune_mu;
static std::map<std::tuple<int64_t, int, int, int, int, int>, int> g_tune;

static bk_status autotune_tiles(Plan* p, cudaStream_t st) {
  const int nvec = p->n_comp * p->max_batch;
  int dev = 0;
  BK_TRY_CUDA(cudaGetDevice(&dev));
  const auto key = std::make_tuple(p->N, p->dtype, (int)p->df, nvec, sm_count(), dev);
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) {
      p->tileE = it->second;
      return fourstep_shapes(p, it->second);
    }
  }
  const int cap = p->mix ? (p->dtype == BK_F64 ? 4096 : 8192) : re_elems_max(p->fs, p->dtype, p->fe);
  const int emin = std::max(p->fs.N1, p->fs.N2);
  const size_t vbytes = dtype_size(p->dtype) * (size_t)p->pitch * nvec;
  void* vin = nullptr;
  void* vout = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  bk_status r = dmalloc(&vin, vbytes);
  if (r == BK_OK) r = dmalloc(&vout, vbytes);
  if (r == BK_OK && (cudaMemsetAsync(vin, 0, vbytes, st) != cudaSuccess || cudaEventCreate(&e0) != cudaSuccess ||
                     cudaEventCreate(&e1) != cudaSuccess)) {
    set_error("autotune: set-up failed");
    r = BK_ERR_CUDA;
  }
  int best = 0;
  float best_ms = 0.f;
  for (int E = emin; r == BK_OK && E <= cap; E *= 2) {
    if (fourstep_shapes(p, E) != BK_OK) continue;  // shape outside the thread/shared-memory caps
    r = plan_apply_n(p, vin, vout, nvec, false, p->s, st);
    if (r == BK_OK) r = plan_apply_n(p, vin, vout, nvec, true, p->s, st);
    for (int rep = 0; rep < 3; ++rep) {   // the least of three: one timing chose between near tiles at random
      if (r == BK_OK && cudaEventRecord(e0, st) != cudaSuccess) r = BK_ERR_CUDA;
      if (r == BK_OK) r = plan_apply_n(p, vin, vout, nvec, false, p->s, st);
      if (r == BK_OK) r = plan_apply_n(p, vin, vout, nvec, true, p->s, st);
      float ms = 0.f;
      if (r == BK_OK && (cudaEventRecord(e1, st) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
                         cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess)) {
        set_error("autotune: timing failed");
        r = BK_ERR_CUDA;
      }
      if (r == BK_OK && (best == 0 || ms < best_ms)) {
        best = E;
        best_ms = ms;
      }
    }
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  dfree(vin);
  dfree(vout);
  if (r != BK_OK) return r;
  if (best == 0) return fourstep_shapes(p, 0);
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune[key] = best;
  }
  p->tileE = best;
  return fourstep_shapes(p, best);
}

#ifndef BK_TRANSFORM_KERNEL_UNIT
bool plan_n_supported(int64_t N, int dtype) {
  return N >= 4 && (is_pow2(N) ? N <= (int64_t(1) << 24) : (dense_supported(N) || N <= blue_max(dtype)));
}

// Whether the one-launch form of the plan's size can run on the current device; asked once per device and
// shape. BK_MAX_CLUSTER (read at plan creation) sets the largest cluster instead, for tuning and tests.
static bool cluster_form_held(const Plan* p) {
  Plan q;
  q.N = p->N;
  q.dtype = p->dtype;
  if (configure_cluster(&q) != BK_OK) return false;
  const char* e = getenv("BK_MAX_CLUSTER");
  if (e) return q.csize <= atoi(e);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, size_t>, bool> seen;
  std::lock_guard<std::mutex> lk(mu);
  const auto key = std::make_tuple(dev, q.dtype, q.csize, q.csmem);
  auto it = seen.find(key);
  if (it == seen.end())
    it = seen.emplace(key, q.dtype == BK_F64 ? clusters_held<double>(q.csize, q.csmem) : clusters_held<float>(q.csize, q.csmem)).first;
  return it->second;
}

bk_status plan_create(Plan** out, int64_t N, int n_comp, int max_batch, int dtype, double t0, double tf, int64_t pitch,
                      cudaStream_t st) {
  *out = nullptr;
  BK_ARG(plan_n_supported(N, dtype),
         "N must be a power of two in [4, 2^24] or any N in [4, %lld] (this precision), got %lld",
         (long long)blue_max(dtype), (long long)N);
  BK_ARG(n_comp >= 1 && n_comp <= 64, "n_comp must be in [1, 64], got %d", n_comp);
  BK_ARG(max_batch >= 1, "max_batch must be >= 1, got %d", max_batch);
  BK_ARG(dtype == BK_F64 || dtype == BK_F32, "dtype must be BK_F64 or BK_F32");
  BK_ARG(tf != t0 && isfinite(t0) && isfinite(tf), "tf must differ from t0 and both be finite");
  const int64_t L = N + 1;
  if (pitch == 0) pitch = round_up(L, 32);
  BK_ARG(pitch >= L, "pitch %lld < N + 1", (long long)pitch);
  BK_ARG((pitch * (int64_t)dtype_size(dtype)) % 16 == 0, "pitch * sizeof(dtype) must be a multiple of 16");
  Plan* p = new Plan();
  p->N = N;
  p->L = L;
  p->n_comp = n_comp;
  p->max_batch = max_batch;
  p->dtype = dtype;
  p->t0 = t0;
  p->tf = tf;
  p->s = 0.5 * (tf - t0);
  p->pitch = pitch;
  // N not a power of two: the FFT chain does not apply; every product is the dense one
  p->generic = !is_pow2(N) && dense_supported(N);
  {
    int n1, n2;
    p->mix = !is_pow2(N) && !dense_supported(N) && mix_factors(N, dtype, &n1, &n2);
  }
  p->blue = !is_pow2(N) && !dense_supported(N) && !p->mix;
  {
    const char* e = getenv("BK_DENSE_TEST_TIMEOUT");  // test mode of the dense kernel, as bk_plan_dense_test_timeout
    p->dtest = (e && e[0] == '1') ? 1 : 0;
  }
  p->df = dtype == BK_F64 && is_pow2(N) && N >= 256 && f64_df_default(N);
  p->small = !p->generic && !p->blue && !p->mix && !p->df && N <= small_limit(dtype);
  const bool fourstep = !p->generic && !p->blue && !p->small;
  p->split = fourstep && (p->df || p->mix || split_passes(dtype, N, n_comp * max_batch));
  if (fourstep && !p->split && !cluster_form_held(p)) {
    p->small = dtype == BK_F32 && N <= 4096;   // the other form without scratch
    p->split = !p->small;
  }
  bk_status st_ = BK_OK;
  AllocCounter counter(&p->bytes);
  do {
    if ((st_ = dmalloc(&p->bsc, sizeof(double) * (size_t)n_comp * max_batch)) != BK_OK) break;
    if (p->generic) {
      if ((st_ = dmalloc((void**)&p->t_nodes, sizeof(double) * (size_t)L)) != BK_OK) break;
      k_grid_tables<<<(int)((L + 255) / 256), 256, 0, st>>>(p->t_nodes, N, t0, p->s);
      note_launch();
      if (cudaGetLastError() != cudaSuccess) { st_ = BK_ERR_CUDA; set_error("grid table launch failed"); break; }
      if ((st_ = dense_build(p, st)) != BK_OK) break;  // also the weights (last row of B^a)
      p->dense = true;
      cudaError_t e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) { set_error("plan tables: %s", cudaGetErrorString(e)); st_ = BK_ERR_CUDA; }
      break;
    }
    if (p->small) {
      p->smemS = dtype == BK_F64 ? smem_small<double>(N) : smem_small<float>(N);
      p->thrS = round_threads(std::max<int64_t>(N / (dtype == BK_F64 ? SmallFft<double>::EPT : SmallFft<float>::EPT), std::min<int64_t>(N, 256)));
    } else if (p->blue) {
      p->M = 1;
      while (p->M < 2 * N - 1) p->M *= 2;
      const int64_t nvec = (int64_t)n_comp * max_batch;
      p->fe = cplx_radix(dtype, p->M);
      if ((st_ = configure_fourstep(p->fsM, p->M, dtype, p->fe, (int)nvec)) != BK_OK) break;
      const size_t csz = 2 * dtype_size(dtype);
      if ((st_ = dmalloc(&p->scrA, csz * (size_t)p->M * 2 * nvec)) != BK_OK) break;   // two M-vectors
      if ((st_ = dmalloc(&p->scrY, dtype_size(dtype) * (size_t)(N + 1) * nvec)) != BK_OK) break;
      if ((st_ = dmalloc(&p->scrG, dtype_size(dtype) * (size_t)(N + 1) * nvec)) != BK_OK) break;
    } else {
      p->fe = p->mix ? 0 : re_radix(N, dtype, p->df);
      if ((st_ = fourstep_shapes(p, 0)) != BK_OK) break;
      const int64_t nvec = (int64_t)n_comp * max_batch;
      const size_t es = dtype_size(dtype);
      if (p->split || dtype == BK_F64) {   // FP32 one-launch plans exchange in shared memory
        if ((st_ = dmalloc(&p->scrA, 2 * es * (size_t)p->fs.a_len() * nvec)) != BK_OK) break;
        if ((st_ = dmalloc(&p->scrY, es * (size_t)(N + 2) * nvec)) != BK_OK) break;
        if ((st_ = dmalloc(&p->part, es * (size_t)p->fs.pairs() * nvec)) != BK_OK) break;
      }
      if (p->split && dtype == BK_F32 && p->fe == 2) {
        p->guest_bytes = (size_t)std::min<int64_t>(nvec, GUEST_VECTORS) * re_scratch_f32(4096, 1);
        if ((st_ = dmalloc(&p->guest, p->guest_bytes)) != BK_OK) break;
      }
    }
    st_ = dtype == BK_F64 ? (p->df ? build_tables<dfl>(p, st) : build_tables<double>(p, st)) : build_tables<float>(p, st);
    if (st_ != BK_OK) break;
    if ((st_ = dmalloc((void**)&p->t_nodes, sizeof(double) * (size_t)L)) != BK_OK) break;
    k_grid_tables<<<(int)((L + 255) / 256), 256, 0, st>>>(p->t_nodes, N, t0, p->s);
    note_launch();
    if (cudaGetLastError() != cudaSuccess) { st_ = BK_ERR_CUDA; set_error("grid table launch failed"); break; }
    st_ = dtype == BK_F64 ? (p->df ? set_smem_attrs<dfl>(p) : set_smem_attrs<double>(p)) : set_smem_attrs<float>(p);
    if (st_ != BK_OK) break;
    if (p->blue && (st_ = dtype == BK_F64 ? blue_spectrum<double>(p, st) : blue_spectrum<float>(p, st)) != BK_OK) break;
    if ((st_ = compute_weights(p, st)) != BK_OK) break;
    if (p->split && autotune_enabled()) {
      if ((st_ = autotune_tiles(p, st)) != BK_OK) break;
    }
    if (dense_default(dtype, N, n_comp * max_batch)) {
      if ((st_ = dense_build(p, st)) != BK_OK) break;
      p->dense = true;
    }
    cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { set_error("plan tables: %s", cudaGetErrorString(e)); st_ = BK_ERR_CUDA; break; }
  } while (0);
  if (st_ != BK_OK) {
    plan_destroy(p);
    return st_;
  }
  *out = p;
  return BK_OK;
}

void plan_destroy(Plan* p) {
  if (!p) return;
  dfree(p->w64);
  dfree(p->wT);
  dfree(p->tw);
  dfree(p->stwS);
  free_fs(p->fs);
  free_fs(p->fsM);
  dfree(p->chirp);
  dfree(p->bh);
  dfree(p->bsc);
  dfree(p->tpost);
  dfree(p->rk);
  dfree(p->scrA);
  dfree(p->scrY);
  dfree(p->scrG);
  dfree(p->part);
  dfree(p->guest);
  dfree(p->t_nodes);
  dfree(p->dA[0]);
  dfree(p->dA[1]);
  dfree(p->derr);
  dfree(p->dpart);
  dfree(p->dcnt);
  delete p;
}
#endif  // BK_TRANSFORM_KERNEL_UNIT

// One length-M complex FFT on the plan's Bluestein layout: src (M complex per vector, as real
// pairs) -> dst (same), through the four-step scratch A; E = EP_CPLX_MC multiplies by the
// spectral table and conjugates in the store.
template <typename T, int E, typename F>
static bk_status blue_fft_F(const Plan* p, const T* src, T* dst, typename V2<T>::t* A, int nvec, cudaStream_t st) {
  typedef typename V2<T>::t C;
  const FourStep& f = p->fsM;
  const int M = (int)p->M;
  BK_TRY(launch(k_passA<T, F>, dim3(f.N2 / f.NB, nvec), f.thrA, f.smemA, st, src, 2 * (int64_t)M, A, M, f.N1, ilog2(f.N1),
                f.N2, f.NB, f.bsA, (const C*)f.stw1, (const C*)f.twN, (const C*)f.twLo, (const C*)f.twHi, f.tw_h));
  BK_TRY(launch(k_passB<T, E, F>, dim3(f.N1 / 2 / f.P, nvec), f.thrB, f.smemB, st, A, dst, 2 * (int64_t)M, M, f.N1, f.N2,
                ilog2(f.N2), f.P, (const C*)f.stw2, (const C*)p->bh));
  return BK_OK;
}
template <typename T, int E>
static bk_status blue_fft(const Plan* p, const T* src, T* dst, typename V2<T>::t* A, int nvec, cudaStream_t st) {
  if constexpr (sizeof(T) == 8) {
    if (p->fe == 2) return blue_fft_F<T, E, FftShape<T, 2>>(p, src, dst, A, nvec, st);
  }
  return blue_fft_F<T, E, FftShape<T, 4>>(p, src, dst, A, nvec, st);
}

// One DCT-I of length N + 1 for N not a power of two: chirp, FFT_M, spectral product, FFT_M,
// chirp and real split (k_bs_pre, blue_fft x 2, k_bs_post).
template <typename T, int K, int E>
static bk_status blue_dct(const Plan* p, const T* src, int64_t sstride, T* dst, int64_t dstride,
                          int64_t zero_to, int nvec, T s, T invN, cudaStream_t st) {
  typedef typename V2<T>::t C;
  const int64_t M = p->M;
  const int N = (int)p->N;
  T* Ma = (T*)p->scrA;
  C* Mb = (C*)(Ma + 2 * M * (int64_t)p->n_comp * p->max_batch);
  const int gp = (int)std::min<int64_t>(1024, (M + 255) / 256);
  BK_TRY(launch(k_bs_pre<T, K>, dim3(gp, nvec), 256, 0, st, src, sstride, N, M, (const C*)p->chirp, Ma));
  BK_TRY((blue_fft<T, EP_CPLX_MC>(p, Ma, Ma, Mb, nvec, st)));
  BK_TRY((blue_fft<T, EP_CPLX>(p, Ma, Ma, Mb, nvec, st)));
  const int gq = (int)std::min<int64_t>(1024, (N / 2 + 256) / 256);
  BK_TRY(launch(k_bs_post<T, E>, dim3(gq, nvec), 256, 0, st, Ma, M, N, (const C*)p->chirp, (const C*)p->tpost, dst, dstride,
                                                  zero_to, s, invN));
  return BK_OK;
}

// The spectral table of a Bluestein plan: bh = FFT_M(b) / M (b from k_bs_kernel, already
// scaled), through the plan's own FFT passes (scratch: the plan's two M-vectors).
template <typename T>
bk_status blue_spectrum(Plan* p, cudaStream_t st) {
  typedef typename V2<T>::t C;
  const int64_t M = p->M;
  T* Ma = (T*)p->scrA;
  C* Mb = (C*)(Ma + 2 * M * (int64_t)p->n_comp * p->max_batch);
  k_bs_kernel<T><<<(int)std::min<int64_t>((M + 255) / 256, 4096), 256, 0, st>>>(Ma, p->N, M);
  BK_CHECK_LAUNCH();
  BK_TRY((blue_fft<T, EP_CPLX>(p, Ma, (T*)p->bh, Mb, 1, st)));
  return BK_OK;
}

template <typename T>
static ReArgs<T> re_args(const Plan* p) {
  typedef typename V2<T>::t C;
  const FourStep& f = p->fs;
  ReArgs<T> g;
  g.N = (int)p->N;
  g.N1 = f.N1;
  g.N2 = f.N2;
  g.log2N1 = ilog2(f.N1);
  g.log2N2 = ilog2(f.N2);
  g.RS = f.RS();
  g.stw1 = (const C*)f.stw1;
  g.stw2 = (const C*)f.stw2;
  g.twA = (const C*)f.twN;
  g.rk = (const T*)p->rk;
  g.cE = (T)(2.0 / ((double)p->N + 1.0));
  g.nst1 = p->nst1;
  g.nst2 = p->nst2;
  memcpy(g.rad1, p->rad1, sizeof(g.rad1));
  memcpy(g.rad2, p->rad2, sizeof(g.rad2));
  return g;
}

// Launch-per-pass form: one pass A and one pass B launch over nvec vectors.
template <typename T, int K, typename F, typename S>
static bk_status re_launch_AF(const Plan* p, const S* src, int64_t sstride, int nvec, cudaStream_t st) {
  typedef typename V2<T>::t C;
  const FourStep& f = p->fs;
  BK_TRY(launch(k_re_passA<T, K, F, S>, dim3(nvec, (f.pairs() + f.NB - 1) / f.NB), f.thrA, f.smemA, st, 
      re_args<T>(p), f.NB, f.bsA, src, sstride, (C*)p->scrA, f.a_len(), (T*)p->part));
  return BK_OK;
}
template <typename T, int K, typename S>
static bk_status re_launch_A(const Plan* p, const S* src, int64_t sstride, int nvec, cudaStream_t st) {
  if constexpr (!std::is_same<T, dfl>::value) {
    if (p->mix) return re_launch_AF<T, K, MixFft>(p, src, sstride, nvec, st);
  }
  if constexpr (sizeof(T) == 4) {
    if (p->fe == 4) return re_launch_AF<T, K, FftShape<T, 4>>(p, src, sstride, nvec, st);
    return re_launch_AF<T, K, FftShape<T, 2>>(p, src, sstride, nvec, st);
  } else {
    return re_launch_AF<T, K, FftShape<T, std::is_same<T, dfl>::value ? 3 : 2>>(p, src, sstride, nvec, st);
  }
}

template <typename T, int E, typename F, typename S>
static bk_status re_launch_BF(const Plan* p, S* dst, int64_t dstride, int64_t zero_to, int nvec, T s, cudaStream_t st) {
  typedef typename V2<T>::t C;
  const FourStep& f = p->fs;
  BK_TRY(launch(k_re_passB<T, E, F, S>, dim3(nvec, (f.N1 / 4 + f.P) / f.P), f.thrB, f.smemB, st, 
      re_args<T>(p), f.P, f.bsB, (const C*)p->scrA, f.a_len(), dst, dstride, zero_to, (const T*)p->part, s,
      T(1.0 / (double)p->N)));
  return BK_OK;
}
template <typename T, int E, typename S>
static bk_status re_launch_B(const Plan* p, S* dst, int64_t dstride, int64_t zero_to, int nvec, T s, cudaStream_t st) {
  if constexpr (!std::is_same<T, dfl>::value) {
    if (p->mix) return re_launch_BF<T, E, MixFft>(p, dst, dstride, zero_to, nvec, s, st);
  }
  if constexpr (sizeof(T) == 4) {
    if (p->fe == 4) return re_launch_BF<T, E, FftShape<T, 4>>(p, dst, dstride, zero_to, nvec, s, st);
    return re_launch_BF<T, E, FftShape<T, 2>>(p, dst, dstride, zero_to, nvec, s, st);
  } else {
    if (re_big(p->fs, p->dtype)) return re_launch_BF<T, E, BigFft<T>>(p, dst, dstride, zero_to, nvec, s, st);
    return re_launch_BF<T, E, FftShape<T, std::is_same<T, dfl>::value ? 3 : 2>>(p, dst, dstride, zero_to, nvec, s, st);
  }
}

template <typename T>
static ReJob<T> re_job(const Plan* p, const void* in, void* out, int nvec, T s) {
  ReJob<T> J;
  J.g = re_args<T>(p);
  J.in = (const Us<T>*)in;
  J.out = (Us<T>*)out;
  J.pitch = p->pitch;
  J.astride = p->fs.a_len();
  J.ystride = p->N + 2;
  J.A = (typename V2<T>::t*)p->scrA;
  J.Y = (T*)p->scrY;
  J.part = (T*)p->part;
  J.s = s;
  J.invN = T(1.0 / (double)p->N);
  J.NB = p->fs.NB;
  J.bsA = p->fs.bsA;
  J.P = p->fs.P;
  J.bsB = p->fs.bsB;
  J.nvec = nvec;
  J.ex = p->cex;
  J.exY = p->cexY;
  J.exP = p->cexP;
  J.csz = p->csize;
  return J;
}

template <typename T>
bk_status apply_impl(const Plan* p, const Us<T>* v, Us<T>* out, int nvec, bool trans, double s_scale, cudaStream_t st) {
  typedef typename V2<T>::t C;
  const int N = (int)p->N;
  const T s = (T)s_scale;
  if constexpr (!std::is_same<T, dfl>::value) {
    const T invN = T(1.0 / (double)N);
    StencilTab<T> tb;
    tb.rk = (const T*)p->rk;
    tb.cN = (T)(1.0 / (4.0 * ((double)N * (double)N - 1.0)));
    if (p->small)
      return launch(trans ? k_birkhoff_small<T, true> : k_birkhoff_small<T, false>, nvec, p->thrS, p->smemS, st, v, out,
                    N, ilog2(N), p->pitch, s, (const C*)p->tw, (const C*)p->stwS, (const C*)p->tpost, tb);
    if (p->blue) {
      const int64_t Ls = N + 1;
      T* Ystage = (T*)p->scrY;
      T* Gst = (T*)p->scrG;
      const dim3 gS((unsigned)std::min<int64_t>(1024, (N + 255) / 256), nvec);
      if (!trans) {
        BK_TRY((blue_dct<T, IN_PLAIN, EP_STORE>(p, v, p->pitch, Ystage, Ls, 0, nvec, s, invN, st)));
        BK_TRY(launch(k_stencil<T, ST_FWD>, gS, 256, 0, st, Ystage, Ls, Gst, N, T(1), tb));
        BK_TRY((blue_dct<T, IN_PLAIN, EP_FWD_OUT>(p, Gst, Ls, out, p->pitch, p->pitch, nvec, s, invN, st)));
      } else {
        BK_TRY((blue_dct<T, IN_WINV, EP_STORE_TRN>(p, v, p->pitch, Ystage, Ls, 0, nvec, s, invN, st)));
        BK_TRY(launch(k_stencil<T, ST_TRN>, gS, 256, 0, st, Ystage, Ls, Gst, N, T(1), tb));
        BK_TRY((blue_dct<T, IN_PLAIN, EP_TRN_OUT>(p, Gst, Ls, out, p->pitch, p->pitch, nvec, s, invN, st)));
      }
      return BK_OK;
    }
    if (!p->split)
      return launch_cl(p->csize, trans ? k_re_cluster<T, true> : k_re_cluster<T, false>, nvec * p->csize, p->cthr,
                       p->csmem, st, re_job<T>(p, v, out, nvec, s), p->csize);
  }
  T* Y = (T*)p->scrY;
  const int64_t Ls = (int64_t)N + 2;   // even: pass A reads aligned pairs
  if (!trans) {
    BK_TRY((re_launch_A<T, IN_PLAIN>(p, v, p->pitch, nvec, st)));
    BK_TRY((re_launch_B<T, EP_STORE>(p, Y, Ls, 0, nvec, s, st)));
    BK_TRY((re_launch_A<T, ST_FWD>(p, (const T*)Y, Ls, nvec, st)));
    BK_TRY((re_launch_B<T, EP_FWD_OUT>(p, out, p->pitch, p->pitch, nvec, s, st)));
  } else {
    BK_TRY((re_launch_A<T, IN_WINV>(p, v, p->pitch, nvec, st)));
    BK_TRY((re_launch_B<T, EP_STORE_TRN>(p, Y, Ls, 0, nvec, s, st)));
    BK_TRY((re_launch_A<T, ST_TRN>(p, (const T*)Y, Ls, nvec, st)));
    BK_TRY((re_launch_B<T, EP_TRN_OUT>(p, out, p->pitch, p->pitch, nvec, s, st)));
  }
  return BK_OK;
}

// Batched products of plans of one precision T (binary32 or binary64 arithmetic): the small
// plans' chains in one launch, the four-step plans' chains in another or their passes in one launch
// each, per chunk of BATCH_MAX plans. Each plan uses its own tables and scratch, so a plan appears at most once among
// the four-step ones (the caller checks). vec[i] / out[i]: nv[i] vectors pitch apart.
template <typename T>
static bk_status launch_small_batch(const Plan* const* ps, const void* const* vin, void* const* vout, const int* nv,
                                    int n, bool trans, cudaStream_t st) {
  typedef typename V2<T>::t C;
  for (int c0 = 0; c0 < n; c0 += BATCH_MAX) {
    Batch<SmallJob<T>> b;
    memset(&b, 0, sizeof(b));
    b.njob = std::min(BATCH_MAX, n - c0);
    int thr = 32;
    size_t smem = 0;
    int cta = 0;
    for (int q = 0; q < b.njob; ++q) {
      const Plan* p = ps[c0 + q];
      SmallJob<T>& J = b.j[q];
      J.in = (const T*)vin[c0 + q];
      J.out = (T*)vout[c0 + q];
      J.pitch = p->pitch;
      J.tw = (const C*)p->tw;
      J.stw = (const C*)p->stwS;
      J.tpost = (const C*)p->tpost;
      J.tb.rk = (const T*)p->rk;
      J.tb.cN = (T)(1.0 / (4.0 * ((double)p->N * (double)p->N - 1.0)));
      J.s = (T)p->s;
      J.N = (int)p->N;
      J.log2N = ilog2(p->N);
      J.nblk = 1;
      b.start[q] = cta;
      cta += nv[c0 + q];
      thr = std::max(thr, p->thrS);
      smem = std::max(smem, p->smemS);
    }
    b.start[b.njob] = cta;
    BK_TRY(launch(trans ? k_small_batch<T, true> : k_small_batch<T, false>, cta, thr, smem, st, b));
  }
  return BK_OK;
}

template <typename T>
static bk_status launch_fourstep_batch(const Plan* const* ps, const void* const* vin, void* const* vout, const int* nv,
                                       int n, bool trans, cudaStream_t st) {
  for (int c0 = 0; c0 < n; c0 += BATCH_MAX) {
    Batch<ReJob<T>> b;
    memset((void*)&b, 0, sizeof(b));
    b.njob = std::min(BATCH_MAX, n - c0);
    int thr = 32, cs = 1, cl = 0;
    size_t smem = 0;
    for (int q = 0; q < b.njob; ++q) {
      const Plan* p = ps[c0 + q];
      b.j[q] = re_job<T>(p, vin[c0 + q], vout[c0 + q], nv[c0 + q], (T)p->s);
      b.start[q] = cl;
      cl += nv[c0 + q];
      thr = std::max(thr, p->cthr);
      cs = std::max(cs, p->csize);
      smem = std::max(smem, p->csmem);
    }
    b.start[b.njob] = cl;
    BK_TRY(launch_cl(cs, trans ? k_re_cluster_batch<T, true> : k_re_cluster_batch<T, false>, cl * cs, thr, smem, st, b, cs));
  }
  return BK_OK;
}

// Four-step plans of radix 4 in the launch-per-pass form, one launch per pass for all of them. guest[i]:
// scratch for entry i when its plan has none of its own (FP32 one-launch plans), else null.
template <typename T, bool TRANS>
static bk_status launch_passes_batch(const Plan* const* ps, const void* const* vin, void* const* vout, const int* nv,
                                     unsigned char* const* guest, int n, cudaStream_t st) {
  typedef FftShape<T, 2> F;
  for (int c0 = 0; c0 < n; c0 += BATCH_MAX) {
    Batch<ReJob<T>> a, b;
    memset((void*)&a, 0, sizeof(a));
    a.njob = std::min(BATCH_MAX, n - c0);
    b = a;
    int thrA = 32, thrB = 32, ca = 0, cb = 0;
    size_t smA = 0, smB = 0;
    for (int q = 0; q < a.njob; ++q) {
      const Plan* p = ps[c0 + q];
      const FourStep& f = p->fs;
      ReJob<T>& J = a.j[q];
      J = re_job<T>(p, vin[c0 + q], vout[c0 + q], nv[c0 + q], (T)p->s);
      if (guest[c0 + q]) {   // laid out as re_scratch_f32 counts it
        unsigned char* m = guest[c0 + q];
        J.A = reinterpret_cast<typename V2<T>::t*>(m);
        m += align256(2 * sizeof(T) * (size_t)J.astride * J.nvec);
        J.Y = reinterpret_cast<T*>(m);
        J.part = reinterpret_cast<T*>(m + align256(sizeof(T) * (size_t)J.ystride * J.nvec));
      }
      b.j[q] = J;
      a.start[q] = ca;
      b.start[q] = cb;
      ca += nv[c0 + q] * ((f.pairs() + f.NB - 1) / f.NB);
      cb += nv[c0 + q] * ((f.N1 / 4 + f.P) / f.P);
      // a one-launch plan's threads and shared memory before its exchange area hold either pass's tiles
      thrA = std::max(thrA, p->split ? f.thrA : p->cthr);
      thrB = std::max(thrB, p->split ? f.thrB : p->cthr);
      smA = std::max(smA, p->split ? f.smemA : (size_t)p->cex);
      smB = std::max(smB, p->split ? f.smemB : (size_t)p->cex);
    }
    a.start[a.njob] = ca;
    b.start[b.njob] = cb;
    BK_TRY(launch(k_re_passA_batch<T, TRANS, false, F>, ca, thrA, smA, st, a));
    BK_TRY(launch(k_re_passB_batch<T, TRANS, false, F>, cb, thrB, smB, st, b));
    BK_TRY(launch(k_re_passA_batch<T, TRANS, true, F>, ca, thrA, smA, st, a));
    BK_TRY(launch(k_re_passB_batch<T, TRANS, true, F>, cb, thrB, smB, st, b));
  }
  return BK_OK;
}

// fs_*: the four-step plans of radix 4. With launch-per-pass plans among them, FP32 one-launch plans
// join those launches on scratch that these plans lend (the same radix and arithmetic, so the same
// results; beside the longer plans they take no time of their own: sizes 2^8..2^16 of 4 FP32
// components, before dependent launches, 79 -> 53 us in all); those that find none left, and the FP64
// ones, of another radix, take their one launch.
template <typename T>
bk_status apply_batch_impl(const Plan* const* small_p, const void* const* small_v, void* const* small_o,
                           const int* small_n, int nsmall, const Plan* const* fs_p, const void* const* fs_v,
                           void* const* fs_o, const int* fs_n, int nfs, bool trans, cudaStream_t st) {
  if (nsmall > 0) BK_TRY(launch_small_batch<T>(small_p, small_v, small_o, small_n, nsmall, trans, st));
  std::vector<const Plan*> p[2];   // 0: one launch, 1: launch per pass
  std::vector<const void*> v[2];
  std::vector<void*> o[2];
  std::vector<int> nv[2];
  std::vector<unsigned char*> guest;
  int lender = 0;   // the launch-per-pass plan that lends next, and the bytes it has lent
  size_t lent = 0;
  for (int i = 0; i < nfs; ++i) {
    unsigned char* g = nullptr;
    int w = fs_p[i]->split ? 1 : 0;
    if constexpr (SmallFft<T>::E == FftShape<T, 2>::E) {
      if (w == 0) {
        const size_t need = re_scratch_f32(fs_p[i]->N, fs_n[i]);
        while (lender < nfs && lent + need > fs_p[lender]->guest_bytes) {
          ++lender;
          lent = 0;
        }
        if (lender < nfs) {
          g = static_cast<unsigned char*>(fs_p[lender]->guest) + lent;
          lent += need;
          w = 1;
        }
      }
    }
    p[w].push_back(fs_p[i]); v[w].push_back(fs_v[i]); o[w].push_back(fs_o[i]); nv[w].push_back(fs_n[i]);
    if (w == 1) guest.push_back(g);
  }
  if (!p[0].empty())
    BK_TRY(launch_fourstep_batch<T>(p[0].data(), v[0].data(), o[0].data(), nv[0].data(), (int)p[0].size(), trans, st));
  if (p[1].empty()) return BK_OK;
  return (trans ? launch_passes_batch<T, true> : launch_passes_batch<T, false>)(
      p[1].data(), v[1].data(), o[1].data(), nv[1].data(), guest.data(), (int)p[1].size(), st);
}

#ifndef BK_TRANSFORM_KERNEL_UNIT
extern template bk_status apply_impl<double>(const Plan* p, const double* v, double* out, int nvec, bool trans,
                                             double s_scale, cudaStream_t st);
extern template bk_status apply_impl<float>(const Plan* p, const float* v, float* out, int nvec, bool trans,
                                            double s_scale, cudaStream_t st);
extern template bk_status apply_batch_impl<double>(const Plan* const*, const void* const*, void* const*,
                                                   const int*, int, const Plan* const*, const void* const*,
                                                   void* const*, const int*, int, bool, cudaStream_t);
extern template bk_status apply_batch_impl<float>(const Plan* const*, const void* const*, void* const*, const int*,
                                                  int, const Plan* const*, const void* const*, void* const*,
                                                  const int*, int, bool, cudaStream_t);
extern template bk_status apply_impl<dfl>(const Plan* p, const double* v, double* out, int nvec, bool trans,
                                          double s_scale, cudaStream_t st);

bk_status plan_apply_n(const Plan* p, const void* v, void* out, int nvec, bool trans, double s,
                       cudaStream_t st) {
  if (p->dense) return dense_apply(p, v, out, nvec, trans, s, st);
  if (p->dtype == BK_F64 && p->df)
    return apply_impl<dfl>(p, (const double*)v, (double*)out, nvec, trans, s, st);
  if (p->dtype == BK_F64)
    return apply_impl<double>(p, (const double*)v, (double*)out, nvec, trans, s, st);
  return apply_impl<float>(p, (const float*)v, (float*)out, nvec, trans, s, st);
}

// b-form helpers: c[vec] = out[vec][N] (forward) or s sum_i u[vec][i] (transpose, one block per
// vector, fixed order), then out[vec][i] -= c[vec] (forward) or c[vec] w_i (transpose), i <= N.
template <typename T>
__global__ void k_bform_last(const T* __restrict__ out, int64_t pitch, int64_t N, T* __restrict__ c) {
  pdl_wait();
  if (threadIdx.x == 0) c[blockIdx.x] = out[(int64_t)blockIdx.x * pitch + N];
}
template <typename T>
__global__ void __launch_bounds__(256) k_bform_sum(const T* __restrict__ u, int64_t pitch, int64_t L, double s,
                                                   T* __restrict__ c) {
  pdl_wait();
  __shared__ double red[8];
  const T* x = u + (int64_t)blockIdx.x * pitch;
  double a = 0.0;
  for (int64_t i = threadIdx.x; i < L; i += blockDim.x) a += (double)x[i];
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    c[blockIdx.x] = (T)(s * t);
  }
}
template <typename T>
__global__ void k_bform_sub(T* __restrict__ out, int64_t pitch, int64_t L, const T* __restrict__ c,
                            const T* __restrict__ w) {
  pdl_wait();
  const T cv = c[blockIdx.y];
  T* o = out + (int64_t)blockIdx.y * pitch;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < L; i += (int64_t)gridDim.x * blockDim.x)
    o[i] -= w ? cv * w[i] : cv;
}

template <typename T>
static bk_status apply_b_impl(const Plan* p, const void* v, void* out, int nvec, bool trans, cudaStream_t st) {
  T* c = (T*)p->bsc;
  const dim3 g((unsigned)std::min<int64_t>(1024, (p->L + 255) / 256), nvec);
  const T* w = p->dtype == BK_F64 ? (const T*)p->w64 : (const T*)p->wT;
  if (trans) {
    // the sum first: v may alias out
    BK_TRY(launch(k_bform_sum<T>, nvec, 256, 0, st, (const T*)v, p->pitch, p->L, p->s, c));
    BK_TRY(plan_apply_n(p, v, out, nvec, true, p->s, st));
    BK_TRY(launch(k_bform_sub<T>, g, 256, 0, st, (T*)out, p->pitch, p->L, c, w));
  } else {
    BK_TRY(plan_apply_n(p, v, out, nvec, false, p->s, st));
    BK_TRY(launch(k_bform_last<T>, nvec, 32, 0, st, (const T*)out, p->pitch, p->N, c));
    BK_TRY(launch(k_bform_sub<T>, g, 256, 0, st, (T*)out, p->pitch, p->L, c, nullptr));
  }
  return BK_OK;
}

bk_status plan_apply_b(const Plan* p, const void* v, void* out, int batch, bool trans, cudaStream_t st) {
  BK_ARG(p != nullptr, "plan is NULL");
  BK_ARG(v != nullptr && out != nullptr, "NULL vector");
  BK_ARG(batch >= 1 && batch <= p->max_batch, "batch %d outside [1, max_batch=%d]", batch, p->max_batch);
  BK_ARG(((uintptr_t)v & 15) == 0 && ((uintptr_t)out & 15) == 0, "vectors must be 16-byte aligned");
  const int nvec = batch * p->n_comp;
  return p->dtype == BK_F64 ? apply_b_impl<double>(p, v, out, nvec, trans, st)
                            : apply_b_impl<float>(p, v, out, nvec, trans, st);
}

bk_status plan_apply(const Plan* p, const void* v, void* out, int batch, bool trans, cudaStream_t st) {
  BK_ARG(p != nullptr, "plan is NULL");
  BK_ARG(v != nullptr && out != nullptr, "NULL vector");
  BK_ARG(batch >= 1 && batch <= p->max_batch, "batch %d outside [1, max_batch=%d]", batch, p->max_batch);
  BK_ARG(((uintptr_t)v & 15) == 0 && ((uintptr_t)out & 15) == 0, "vectors must be 16-byte aligned");
  return plan_apply_n(p, v, out, batch * p->n_comp, trans, p->s, st);
}

// Products of several plans of one precision, N free per plan: small plans in one launch, four-step
// plans of radix 4 in another, or in one launch per pass where one of them needs it (each per
// BATCH_MAX plans), every other plan (dense, Bluestein, radix 8 and 16) by its own launches. The shared
// launches use a four-step plan's scratch once, so a plan that has some comes in them once; the later
// entries of an FP64 plan of N >= 2^17 follow as launches of their own, those of a shorter one are refused.
bk_status plan_apply_batch(const Plan* const* ps, const void* const* v, void* const* out, const int* batch, int count,
                           bool trans, cudaStream_t st) {
  BK_ARG(ps != nullptr && v != nullptr && out != nullptr && batch != nullptr, "NULL argument");
  BK_ARG(count >= 1 && count <= 4096, "count %d outside [1, 4096]", count);
  BK_ARG(ps[0] != nullptr, "plan 0 is NULL");
  const int dtype = ps[0]->dtype;
  std::vector<const Plan*> sp, fp, op;
  std::vector<const void*> sv, fv, ov;
  std::vector<void*> so, fo, oo;
  std::vector<int> sn, fn, on;
  for (int i = 0; i < count; ++i) {
    const Plan* p = ps[i];
    BK_ARG(p != nullptr, "plan %d is NULL", i);
    BK_ARG(p->dtype == dtype, "plan %d: every plan of a batch has the same dtype", i);
    BK_ARG(v[i] != nullptr && out[i] != nullptr, "entry %d: NULL vector", i);
    BK_ARG(batch[i] >= 1 && batch[i] <= p->max_batch, "entry %d: batch %d outside [1, max_batch=%d]", i, batch[i],
           p->max_batch);
    BK_ARG(((uintptr_t)v[i] & 15) == 0 && ((uintptr_t)out[i] & 15) == 0, "entry %d: vectors must be 16-byte aligned",
           i);
    const int nv = batch[i] * p->n_comp;
    if (p->dense || p->blue || p->df || (p->split && p->fe != 2)) {
      op.push_back(p); ov.push_back(v[i]); oo.push_back(out[i]); on.push_back(nv);
    } else if (p->small) {
      sp.push_back(p); sv.push_back(v[i]); so.push_back(out[i]); sn.push_back(nv);
    } else {
      // FP32 one-launch plans have no scratch to share
      const bool again = (p->split || dtype == BK_F64) && std::find(fp.begin(), fp.end(), p) != fp.end();
      if (again && dtype == BK_F64 && p->N >= (int64_t(1) << 17)) {   // as the double-float plans of that size
        op.push_back(p); ov.push_back(v[i]); oo.push_back(out[i]); on.push_back(nv);
        continue;
      }
      BK_ARG(!again, "entry %d: a four-step plan may appear once per batch (its scratch)", i);
      fp.push_back(p); fv.push_back(v[i]); fo.push_back(out[i]); fn.push_back(nv);
    }
  }
  if (dtype == BK_F64)
    BK_TRY(apply_batch_impl<double>(sp.data(), sv.data(), so.data(), sn.data(), (int)sp.size(), fp.data(), fv.data(),
                                    fo.data(), fn.data(), (int)fp.size(), trans, st));
  else
    BK_TRY(apply_batch_impl<float>(sp.data(), sv.data(), so.data(), sn.data(), (int)sp.size(), fp.data(), fv.data(),
                                   fo.data(), fn.data(), (int)fp.size(), trans, st));
  for (size_t k = 0; k < op.size(); ++k) BK_TRY(plan_apply_n(op[k], ov[k], oo[k], on[k], trans, op[k]->s, st));
  return BK_OK;
}

#endif  // BK_TRANSFORM_KERNEL_UNIT
}  // namespace bk

#ifndef BK_TRANSFORM_KERNEL_UNIT

namespace bk {

// ---------------------------------------------------------------------------------------------
// Allocation-free variant of the four-step forward product.
//
// For callers that must not allocate device memory once they run: real-time or flight control
// loops with a memory budget fixed at start-up, and host programs whose own allocator owns the
// device. They cannot create a bk_plan (plan creation allocates tables and scratch). This
// variant keeps its twiddle tables and transform scratch in one file-scope device array of
// NOALLOC_BYTES, reserved on every GPU that loads the library until the process exits.
// ---------------------------------------------------------------------------------------------
static constexpr size_t NOALLOC_BYTES = size_t(16) << 20;   // 16 MiB
static constexpr int NOALLOC_MAX_DEV = 64;
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

// Device address of g_noalloc_scratch per device (host code cannot use the symbol itself).
static void* g_noalloc_ptr[NOALLOC_MAX_DEV] = {nullptr};
static std::mutex g_noalloc_mu;

// Bytes of the scratch layout for N (FP64) and nvec vectors, and the sub-buffer offsets.
static size_t noalloc_layout(const Plan& p, int nvec, size_t off[7]) {
  const int64_t N = p.N;
  size_t o = 0;
  off[0] = o; o += align256(sizeof(double2) * stage_tw_len(ilog2(p.fs.N1), 2));  // stw1
  off[1] = o; o += align256(sizeof(double2) * stage_tw_len(ilog2(p.fs.N2), 2));  // stw2
  off[2] = o; o += align256(sizeof(double2) * p.fs.a_len());                          // twN
  off[3] = o; o += align256(sizeof(double2) * p.fs.a_len() * nvec);                   // scrA
  off[4] = o; o += align256(sizeof(double) * (size_t)(N + 2) * nvec);                 // scrY
  off[5] = o; o += align256(sizeof(double) * (size_t)p.fs.pairs() * nvec);            // part
  off[6] = o; o += align256(sizeof(double) * (size_t)(N + 2));                        // rk
  return o;
}

// Per-device set-up: device address of the scratch array and the shared-memory attributes of
// the pass kernels. Runs on the first call on each device.
static bk_status noalloc_setup(int dev, void** out) {
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (g_noalloc_ptr[dev] == nullptr) {
    void* ptr = nullptr;
    BK_TRY_CUDA(cudaGetSymbolAddress(&ptr, g_noalloc_scratch));
    BK_TRY(re_attrs<double>());
    g_noalloc_ptr[dev] = ptr;
  }
  *out = g_noalloc_ptr[dev];
  return BK_OK;
}

bk_status noalloc_apply(const double* v, double* out, int64_t N, int nvec, int64_t pitch, double t0, double tf,
                        cudaStream_t st) {
  BK_ARG(v != nullptr && out != nullptr, "NULL vector");
  BK_ARG(is_pow2(N) && N >= 8192 && N <= 65536, "N must be a power of two in [8192, 65536], got %lld", (long long)N);
  BK_ARG(nvec >= 1 && nvec <= 8, "nvec must be in [1, 8], got %d", nvec);
  BK_ARG(pitch >= N + 1 && pitch % 2 == 0, "pitch must be >= N + 1 and even");
  BK_ARG(tf != t0 && isfinite(t0) && isfinite(tf), "tf must differ from t0 and both be finite");
  BK_ARG(((uintptr_t)v & 15) == 0 && ((uintptr_t)out & 15) == 0, "vectors must be 16-byte aligned");
  {
    // shifted ranges would have one vector's output over another's input, and this entry point has no
    // in-place form
    const uintptr_t vb = (uintptr_t)v, ob = (uintptr_t)out, span = sizeof(double) * (uintptr_t)pitch * nvec;
    BK_ARG(vb + span <= ob || ob + span <= vb, "v and out overlap");
  }
  int dev = 0;
  BK_TRY_CUDA(cudaGetDevice(&dev));
  BK_ARG(dev >= 0 && dev < NOALLOC_MAX_DEV, "device index %d not supported", dev);
  Plan p;  // configuration only; owns nothing
  p.N = N;
  p.L = N + 1;
  p.pitch = pitch;
  p.n_comp = nvec;
  p.max_batch = 1;
  p.dtype = BK_F64;
  p.t0 = t0;
  p.tf = tf;
  p.s = 0.5 * (tf - t0);
  p.small = false;
  p.split = 1;
  BK_TRY(configure_re(p.fs, N, BK_F64, 2, nvec));
  size_t off[7];
  const size_t need = noalloc_layout(p, nvec, off);
  BK_ARG(need <= NOALLOC_BYTES, "N=%lld with %d vectors needs %zu bytes of scratch, more than the %zu reserved",
         (long long)N, nvec, need, NOALLOC_BYTES);
  void* base = nullptr;
  BK_TRY(noalloc_setup(dev, &base));
  unsigned char* b = (unsigned char*)base;
  p.fs.stw1 = b + off[0];
  p.fs.stw2 = b + off[1];
  p.fs.twN = b + off[2];
  p.scrA = b + off[3];
  p.scrY = b + off[4];
  p.part = b + off[5];
  p.rk = b + off[6];
  // every table is rewritten by each call: nothing in the array has to start at zero
  k_rk_table<double><<<(int)std::min<int64_t>((N + 2 + 255) / 256, 4096), 256, 0, st>>>((double*)p.rk, N + 2);
  BK_CHECK_LAUNCH();
  constexpr int e = 2;
  const int len1 = stage_tw_len(ilog2(p.fs.N1), e), len2 = stage_tw_len(ilog2(p.fs.N2), e);
  k_stage_tw<double><<<(len1 + 255) / 256, 256, 0, st>>>((double2*)p.fs.stw1, ilog2(p.fs.N1), e, len1);
  BK_CHECK_LAUNCH();
  k_stage_tw<double><<<(len2 + 255) / 256, 256, 0, st>>>((double2*)p.fs.stw2, ilog2(p.fs.N2), e, len2);
  BK_CHECK_LAUNCH();
  k_re_tw<double><<<re_tw_blocks(p.fs), 256, 0, st>>>((double2*)p.fs.twN, p.fs.N1, p.fs.N2);
  BK_CHECK_LAUNCH();
  return apply_impl<double>(&p, v, out, nvec, false, p.s, st);
}

}  // namespace bk

// ---------------------------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------------------------
extern "C" {

const char* bk_last_error(void) { return bk::g_last_error.c_str(); }
const char* bk_version(void) { return "birkhoff-gb300 0.1 (sm_103a)"; }
uint64_t bk_launch_count(void) { return bk::g_launches.load(); }

bk_status bk_plan_create(bk_plan** plan, int64_t N, int n_comp, int max_batch, bk_dtype dtype,
                         double t0, double tf, int64_t pitch, void* stream) {
  BK_ARG(plan != nullptr, "plan output pointer is NULL");
  bk::Plan* p = nullptr;
  bk_status s = bk::plan_create(&p, N, n_comp, max_batch, (int)dtype, t0, tf, pitch, (cudaStream_t)stream);
  *plan = reinterpret_cast<bk_plan*>(p);
  return s;
}

void bk_plan_destroy(bk_plan* plan) { bk::plan_destroy(reinterpret_cast<bk::Plan*>(plan)); }

bk_status bk_plan_info(const bk_plan* plan, int64_t* N, int64_t* L, int64_t* pitch, int* dtype) {
  BK_ARG(plan != nullptr, "plan is NULL");
  const bk::Plan* p = reinterpret_cast<const bk::Plan*>(plan);
  if (N) *N = p->N;
  if (L) *L = p->L;
  if (pitch) *pitch = p->pitch;
  if (dtype) *dtype = p->dtype;
  return BK_OK;
}

bk_status bk_plan_grid(const bk_plan* plan, double* t_host, double* w_host) {
  BK_ARG(plan != nullptr, "plan is NULL");
  const bk::Plan* p = reinterpret_cast<const bk::Plan*>(plan);
  if (t_host) BK_TRY_CUDA(cudaMemcpy(t_host, p->t_nodes, sizeof(double) * p->L, cudaMemcpyDeviceToHost));
  if (w_host) BK_TRY_CUDA(cudaMemcpy(w_host, p->w64, sizeof(double) * p->L, cudaMemcpyDeviceToHost));
  return BK_OK;
}

bk_status birkhoff_apply(const bk_plan* plan, const void* v, void* out, int batch, void* stream) {
  return bk::plan_apply(reinterpret_cast<const bk::Plan*>(plan), v, out, batch, false, (cudaStream_t)stream);
}

bk_status birkhoff_apply_noalloc(const double* v, double* out, int64_t N, int nvec, int64_t pitch, double t0,
                                 double tf, void* stream) {
  return bk::noalloc_apply(v, out, N, nvec, pitch, t0, tf, (cudaStream_t)stream);
}

bk_status birkhoff_apply_b(const bk_plan* plan, const void* v, void* out, int batch, void* stream) {
  return bk::plan_apply_b(reinterpret_cast<const bk::Plan*>(plan), v, out, batch, false, (cudaStream_t)stream);
}

bk_status birkhoff_apply_b_T(const bk_plan* plan, const void* v, void* out, int batch, void* stream) {
  return bk::plan_apply_b(reinterpret_cast<const bk::Plan*>(plan), v, out, batch, true, (cudaStream_t)stream);
}

bk_status birkhoff_apply_batch(const bk_plan* const* plans, const void* const* v, void* const* out, const int* batch,
                               int count, int trans, void* stream) {
  return bk::plan_apply_batch(reinterpret_cast<const bk::Plan* const*>(plans), v, out, batch, count, trans != 0,
                              (cudaStream_t)stream);
}

bk_status birkhoff_apply_T(const bk_plan* plan, const void* v, void* out, int batch, void* stream) {
  return bk::plan_apply(reinterpret_cast<const bk::Plan*>(plan), v, out, batch, true, (cudaStream_t)stream);
}

bk_status bk_plan_set_dense(bk_plan* plan, int on, void* stream) {
  BK_ARG(plan != nullptr, "plan is NULL");
  bk::Plan* p = reinterpret_cast<bk::Plan*>(plan);
  if (!on) {
    if (p->generic) {
      bk::set_error("N = %lld is not a power of two: the plan has no FFT path", (long long)p->N);
      return BK_ERR_UNSUPPORTED;
    }
    p->dense = false;
    return BK_OK;
  }
  if (!bk::dense_supported(p->N)) {
    bk::set_error("dense products need N <= 1024 (N = %lld)", (long long)p->N);
    return BK_ERR_UNSUPPORTED;
  }
  if (!p->dA[0]) {
    bk::AllocCounter counter(&p->bytes);
    BK_TRY(bk::dense_build(p, (cudaStream_t)stream));
  }
  p->dense = true;
  return BK_OK;
}

bk_status bk_plan_shape(const bk_plan* plan, int* path, int* N1, int* N2, int* elems) {
  BK_ARG(plan != nullptr, "plan is NULL");
  const bk::Plan* p = reinterpret_cast<const bk::Plan*>(plan);
  const int pth = p->dense ? 3 : (p->blue ? 4 : (p->small ? 0 : (p->split ? 2 : 1)));
  if (path) *path = pth;
  if (N1) *N1 = (pth == 1 || pth == 2) ? p->fs.N1 / 2 : 0;
  if (N2) *N2 = (pth == 1 || pth == 2) ? p->fs.N2 / 2 : 0;
  if (elems) *elems = (pth == 1 || pth == 2) ? std::max(p->fs.NB * p->fs.N1, p->fs.P * p->fs.N2) : 0;
  return BK_OK;
}

bk_status bk_set_f64_transform(int mode) {
  BK_ARG(mode == 0 || mode == 1 || mode == -1, "mode must be 0 (FP64), 1 (double-float) or -1 (default)");
  bk::g_f64_df.store(mode);
  return BK_OK;
}

bk_status bk_plan_f64_mode(const bk_plan* plan, int* mode) {
  BK_ARG(plan != nullptr && mode != nullptr, "NULL argument");
  const bk::Plan* p = reinterpret_cast<const bk::Plan*>(plan);
  *mode = p->df ? 1 : 0;
  return BK_OK;
}

bk_status bk_plan_dense_state(const bk_plan* plan, int* on) {
  BK_ARG(plan != nullptr && on != nullptr, "NULL argument");
  *on = reinterpret_cast<const bk::Plan*>(plan)->dense ? 1 : 0;
  return BK_OK;
}

bk_status bk_plan_dense_test_timeout(bk_plan* plan, int on) {
  BK_ARG(plan != nullptr, "plan is NULL");
  reinterpret_cast<bk::Plan*>(plan)->dtest = on ? 1 : 0;
  return BK_OK;
}

bk_status bk_plan_dense_check(const bk_plan* plan, int* err) {
  BK_ARG(plan != nullptr && err != nullptr, "NULL argument");
  const bk::Plan* p = reinterpret_cast<const bk::Plan*>(plan);
  *err = 0;
  if (!p->derr) return BK_OK;
  BK_TRY_CUDA(cudaDeviceSynchronize());
  BK_TRY_CUDA(cudaMemcpy(err, p->derr, sizeof(int), cudaMemcpyDeviceToHost));
  BK_TRY_CUDA(cudaMemset(p->derr, 0, sizeof(int)));
  return BK_OK;
}

}  // extern "C"

#endif  // BK_TRANSFORM_KERNEL_UNIT
