// Shared-memory batched complex FFT used by the DCT-I transforms of the Birkhoff products.
// Forward transform, omega_n = exp(-2 pi i / n).
//
// In-place Stockham autosort with radix 2^E (one smaller mixed-radix stage first when log2 n is not
// a multiple of E). Every thread stages EPT values per stage in registers (EPT / R butterflies of
// radix R), so one buffer suffices: read, barrier, compute, write, barrier. Shared addresses are
// padded, a -> a + a/16; batches sit bs >= n + n/16 + 1 apart.
//
// The radix follows what bounds the kernel. FP64: GB300 issues a warp's FP64 instruction every 64
// cycles per SM sub-partition, whatever its active lanes, and radix 4 needs as many FP64
// instructions per point as radix 16 (28 per 4 points and 2 bits against 220 per 16 points and 4
// bits), so radix 4 with 4 values per thread spreads the same work over four times the warps
// (products of 4 components, radix 16 / radix 4, us: N = 2^10 55 / 27, 2^14 90 / 47, 2^16 122 / 70).
// The few CTAs of the one-CTA and one-launch FP64 kernels go on to radix 2 (2^8 13.0 / 12.0, 2^12 26.4 /
// 23.8 radix 4 / radix 2). FP32 while latency bounds it: radix 4 as well (2^14 35 / 26, 2^16 47 / 31, 2^18 50 / 41); from
// 2^19 on, bound by issue and shared memory: radix 16 (2^20 87 / 81). Double-float: radix 8, whose
// code and registers are half of radix 16's (2^18 130 / 90, 2^20 339 / 260 radix 16 / radix 8).
//
// Twiddles come from a per-size stage table built on the device with sincospi at plan creation:
// for each radix-R stage with Ns > 1 (in stage order) a block stw[off + (r - 1) Ns + k] =
// omega_{R Ns}^{r k}, r = 1..R-1, k < Ns. Lanes hold consecutive k, so a warp reads consecutive
// entries: no shared-memory bank conflicts, coalesced global loads. (Indexing one table of
// omega_n^i by r k instead gave stride-r lane patterns, up to 16-way conflicts.) The table may
// be the global one or a copy in shared memory (load_tw_smem).
#pragma once

#include <type_traits>

#include "bk_common.cuh"

namespace bk {

__device__ __forceinline__ int padi(int a) { return a + (a >> 4); }
__host__ __device__ inline int pad_stride(int n) { return n + (n >> 4) + 1; }

// Entries of the stage twiddle table of a length-2^log2n FFT of radix 2^e (stages with Ns > 1).
__host__ __device__ inline int stage_tw_len(int log2n, int e) {
  int len = 0;
  for (int l = log2n % e ? log2n % e : e; l < log2n; l += e) len += ((1 << e) - 1) << l;
  return len;
}

// Shape of the transform kernels of a type and log2 radix E: values per thread, thread cap and
// resident CTAs per SM they are compiled for (64K registers / (threads x this) per thread).
template <typename T, int E_> struct FftShape {
  static constexpr int E = E_, EPT = 1 << E_, MT = E_ == 4 ? 512 : (E_ == 3 ? 512 : 1024), MINB = MT == 512 ? 2 : 1;
  static constexpr bool MIX = false;
};
template <> struct FftShape<double, 4> {
  static constexpr int E = 4, EPT = 16, MT = 256, MINB = 2;
  static constexpr bool MIX = false;
};
// Launch-per-pass kernels of lengths 2^a 3^b 5^c (fft_mix).
struct MixFft { static constexpr int E = 2, MT = 256, MINB = 2; static constexpr bool MIX = true; };
// Radix of the one-CTA and one-launch kernels, whose few CTAs are bound by latency (re_radix and
// cplx_radix choose that of the launch-per-pass kernels).
template <typename T> struct SmallFft : FftShape<T, sizeof(T) == 8 ? 1 : 2> {};
template <typename T> struct BigFft { static constexpr int E = std::is_same<T, dfl>::value ? 3 : 2, EPT = 16, MT = 512, MINB = 1; static constexpr bool MIX = false; };

// Radix-R DFT of v[0..R-1] in registers (forward, natural order in and out).
template <typename C, typename T, int R> struct Radix;

template <typename C, typename T> struct Radix<C, T, 2> {
  static __device__ __forceinline__ void run(C* v) {
    C a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <typename C, typename T> struct Radix<C, T, 4> {
  static __device__ __forceinline__ void run(C* v) {
    C t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    C t2 = cadd(v[1], v[3]), t3 = cmul_mi(csub(v[1], v[3]));
    v[0] = cadd(t0, t2);
    v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3);
    v[3] = csub(t1, t3);
  }
};

template <typename C, typename T> struct Radix<C, T, 8> {
  static __device__ __forceinline__ void run(C* v) {
    C e[4] = {v[0], v[2], v[4], v[6]};
    C o[4] = {v[1], v[3], v[5], v[7]};
    Radix<C, T, 4>::run(e);
    Radix<C, T, 4>::run(o);
    const T h = T(0.70710678118654752440084436210484903928483593768847);
    // omega_8^1 = (1 - i) h, omega_8^2 = -i, omega_8^3 = -(1 + i) h
    C o1, o2, o3;
    o1.x = h * (o[1].x + o[1].y);
    o1.y = h * (o[1].y - o[1].x);
    o2 = cmul_mi(o[2]);
    o3.x = h * (o[3].y - o[3].x);
    o3.y = -h * (o[3].x + o[3].y);
    v[0] = cadd(e[0], o[0]);
    v[4] = csub(e[0], o[0]);
    v[1] = cadd(e[1], o1);
    v[5] = csub(e[1], o1);
    v[2] = cadd(e[2], o2);
    v[6] = csub(e[2], o2);
    v[3] = cadd(e[3], o3);
    v[7] = csub(e[3], o3);
  }
};

// omega_3 = -1/2 - i sqrt(3)/2.
template <typename C, typename T> struct Radix<C, T, 3> {
  static __device__ __forceinline__ void run(C* v) {
    const T q = T(0.86602540378443864676372317075293618347140262690519);   // sqrt(3) / 2
    const C t = cadd(v[1], v[2]), e = csub(v[1], v[2]);
    C m;
    m.x = v[0].x - T(0.5) * t.x;
    m.y = v[0].y - T(0.5) * t.y;
    v[0] = cadd(v[0], t);
    v[1].x = m.x + q * e.y;
    v[1].y = m.y - q * e.x;
    v[2].x = m.x - q * e.y;
    v[2].y = m.y + q * e.x;
  }
};

// X_1,4 = v0 + c1 a1 + c2 a2 -+ i (s1 b1 + s2 b2), X_2,3 = v0 + c2 a1 + c1 a2 -+ i (s2 b1 - s1 b2)
// with a_j = v_j + v_{5-j}, b_j = v_j - v_{5-j}, c_j + i s_j = e^{2 pi i j / 5}.
template <typename C, typename T> struct Radix<C, T, 5> {
  static __device__ __forceinline__ void run(C* v) {
    const T c1 = T(0.30901699437494742410229341718281905886015458990288);
    const T c2 = T(-0.80901699437494742410229341718281905886015458990288);
    const T s1 = T(0.95105651629515357211643933337938214340569863412575);
    const T s2 = T(0.58778525229247312916870595463907276859765243764314);
    const C a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]), a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
    C t1, t2, u1, u2;
    t1.x = v[0].x + c1 * a1.x + c2 * a2.x;
    t1.y = v[0].y + c1 * a1.y + c2 * a2.y;
    t2.x = v[0].x + c2 * a1.x + c1 * a2.x;
    t2.y = v[0].y + c2 * a1.y + c1 * a2.y;
    u1.x = s1 * b1.x + s2 * b2.x;
    u1.y = s1 * b1.y + s2 * b2.y;
    u2.x = s2 * b1.x - s1 * b2.x;
    u2.y = s2 * b1.y - s1 * b2.y;
    v[0] = cadd(v[0], cadd(a1, a2));
    v[1] = mk2<T>(t1.x + u1.y, t1.y - u1.x);
    v[4] = mk2<T>(t1.x - u1.y, t1.y + u1.x);
    v[2] = mk2<T>(t2.x + u2.y, t2.y - u2.x);
    v[3] = mk2<T>(t2.x - u2.y, t2.y + u2.x);
  }
};

// Radix 16 as 4 x 4: r = r1 + 4 r2, s = s1 + 4 s2,
//   X[s1 + 4 s2] = sum_r1 omega_4^{r1 s2} omega_16^{r1 s1} sum_r2 v[r1 + 4 r2] omega_4^{r2 s1}.
template <typename C, typename T> struct Radix<C, T, 16> {
  static __device__ __forceinline__ void run(C* v) {
    // cos(pi/8) = sqrt(2 + sqrt 2)/2, sin(pi/8) = sqrt(2 - sqrt 2)/2, sqrt(1/2)
    const T c1 = T(0.92387953251128675612818318939678828682241662586364);
    const T s1 = T(0.38268343236508977172845998403039886676134456248563);
    const T h = T(0.70710678118654752440084436210484903928483593768847);
    C y[4][4];
#pragma unroll
    for (int r1 = 0; r1 < 4; ++r1) {
      C t[4] = {v[r1], v[r1 + 4], v[r1 + 8], v[r1 + 12]};
      Radix<C, T, 4>::run(t);
#pragma unroll
      for (int q = 0; q < 4; ++q) y[r1][q] = t[q];
    }
    // internal twiddles omega_16^{r1 s1}, r1, s1 in 1..3 (exponents 1,2,3,2,4,6,3,6,9)
    C a;
    a = y[1][1]; y[1][1].x = c1 * a.x + s1 * a.y; y[1][1].y = c1 * a.y - s1 * a.x;       // w^1
    a = y[1][2]; y[1][2].x = h * (a.x + a.y); y[1][2].y = h * (a.y - a.x);                // w^2
    a = y[1][3]; y[1][3].x = s1 * a.x + c1 * a.y; y[1][3].y = s1 * a.y - c1 * a.x;       // w^3
    a = y[2][1]; y[2][1].x = h * (a.x + a.y); y[2][1].y = h * (a.y - a.x);                // w^2
    y[2][2] = cmul_mi(y[2][2]);                                                           // w^4
    a = y[2][3]; y[2][3].x = h * (a.y - a.x); y[2][3].y = -h * (a.x + a.y);               // w^6
    a = y[3][1]; y[3][1].x = s1 * a.x + c1 * a.y; y[3][1].y = s1 * a.y - c1 * a.x;       // w^3
    a = y[3][2]; y[3][2].x = h * (a.y - a.x); y[3][2].y = -h * (a.x + a.y);               // w^6
    a = y[3][3]; y[3][3].x = -c1 * a.x - s1 * a.y; y[3][3].y = s1 * a.x - c1 * a.y;      // w^9
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      C t[4] = {y[0][q], y[1][q], y[2][q], y[3][q]};
      Radix<C, T, 4>::run(t);
#pragma unroll
      for (int s2 = 0; s2 < 4; ++s2) v[q + 4 * s2] = t[s2];
    }
  }
};

// One in-place stage of radix R (EPT/R butterflies per thread) of a length-2^LOG2N FFT whose
// previous radices multiply to Ns = 2^LOG2NS. Threads t < nbatch * n/EPT work; all threads must
// reach the barriers.
//
// Addressing. padi(a + c) = padi(a) + padi(c) whenever the low four bits do not carry, so with
// n and Ns known at compile time every shared address of a stage is one per-thread base plus an
// immediate offset:
//   reads  tt + q n/EPT + r n/R : offsets that are multiples of 16 (else generic);
//   writes idxD + r Ns, idxD = (j / Ns) R Ns + (j mod Ns): the two terms share no bits;
//   twiddles stw[(r - 1) Ns + k] from stw + k.
template <typename T, int LOG2N, int R, int LOG2NS, int EPT>
__device__ __forceinline__ void stage_ct(typename V2<T>::t* __restrict__ buf, int nbatch, int bs,
                                         const typename V2<T>::t* __restrict__ stw) {
  typedef typename V2<T>::t C;
  constexpr int log2R = R == 16 ? 4 : (R == 8 ? 3 : (R == 4 ? 2 : 1));
  constexpr int log2EPT = EPT == 16 ? 4 : (EPT == 8 ? 3 : (EPT == 4 ? 2 : 1));
  constexpr int PER = EPT / R;
  constexpr int LOG2TP = LOG2N - log2EPT;
  constexpr int nTP = 1 << LOG2TP;
  constexpr int nR = (1 << LOG2N) >> log2R;
  constexpr int Ns = 1 << LOG2NS;
  constexpr bool lin_rd = (nR % 16 == 0) && (PER == 1 || nTP % 16 == 0);
  const int t = threadIdx.x;
  const bool active = t < (nbatch << LOG2TP);
  const int tt = t & (nTP - 1);
  C* base = buf + (size_t)(t >> LOG2TP) * bs;
  C v[EPT];
  if (active) {
    const C* src = base + padi(tt);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int c = q * nTP + r * nR;
        v[q * R + r] = lin_rd ? src[c + (c >> 4)] : base[padi(tt + c)];
      }
    }
  }
  __syncthreads();
  if (active) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int j = tt + q * nTP;
      const int k = j & (Ns - 1);
      C* u = v + q * R;
      if (Ns > 1) {
        const C* tw = stw + k;
#pragma unroll
        for (int r = 1; r < R; ++r) u[r] = cmul(u[r], tw[(r - 1) * Ns]);
      }
      Radix<C, T, R>::run(u);
      C* dst = base + padi(((j >> LOG2NS) << (LOG2NS + log2R)) + k);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int c = r * Ns;
        dst[c + (c >> 4)] = u[r];
      }
    }
  }
  __syncthreads();
}

// Radix-2^E stages from Ns = 2^LOG2NS on; OFF is the stage table offset of the first of them.
template <typename T, int LOG2N, int E, int EPT, int LOG2NS, int OFF>
__device__ __forceinline__ void fft_ct_stages(typename V2<T>::t* buf, int nbatch, int bs,
                                              const typename V2<T>::t* __restrict__ stw) {
  if constexpr (LOG2NS < LOG2N) {
    stage_ct<T, LOG2N, (1 << E), LOG2NS, EPT>(buf, nbatch, bs, stw + OFF);
    fft_ct_stages<T, LOG2N, E, EPT, LOG2NS + E, OFF + (LOG2NS > 0 ? (((1 << E) - 1) << LOG2NS) : 0)>(buf, nbatch, bs,
                                                                                                      stw);
  }
}

// Length-2^LOG2N FFT: one mixed-radix stage when LOG2N is not a multiple of E, then radix 2^E.
template <typename T, int LOG2N, int E, int EPT>
__device__ __forceinline__ void fft_ct(typename V2<T>::t* buf, int nbatch, int bs,
                                       const typename V2<T>::t* __restrict__ stw) {
  constexpr int rem = LOG2N % E;
  if constexpr (rem != 0) stage_ct<T, LOG2N, (1 << rem), 0, EPT>(buf, nbatch, bs, stw);
  fft_ct_stages<T, LOG2N, E, EPT, rem, 0>(buf, nbatch, bs, stw);
}

template <typename T, int E, int EPT, int LO, int HI>
__device__ __forceinline__ void fft_ct_dispatch(typename V2<T>::t* buf, int log2n, int nbatch, int bs,
                                                const typename V2<T>::t* __restrict__ stw) {
  if constexpr (LO <= HI) {
    if (log2n == LO) fft_ct<T, LO, E, EPT>(buf, nbatch, bs, stw);
    else fft_ct_dispatch<T, E, EPT, LO + 1, HI>(buf, log2n, nbatch, bs, stw);
  }
}

// Copy a stage table (len entries) into shared memory.
template <typename T>
__device__ __forceinline__ void load_tw_smem(typename V2<T>::t* dst, const typename V2<T>::t* __restrict__ stw,
                                             int len) {
  for (int i = threadIdx.x; i < len; i += blockDim.x) dst[i] = ldg(&stw[i]);
}

}  // namespace bk

namespace bk {

// The same FFT with the length and the stage known only at run time: one radix-16 stage body
// (and one mixed-radix first stage) per kernel instead of one unrolled instance per length and
// stage. Used by the double-float kernels, whose butterflies are an order of magnitude longer
// than binary32 or binary64 ones, so that compile time and code size stay bounded; the address
// arithmetic is generic (padi per element), which costs little next to double-float arithmetic.
template <typename T, int R, int EPT>
__device__ __forceinline__ void stage_rt(typename V2<T>::t* __restrict__ buf, int nbatch, int bs,
                                         const typename V2<T>::t* __restrict__ stw, int log2n, int log2ns) {
  typedef typename V2<T>::t C;
  constexpr int log2R = R == 16 ? 4 : (R == 8 ? 3 : (R == 4 ? 2 : 1));
  constexpr int log2EPT = EPT == 16 ? 4 : (EPT == 8 ? 3 : (EPT == 4 ? 2 : 1));
  constexpr int PER = EPT / R;
  const int log2tp = log2n - log2EPT;
  const int ntp = 1 << log2tp;
  const int nR = (1 << log2n) >> log2R;
  const int Ns = 1 << log2ns;
  const int t = threadIdx.x;
  const bool active = t < (nbatch << log2tp);
  const int tt = t & (ntp - 1);
  C* base = buf + (size_t)(t >> log2tp) * bs;
  C v[EPT];
  if (active) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[q * R + r] = base[padi(tt + q * ntp + r * nR)];
    }
  }
  __syncthreads();
  if (active) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int j = tt + q * ntp;
      const int k = j & (Ns - 1);
      C* u = v + q * R;
      if (Ns > 1) {
        const C* tw = stw + k;
#pragma unroll
        for (int r = 1; r < R; ++r) u[r] = cmul(u[r], tw[(r - 1) * Ns]);
      }
      Radix<C, T, R>::run(u);
      const int d0 = ((j >> log2ns) << (log2ns + log2R)) + k;
#pragma unroll
      for (int r = 0; r < R; ++r) base[padi(d0 + r * Ns)] = u[r];
    }
  }
  __syncthreads();
}

template <typename T, int E, int EPT>
__device__ __forceinline__ void fft_rt(typename V2<T>::t* buf, int log2n, int nbatch, int bs,
                                       const typename V2<T>::t* __restrict__ stw) {
  const int rem = log2n % E;
  if (rem == 1) stage_rt<T, 2, EPT>(buf, nbatch, bs, stw, log2n, 0);
  else if (E > 2 && rem == 2) stage_rt<T, 4, EPT>(buf, nbatch, bs, stw, log2n, 0);
  else if (E > 3 && rem == 3) stage_rt<T, (E > 3 ? 8 : 2), EPT>(buf, nbatch, bs, stw, log2n, 0);
  int off = 0;
  for (int l = rem; l < log2n; l += E) {
    stage_rt<T, (1 << E), EPT>(buf, nbatch, bs, stw + off, log2n, l);
    if (l > 0) off += ((1 << E) - 1) << l;
  }
}

// Batched in-place forward FFT of length n = 2^log2n (16 <= n <= 8192) over `nbatch` padded
// transforms bs apart in shared memory (element i of batch b at buf[b * bs + padi(i)]), stw the
// radix-2^E stage table of length n. The block needs at least nbatch * n / EPT threads. Input
// complete before the call (barrier); result complete on return, in natural order, in place. Each
// length 2^LO..2^HI is its own compile-time instance (log2n is uniform over the block); double-float
// takes the run-time form.
template <typename T, int E, int EPT, int LO = 4, int HI = 13>
__device__ __forceinline__ void fft_any(typename V2<T>::t* buf, int log2n, int nbatch, int bs,
                                        const typename V2<T>::t* __restrict__ stw) {
  if constexpr (std::is_same<T, dfl>::value) fft_rt<T, E, EPT>(buf, log2n, nbatch, bs, stw);
  else fft_ct_dispatch<T, E, EPT, LO, HI>(buf, log2n, nbatch, bs, stw);
}

// Batched forward FFT of length n = product of rad[0..nst), radices 2 to 5, over `nbatch` transforms bs
// apart: Stockham stages between the two buffers a and b (the input in b when nst is odd, else in
// a; the result in a), any thread count. stw: for each stage after the first, (R - 1) Ns twiddles
// omega_{R Ns}^{r k} as in the power-of-two tables.
template <typename T, int R>
__device__ __forceinline__ void mix_stage(const typename V2<T>::t* src, typename V2<T>::t* dst, int n, int nbatch, int bs,
                                          unsigned Ns, const typename V2<T>::t* __restrict__ stw) {
  typedef typename V2<T>::t C;
  const unsigned nb = (unsigned)n / R;
  for (unsigned idx = threadIdx.x; idx < nb * nbatch; idx += blockDim.x) {
    const unsigned q = idx / nb, j = idx - q * nb;
    const unsigned jq = j / Ns, k = j - jq * Ns;
    const C* s = src + q * bs;
    C v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = s[padi(j + r * nb)];
    if (Ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], ldg(stw + (r - 1) * Ns + k));
    }
    Radix<C, T, R>::run(v);
    C* o = dst + q * bs;
    const unsigned d0 = jq * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) o[padi(d0 + r * Ns)] = v[r];
  }
  __syncthreads();
}

template <typename T>
__device__ __forceinline__ void fft_mix(typename V2<T>::t* a, typename V2<T>::t* b, int n, const unsigned char* rad,
                                        int nst, int nbatch, int bs, const typename V2<T>::t* __restrict__ stw) {
  typedef typename V2<T>::t C;
  C* src = (nst & 1) ? b : a;
  C* dst = (nst & 1) ? a : b;
  unsigned Ns = 1;
  for (int s = 0; s < nst; ++s) {
    const int R = rad[s];
    if (R == 4) mix_stage<T, 4>(src, dst, n, nbatch, bs, Ns, stw);
    else if (R == 5) mix_stage<T, 5>(src, dst, n, nbatch, bs, Ns, stw);
    else if (R == 3) mix_stage<T, 3>(src, dst, n, nbatch, bs, Ns, stw);
    else mix_stage<T, 2>(src, dst, n, nbatch, bs, Ns, stw);
    if (Ns > 1) stw += (R - 1) * Ns;
    Ns *= R;
    C* t = src;
    src = dst;
    dst = t;
  }
}

}  // namespace bk
