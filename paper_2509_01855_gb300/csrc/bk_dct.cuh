// DCT-I passes of the Birkhoff products for N a power of two, N >= 128 (internal; included by
// bk_birkhoff.cu after the element accessors).
//
// R(x)_k, k = 0..N, is the length-2N DFT of the even extension of x. With 2N = N1 N2, input index
// m = N2 n1 + n2 and output index k = k1 + N1 k2 the four-step split reads
//   C_{n2}[k1] = sum_{n1} x[N2 n1 + n2] omega_N1^{n1 k1},   A[k1][n2] = C_{n2}[k1] omega_2N^{n2 k1},
//   R_{k1 + N1 k2} = sum_{n2} A[k1][n2] omega_N2^{n2 k2}.
// x is real and even, so every column is real, A[k1][N2 - n2] = conj A[k1][n2], and every row's
// DFT is real, with the row N1 - k1 giving the same outputs as the row k1. Hence the columns
// n2 = 0..N2/2 and the rows k1 = 0..N1/2 suffice, two real columns travel as the two parts of one
// complex FFT of length N1, and two Hermitian rows as one complex FFT of length N2 whose real and
// imaginary parts are the two rows' outputs. Per vector that is N/2 complex points in each pass,
// N/2 complex values of scratch between them, every input read once and no separate real-FFT split:
// half the transform work and traffic of a length-N complex FFT of the extension's pairs, without
// the prefix sums of the half-length real DFT (whose rounding grows like sqrt(N)).
//
// Pass A takes column pairs p = 0..N2/4: p = 0 the columns 0 and N2/2, p >= 1 the columns 2p - 1
// and 2p (p = N2/4 its first one only). A is stored [k1][pos], RS = N2/2 + 2 per row, with column
// 2p - 1 at pos 2p and column 2p at pos 2p + 1 (columns 0 and N2/2 at 0 and 1), so a pair's two
// values are adjacent. Pass B takes row pairs q = 0..N1/4: rows 2q - 1 and 2q (q = 0: N1/2 and 0;
// q = N1/4: the first one only). The twiddle table has A's layout, so its reads are coalesced (an
// omega^m table indexed by n2 k1 cost one 32-byte sector per value), and holds the unpacking
// factors 1/2 and -i/2.
//
// N that is 16 times a product of 2, 3 and 5 runs the same passes with N1 and N2 multiples of 4 and
// mixed-radix FFTs.
//
// The second DCT's input is the integration stencil of the first one's output; pass A forms it in
// its loads (two aligned pair loads per column pair), so a product is four passes and no stencil pass.
#pragma once

namespace bk {

template <typename T> struct ReArgs {
  typedef typename V2<T>::t C;
  int N, N1, N2, log2N1, log2N2, RS;
  const C* stw1;   // stage tables of the two FFT lengths
  const C* stw2;
  const C* twA;    // [N1/2 + 1][RS]
  const T* rk;     // 1 / (4k), k = 0..N+1 (0 at k = 0)
  T cE;            // 2 / (N + 1)
  // radices of the two FFT lengths (N not a power of two; bk_fft.cuh, fft_mix)
  int nst1, nst2;
  unsigned char rad1[12], rad2[12];
};

// Longest FFT of the one-launch form (its kernels hold an instance per length): N <= 2^17.
constexpr int CL_MAXLOG2 = 9;

// The sub-FFTs of a pass. The one-launch kernels run four passes of run-time lengths: there the FFT
// is one out-of-line function per type (inlined four times over, its length instances exceeded the
// registers), taking byte offsets into dynamic shared memory so that its accesses stay shared ones.
template <typename T>
__device__ __noinline__ void re_fft_call(unsigned off, int log2n, int nbatch, int bs, unsigned tw_off) {
  typedef typename V2<T>::t C;
  extern __shared__ __align__(16) unsigned char smem[];
  fft_any<T, SmallFft<T>::E, SmallFft<T>::EPT, 4, CL_MAXLOG2>(reinterpret_cast<C*>(smem + off), log2n, nbatch, bs,
                                                        reinterpret_cast<const C*>(smem + tw_off));
}
// F: the FFT's shape, void for the one-launch kernels' call.
template <typename F> struct IsMix { static constexpr bool v = F::MIX; };
template <> struct IsMix<void> { static constexpr bool v = false; };
template <typename T, typename F>
__device__ __forceinline__ void re_fft(const ReArgs<T>& g, bool first, typename V2<T>::t* buf, typename V2<T>::t* alt,
                                       int nbatch, int bs, const typename V2<T>::t* stw) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int log2n = first ? g.log2N1 : g.log2N2;
  if constexpr (IsMix<F>::v)
    fft_mix<T>(buf, alt, first ? g.N1 : g.N2, first ? g.rad1 : g.rad2, first ? g.nst1 : g.nst2, nbatch, bs, stw);
  else if constexpr (std::is_void<F>::value)
    re_fft_call<T>((unsigned)(reinterpret_cast<unsigned char*>(buf) - smem), log2n, nbatch, bs,
                   (unsigned)(reinterpret_cast<const unsigned char*>(stw) - smem));
  else
    fft_any<T, F::E, F::EPT>(buf, log2n, nbatch, bs, stw);
}

// Loads that bypass L1 (CG: data other CTAs of the running kernel wrote to global memory) or not.
template <bool CG> __device__ __forceinline__ float ldr(const float* p) { return CG ? __ldcg(p) : *p; }
template <bool CG> __device__ __forceinline__ double ldr(const double* p) { return CG ? __ldcg(p) : *p; }
template <bool CG> __device__ __forceinline__ dfl ldr(const dfl* p) {
  const float2* q = reinterpret_cast<const float2*>(p);
  const float2 f = CG ? __ldcg(q) : *q;
  return dfl(f.x, f.y);
}
template <bool CG> __device__ __forceinline__ float2 ldc(const float2* p) { return CG ? __ldcg(p) : *p; }
template <bool CG> __device__ __forceinline__ double2 ldc(const double2* p) { return CG ? __ldcg(p) : *p; }
template <bool CG> __device__ __forceinline__ dfl2 ldc(const dfl2* p) {
  const float4* q = reinterpret_cast<const float4*>(p);
  const float4 f = CG ? __ldcg(q) : *q;
  dfl2 r;
  r.x = dfl(f.x, f.y);
  r.y = dfl(f.z, f.w);
  return r;
}
// Two adjacent complex values at an even index of a 16-byte aligned row.
__device__ __forceinline__ void ld2(const float2* p, float2& a, float2& b) {
  const float4 f = __ldg(reinterpret_cast<const float4*>(p));
  a = make_float2(f.x, f.y);
  b = make_float2(f.z, f.w);
}
template <typename C> __device__ __forceinline__ void ld2(const C* p, C& a, C& b) { a = ldg(p); b = ldg(p + 1); }
__device__ __forceinline__ void st2(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st2(double2* p, double2 a, double2 b) { p[0] = a; p[1] = b; }
__device__ __forceinline__ void st2(dfl2* p, dfl2 a, dfl2 b) {
  float4* q = reinterpret_cast<float4*>(p);
  q[0] = make_float4(a.x.hi, a.x.lo, a.y.hi, a.y.lo);
  q[1] = make_float4(b.x.hi, b.x.lo, b.y.hi, b.y.lo);
}

// Where a pass finds element m of a vector and row k of A: in global memory, or (FP32 one-launch form)
// spread over the exchange areas of the cluster's CTAs. Row k of A is kept by the CTA whose pass B reads
// it (tile = pair / P, rank = tile mod csize), so pass A writes to all CTAs and pass B reads its own;
// the stage buffer is cut into csz blocks of 2^sh elements (the last two more); the shares of R_0 go to
// every CTA, so that the last pass touches no other CTA's memory.
template <typename S> __device__ __forceinline__ S* at(S* x, int m) { return x + m; }
template <typename T> __device__ __forceinline__ void put_share(T* part, int p, T v) { part[p] = v; }
template <typename C> __device__ __forceinline__ C* row(C* A, int k, int RS) { return A + (int64_t)k * RS; }

// The address of the same shared variable in CTA `rank` of the cluster.
template <typename P> __device__ __forceinline__ P* cluster_map(P* p, unsigned rank) {
  unsigned long long r;
  asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"((unsigned long long)p), "r"(rank));
  return reinterpret_cast<P*>(r);
}
struct ClusterStage {
  float* base;
  int sh, csz;
};
struct ClusterRows {
  float2* base;
  int P, csize, half;
};
struct ClusterShares {
  float* base;
  int csize;
};
__device__ __forceinline__ float* at(const ClusterShares& c, int p) { return c.base + p; }
__device__ __forceinline__ void put_share(const ClusterShares& c, int p, float v) {
  for (int o = 0; o < c.csize; ++o) cluster_map(c.base, o)[p] = v;
}
__device__ __forceinline__ float* at(const ClusterStage& y, int m) {
  const int o = min(m >> y.sh, y.csz - 1);
  return cluster_map(y.base, o) + (m - (o << y.sh));
}
__device__ __forceinline__ float2* row(const ClusterRows& a, int k, int RS) {
  const int q = k == a.half ? 0 : (k + 1) >> 1;   // its pair: rows 2q - 1 and 2q (q = 0: N1/2 and 0)
  const int second = k != a.half && !(k & 1);
  const int tile = q / a.P, o = tile % a.csize;
  return cluster_map(a.base, o) + (((tile / a.csize) * a.P + (q - tile * a.P)) * 2 + second) * RS;
}

// Second-DCT input x_m from the stage buffer Y, any m (see stencil_fwd / stencil_trn; ST_TRN's
// buffer holds T_k = (Y_k - Y_0) / (4k), for which the transposed stencil is T_{m-1} - T_{m+1}).
template <typename T, int K, bool CG, typename X>
__device__ __forceinline__ T re_stencil(X Y, int m, const ReArgs<T>& g) {
  const int N = g.N;
  if (K == ST_FWD) {
    if (m == 0) return T(0);
    if (m == N) return -ldr<CG>(at(Y, N - 1)) * (T(2) * g.rk[N]);
    if (m == N - 1) {
      const T yN = ldr<CG>(at(Y, N));
      const T a = T(0.5) * g.rk[N - 1] - T(0.5) * g.rk[N + 1];
      return dot2(yN, a, -ldr<CG>(at(Y, N - 2)), g.rk[N - 1]);
    }
    return (ldr<CG>(at(Y, m + 1)) - ldr<CG>(at(Y, m - 1))) * g.rk[m];
  }
  if (m == 0) return T(-2) * ldr<CG>(at(Y, 1));
  if (m == N) return ldr<CG>(at(Y, N - 1)) * g.cE;
  return ldr<CG>(at(Y, m - 1)) - ldr<CG>(at(Y, m + 1));
}

// 1 / (4k), k >= 1: correctly rounded either way (4k is exact in binary32 for k <= 2^24); the FP32
// passes, bound by load latency, compute it, the others read the table.
template <typename T> __device__ __forceinline__ T re_rk(const ReArgs<T>& g, int k) { return g.rk[k]; }
template <> __device__ __forceinline__ float re_rk<float>(const ReArgs<float>& g, int k) {
  return __frcp_rn((float)(4 * k));
}

// Pass A of column pairs [tile NB, tile NB + NB) of one vector x into A; part[p] gets the pair's
// share of R_0 = sum over all N2 columns of A[0][n2]. buf: NB padded transforms bs apart. S: stored
// type (the caller's for IN_PLAIN / IN_WINV, T for the stage buffer). The results of a pair do not
// depend on the tile or the thread count. A thread keeps one pair and steps over its rows, so that
// its addresses are one base plus constant strides (per-element index arithmetic was half of the
// FP32 kernel's instructions).
template <typename T, int K, bool CG, typename F, typename S, typename X, typename AP, typename PP>
__device__ __forceinline__ void re_passA(const ReArgs<T>& g, int tile, int NB, int bs, X x, AP A, PP part,
                                         typename V2<T>::t* buf, const typename V2<T>::t* stw) {
  typedef typename V2<T>::t C;
  typedef Cv<T, S> CV;
  const int N = g.N, N1 = g.N1, N2 = g.N2, half = N1 >> 1;
  const int p0 = tile * NB;
  const int na = min(NB, (N2 >> 2) + 1 - p0);
  const int step = blockDim.x / NB;
  const int row0 = threadIdx.x / NB;
  const int b = threadIdx.x - row0 * NB;
  const int p = p0 + b;
  const bool on = b < na && row0 < step;
  const bool last = p == (N2 >> 2);   // no second column
  // fft_mix alternates between two buffers: with an odd number of stages its input is the second
  C* const alt = buf + NB * bs;
  C* z = (IsMix<F>::v && (g.nst1 & 1) ? alt : buf) + b * bs;
  if (on && p != 0) {
    // rows j and N1 - 1 - j: x at m = j N2 + 2p - 1 and m + 1, and, reflected, at
    // i = (j + 1) N2 - 2p + 1 and i - 1 (m and i are odd)
    constexpr int LD = sizeof(T) == 8 ? 2 : 4;
    for (int j0 = row0; j0 < half; j0 += LD * step) {
      C d[LD], r[LD];
#pragma unroll
      for (int u = 0; u < LD; ++u) {
        const int j = j0 + u * step;
        if (j >= half) continue;
        const int m = j * N2 + 2 * p - 1, i = (j + 1) * N2 - 2 * p + 1;
        if constexpr (K == IN_PLAIN || K == IN_WINV) {
          d[u] = mk2<T>(CV::in(*at(x, m)), last ? T(0) : CV::in(*at(x, m + 1)));
          r[u] = mk2<T>(CV::in(*at(x, i)), last ? T(0) : CV::in(*at(x, i - 1)));
          if (K == IN_WINV) {
            d[u].x = T(0.5) * d[u].x;
            d[u].y = T(0.5) * d[u].y;
            r[u].x = T(0.5) * r[u].x;
            r[u].y = T(0.5) * r[u].y;
          }
        } else {
          const C a0 = ldc<CG>(reinterpret_cast<const C*>(at(x, m - 1)));   // x_{m-1}, x_m
          const C a1 = ldc<CG>(reinterpret_cast<const C*>(at(x, m + 1)));   // x_{m+1}, x_{m+2}
          const C c0 = ldc<CG>(reinterpret_cast<const C*>(at(x, i - 1)));   // x_{i-1}, x_i
          const T hi = ldr<CG>(at(x, i + 1)), lo = ldr<CG>(at(x, i - 2));
          if (K == ST_FWD) {
            d[u] = mk2<T>((a1.x - a0.x) * re_rk<T>(g, m), (a1.y - a0.y) * re_rk<T>(g, m + 1));
            r[u] = mk2<T>((hi - c0.x) * re_rk<T>(g, i), (c0.y - lo) * re_rk<T>(g, i - 1));
            if (i == N - 1) r[u].x = re_stencil<T, K, CG>(x, i, g);   // the aliasing fold
          } else {
            d[u] = mk2<T>(a0.x - a1.x, a0.y - a1.y);
            r[u] = mk2<T>(c0.x - hi, lo - c0.y);
          }
          if (last) d[u].y = r[u].y = T(0);
        }
      }
#pragma unroll
      for (int u = 0; u < LD; ++u) {
        const int j = j0 + u * step;
        if (j >= half) continue;
        z[padi(j)] = d[u];
        z[padi(N1 - 1 - j)] = r[u];
      }
    }
  } else if (on) {   // columns 0 and N2/2
    for (int n1 = row0; n1 < N1; n1 += step) {
      const int ma = n1 * N2, mb = ma + (N2 >> 1);
      const int ia = ma <= N ? ma : 2 * N - ma, ib = mb <= N ? mb : 2 * N - mb;
      if constexpr (K == IN_PLAIN || K == IN_WINV) {
        T a = CV::in(*at(x, ia)), c = CV::in(*at(x, ib));
        if (K == IN_WINV) {
          if (ia != 0 && ia != N) a = T(0.5) * a;
          c = T(0.5) * c;
        }
        z[padi(n1)] = mk2<T>(a, c);
      } else {
        z[padi(n1)] = mk2<T>(re_stencil<T, K, CG>(x, ia, g), re_stencil<T, K, CG>(x, ib, g));
      }
    }
  }
  __syncthreads();
  re_fft<T, F>(g, true, buf, alt, na, bs, stw);
  z = buf + b * bs;
  if (on) {
    constexpr int LD = sizeof(T) == 8 ? 2 : 4;
    const C* tw = g.twA + 2 * p;
    for (int k0 = row0; k0 <= half; k0 += LD * step) {
      C wa[LD], wb[LD];
#pragma unroll
      for (int u = 0; u < LD; ++u) {
        const int k = k0 + u * step;
        if (k <= half) ld2(tw + (int64_t)k * g.RS, wa[u], wb[u]);
      }
#pragma unroll
      for (int u = 0; u < LD; ++u) {
        const int k = k0 + u * step;
        if (k > half) continue;
        const C zk = z[padi(k)];
        const C zm = z[padi(k == 0 ? 0 : N1 - k)];
        if (k == 0) put_share(part, p, p == 0 ? zk.x + zk.y : T(2) * (zk.x + zk.y));
        const C sa = mk2<T>(zk.x + zm.x, zk.y - zm.y);   // Z_k + conj Z_{N1-k}
        const C sb = mk2<T>(zk.x - zm.x, zk.y + zm.y);   // Z_k - conj Z_{N1-k}
        st2(row(A, k, g.RS) + 2 * p, cmul(sa, wa[u]), cmul(sb, wb[u]));
      }
    }
  }
}

// Epilogue kinds of pass B:
//   EP_STORE     : stage[k] = R_k / N                        (after the first DCT, forward)
//   EP_STORE_TRN : stage[k] = (R_k - R_0) / (4k), 0 at k = 0 (after the first DCT, transpose)
//   EP_FWD_OUT   : out[k] = s (R_k - R_0), 0 at k = 0        (after the second DCT, forward)
//   EP_TRN_OUT   : out[k] = (s/N) W_k R_k                    (after the second DCT, transpose)
// Pass B of row pairs [tile P, tile P + P) of one vector.
template <typename T, int E, bool CG, typename F, typename S, typename X, typename AP, typename PP>
__device__ __forceinline__ void re_passB(const ReArgs<T>& g, int tile, int P, int bs, AP A, X out, int64_t zero_to,
                                         PP part, typename V2<T>::t* buf,
                                         const typename V2<T>::t* stw, T* y0s, T s, T invN) {
  typedef typename V2<T>::t C;
  typedef Cv<T, S> CV;
  constexpr bool DC = E == EP_STORE_TRN || E == EP_FWD_OUT;
  const int q0 = tile * P;
  const int nt = blockDim.x;
  const int N = g.N, N1 = g.N1, N2 = g.N2, h2 = N2 >> 1;
  const int na = min(P, (N1 >> 2) + 1 - q0);
  C* const alt = buf + P * bs;
  {
    // positions 0..N2/2 of the two rows (pos 0, 1: columns 0 and N2/2, whose values are real;
    // pos >= 2: column pos - 1 and its mirror image N2 - pos + 1); threads along the rows
    const int tpr = min(nt, h2);
    const int i0 = threadIdx.x / tpr, istep = nt / tpr, ps0 = threadIdx.x - i0 * tpr;
    constexpr int LD = 4;
    for (int i = i0 < istep ? i0 : na; i < na; i += istep) {
      const int q = q0 + i;
      const C* ra = row(A, q == 0 ? N1 >> 1 : 2 * q - 1, g.RS);
      const C* rb = row(A, 2 * q, g.RS);
      const bool two = q != (N1 >> 2);
      C* z = (IsMix<F>::v && (g.nst2 & 1) ? alt : buf) + i * bs;
      for (int ps = ps0; ps <= h2; ps += LD * tpr) {
        C a[LD], c[LD];
#pragma unroll
        for (int u = 0; u < LD; ++u) {
          const int pos = ps + u * tpr;
          if (pos > h2) continue;
          a[u] = ldc<CG>(ra + pos);
          c[u] = two ? ldc<CG>(rb + pos) : mk2<T>(T(0), T(0));
        }
#pragma unroll
        for (int u = 0; u < LD; ++u) {
          const int pos = ps + u * tpr;
          if (pos > h2) continue;
          if (pos < 2) {
            z[padi(pos == 0 ? 0 : h2)] = mk2<T>(a[u].x, c[u].x);
          } else {
            z[padi(pos - 1)] = mk2<T>(a[u].x - c[u].y, a[u].y + c[u].x);
            z[padi(N2 - pos + 1)] = mk2<T>(a[u].x + c[u].y, c[u].x - a[u].y);
          }
        }
      }
    }
  }
  if (DC && threadIdx.x < 32) {   // one warp, so the order does not depend on the thread count
    const int np = (N2 >> 2) + 1;
    T acc[4] = {T(0), T(0), T(0), T(0)};
    for (int i = threadIdx.x; i < np; i += 128) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i + 32 * u < np) acc[u] += ldr<CG>(at(part, i + 32 * u));
    }
    T a = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    for (int o = 16; o > 0; o >>= 1) a += shfl_xor(a, o);
    if (threadIdx.x == 0) *y0s = a;
  }
  __syncthreads();
  re_fft<T, F>(g, false, buf, alt, na, bs, stw);
  const T Y0 = DC ? *y0s : T(0);
  // threads along consecutive rows r = 2 q0 - 1 + c, so that each store run covers 2P consecutive
  // outputs: row r gives k = r + N1 j and, reflected, k = N1 (j + 1) - r from column N2 - 1 - j
  const int step = nt / (2 * P);
  const int j0 = (int)threadIdx.x / (2 * P);
  const int c = threadIdx.x - j0 * 2 * P;
  const bool mid = q0 == 0 && c == 0;    // row N1/2: its direct outputs only
  const bool zero = q0 == 0 && c == 1;   // row 0: its direct outputs and k = N
  const int r = mid ? N1 >> 1 : 2 * q0 - 1 + c;
  const T sN = s * invN;
  auto val = [&](T v, int k, T rk) {
    if (E == EP_STORE) return v * invN;
    if (E == EP_STORE_TRN) return (v - Y0) * rk;
    if (E == EP_FWD_OUT) return s * (v - (k == 0 ? v : Y0));   // Y0's sum rounds apart from the row's R_0
    return (k == 0 || k == N ? sN : T(2) * sN) * v;
  };
  if (j0 < step && (mid || r < (N1 >> 1))) {
    const T* w = reinterpret_cast<const T*>(buf + (c >> 1) * bs) + (c & 1);
    constexpr int LD = sizeof(T) == 8 ? 2 : 4;
    for (int jj = j0; jj < h2; jj += LD * step) {
      T vd[LD], vm[LD], rd[LD], rm[LD];
#pragma unroll
      for (int u = 0; u < LD; ++u) {
        const int j = jj + u * step;
        if (j >= h2) continue;
        vd[u] = w[2 * padi(j)];
        vm[u] = w[2 * padi(N2 - 1 - j)];
        if (E == EP_STORE_TRN) {
          rd[u] = r + N1 * j == 0 ? T(0) : re_rk<T>(g, r + N1 * j);
          rm[u] = re_rk<T>(g, N1 * (j + 1) - r);
        }
      }
#pragma unroll
      for (int u = 0; u < LD; ++u) {
        const int j = jj + u * step;
        if (j >= h2) continue;
        const int kd = r + N1 * j, km = N1 * (j + 1) - r;
        *at(out, kd) = CV::out(val(vd[u], kd, rd[u]));
        if (!mid && (!zero || j == h2 - 1)) *at(out, km) = CV::out(val(vm[u], km, rm[u]));
      }
    }
  }
  if ((E == EP_FWD_OUT || E == EP_TRN_OUT) && tile == 0) {
    for (int64_t m = N + 1 + threadIdx.x; m < zero_to; m += nt) *at(out, m) = S(0);
  }
}

// ---- one launch per pass: blockIdx.x the vector (fastest, so that the vectors of one tile share
// its twiddles in L2), blockIdx.y the tile -----------------------------------------------------
template <typename T, int K, typename F, typename S>
__device__ __forceinline__ void re_passA_cta(const ReArgs<T>& g, int vec, int tile, int NB, int bs, const S* src,
                                             int64_t sstride, typename V2<T>::t* A, int64_t astride, T* part) {
  typedef typename V2<T>::t C;
  extern __shared__ __align__(16) unsigned char smem[];
  C* buf = reinterpret_cast<C*>(smem);
  const C* stw = g.stw1;
  if (sizeof(T) == 4 && !F::MIX) {   // FP32: stage twiddles in shared memory after the tile
    C* tws = buf + (size_t)NB * bs;
    load_tw_smem<T>(tws, stw, stage_tw_len(g.log2N1, F::E));
    stw = tws;
  }
  re_passA<T, K, false, F, S>(g, tile, NB, bs, src + vec * sstride, A + vec * astride,
                              part + (int64_t)vec * ((g.N2 >> 2) + 1), buf, stw);
}

template <typename T, int E, typename F, typename S>
__device__ __forceinline__ void re_passB_cta(const ReArgs<T>& g, int vec, int tile, int P, int bs,
                                             const typename V2<T>::t* A, int64_t astride, S* dst, int64_t dstride,
                                             int64_t zero_to, const T* part, T s, T invN) {
  typedef typename V2<T>::t C;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ T y0s;
  C* buf = reinterpret_cast<C*>(smem);
  const C* stw = g.stw2;
  if (sizeof(T) == 4 && !F::MIX) {
    C* tws = buf + (size_t)P * bs;
    load_tw_smem<T>(tws, stw, stage_tw_len(g.log2N2, F::E));
    stw = tws;
  }
  re_passB<T, E, false, F, S>(g, tile, P, bs, A + vec * astride, dst + vec * dstride, zero_to,
                              part + (int64_t)vec * ((g.N2 >> 2) + 1), buf, stw, &y0s, s, invN);
}

template <typename T, int K, typename F, typename S>
__global__ void __launch_bounds__(F::MT, F::MINB)
    k_re_passA(const __grid_constant__ ReArgs<T> g, int NB, int bs, const S* __restrict__ src, int64_t sstride,
               typename V2<T>::t* __restrict__ A, int64_t astride, T* __restrict__ part) {
  pdl_wait();
  re_passA_cta<T, K, F, S>(g, blockIdx.x, blockIdx.y, NB, bs, src, sstride, A, astride, part);
}

// F = BigFft: rows of 8192 points in FP64 and double-float (N = 2^24).
template <typename T, int E, typename F, typename S>
__global__ void __launch_bounds__(F::MT, F::MINB)
    k_re_passB(const __grid_constant__ ReArgs<T> g, int P, int bs, const typename V2<T>::t* __restrict__ A,
               int64_t astride, S* __restrict__ dst, int64_t dstride, int64_t zero_to, const T* __restrict__ part,
               T s, T invN) {
  pdl_wait();
  re_passB_cta<T, E, F, S>(g, blockIdx.x, blockIdx.y, P, bs, A, astride, dst, dstride, zero_to, part, s, invN);
}

// ---- all four passes of a vector in one launch: one cluster of CTAs per vector ------------------
// The passes exchange A, the stage buffer and the shares of R_0, separated by cluster barriers
// (release / acquire) in place of launches. FP32: in shared memory, spread over the exchange areas of the
// cluster's CTAs, so that such a plan owns no scratch and any number of its products may run at a time,
// on any streams. FP64: through global memory (L2), with reads that bypass L1.
template <typename T> struct ReJob {
  typedef typename V2<T>::t C;
  ReArgs<T> g;
  const Us<T>* in;
  Us<T>* out;
  int64_t pitch, astride, ystride;
  C* A;
  T* Y;
  T* part;
  T s, invN;
  int NB, bsA, P, bsB, nvec;
  int ex, exY, exP, csz;   // FP32 one-launch form: byte offsets of A's rows, the stage block and the
                           // shares in a CTA's shared memory; blocks of the stage buffer
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier() {
  cluster_arrive();
  cluster_wait();
}

template <typename T, bool TRANS>
__device__ __forceinline__ void re_cluster_body(const ReJob<T>& J, int vec, int rank, int csize) {
  typedef typename V2<T>::t C;
  typedef Us<T> U;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ T y0s;
  constexpr bool DS = sizeof(T) == 4;   // exchange in shared memory
  constexpr bool CG = !DS;
  if (DS) cluster_arrive();   // waited for below: every CTA of the cluster runs before another writes to it
  const ReArgs<T>& g = J.g;
  C* tw1 = reinterpret_cast<C*>(smem);
  const int l1 = stage_tw_len(g.log2N1, SmallFft<T>::E), l2 = stage_tw_len(g.log2N2, SmallFft<T>::E);
  C* tw2 = tw1 + l1;
  C* buf = tw2 + l2;
  load_tw_smem<T>(tw1, g.stw1, l1);
  load_tw_smem<T>(tw2, g.stw2, l2);
  const U* in = J.in + vec * J.pitch;
  U* out = J.out + vec * J.pitch;
  const int ta = ((g.N2 >> 2) + J.NB) / J.NB;   // tiles of the N2/4 + 1 column pairs
  const int tb = ((g.N1 >> 2) + J.P) / J.P;     // tiles of the N1/4 + 1 row pairs
  auto passes = [&](auto A, auto Y, auto part) {
    for (int t = rank; t < ta; t += csize) {
      re_passA<T, TRANS ? IN_WINV : IN_PLAIN, CG, void, U>(g, t, J.NB, J.bsA, in, A, part, buf, tw1);
      __syncthreads();
    }
    cluster_barrier();
    for (int t = rank; t < tb; t += csize) {
      re_passB<T, TRANS ? EP_STORE_TRN : EP_STORE, CG, void, T>(g, t, J.P, J.bsB, A, Y, 0, part, buf, tw2, &y0s, J.s, J.invN);
      __syncthreads();
    }
    cluster_barrier();
    for (int t = rank; t < ta; t += csize) {
      re_passA<T, TRANS ? ST_TRN : ST_FWD, CG, void, T>(g, t, J.NB, J.bsA, Y, A, part, buf, tw1);
      __syncthreads();
    }
    cluster_barrier();
    for (int t = rank; t < tb; t += csize) {
      re_passB<T, TRANS ? EP_TRN_OUT : EP_FWD_OUT, CG, void, U>(g, t, J.P, J.bsB, A, out, J.pitch, part, buf, tw2, &y0s, J.s,
                                                            J.invN);
      __syncthreads();
    }
  };
  if constexpr (DS) {
    const ClusterRows A = {reinterpret_cast<C*>(smem + J.ex), J.P, csize, g.N1 >> 1};
    const ClusterStage Y = {reinterpret_cast<T*>(smem + J.exY), __clz(J.csz) - __clz(g.N), J.csz};
    cluster_wait();
    passes(A, Y, ClusterShares{reinterpret_cast<T*>(smem + J.exP), csize});
  } else {
    passes(J.A + vec * J.astride, J.Y + vec * J.ystride, J.part + (int64_t)vec * ((g.N2 >> 2) + 1));
  }
}

template <typename T, bool TRANS>
__global__ void __launch_bounds__(512, sizeof(T) == 8 ? 1 : 2) k_re_cluster(const __grid_constant__ ReJob<T> J, int csize) {
  pdl_wait();
  re_cluster_body<T, TRANS>(J, blockIdx.x / csize, blockIdx.x % csize, csize);
}

}  // namespace bk
