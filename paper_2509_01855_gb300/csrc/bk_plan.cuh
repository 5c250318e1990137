// Plan object of the Birkhoff products (internal).
#pragma once

#include "bk_common.cuh"

namespace bk {

// One four-step layout, n = N1 * N2 (pass A: columns of length N1, pass B: rows of length N2), and
// its tables in the working type. Power-of-two plans: the real-even passes of bk_dct.cuh, n = 2N
// (NB column pairs and P row pairs per CTA). Bluestein plans: a plain complex FFT of length n (NB
// columns and 2P rows per CTA).
struct FourStep {
  int64_t n = 0;
  int N1 = 0, N2 = 0;
  int NB = 0, P = 0;
  int bsA = 0, bsB = 0;       // batch strides in shared memory (complex elements)
  size_t smemA = 0, smemB = 0;
  int thrA = 256, thrB = 256; // threads of the pass kernels
  void* stw1 = nullptr;       // stage twiddle table of the length-N1 FFT
  void* stw2 = nullptr;       // stage twiddle table of the length-N2 FFT
  void* twN = nullptr;        // real-even: the [N1/2 + 1][N2/2 + 2] table; else omega_n^m, m < n (FP64)
  void* twLo = nullptr;       // omega_n^m, m < 2^tw_h (FP32, plain complex)
  void* twHi = nullptr;       // omega_n^{m 2^tw_h}, m < n / 2^tw_h (FP32, plain complex)
  int tw_h = 0;
  // real-even sizes per vector: row length and total of the scratch A, column pairs
  int RS() const { return N2 / 2 + 2; }
  int64_t a_len() const { return (int64_t)(N1 / 2 + 1) * RS(); }
  int pairs() const { return N2 / 4 + 1; }
};

struct Plan {
  int64_t N = 0, L = 0, pitch = 0;
  int n_comp = 1, max_batch = 1, dtype = BK_F64;
  double t0 = 0, tf = 0, s = 0;
  bool small = true;          // whole chain in one CTA per vector
  bool generic = false;       // N not a power of two: dense products only
  bool df = false;            // FP64 plan whose transforms compute in double-float arithmetic
  // N not a power of two above the dense range: each DCT-I's length-N DFT by Bluestein's
  // convolution of length M (a power of two >= 2N - 1) on the four-step layout fsM
  bool blue = false;
  int64_t M = 0;
  FourStep fsM;
  void* chirp = nullptr;      // w_j = exp(-i pi j^2 / N), j < N (working type)
  void* bh = nullptr;         // FFT_M(b) / M of the conjugate chirp b (working type)
  void* bsc = nullptr;        // one scalar per vector (b-form products), working type
  int tileE = 0;              // four-step elements per CTA chosen by the autotuner (0: heuristic)
  size_t smemS = 0;           // dynamic shared memory of the single-CTA kernel
  int thrS = 256;             // threads of the single-CTA kernel
  void* tw = nullptr;         // omega_N^i, i < N (single-CTA plans; the N < 16 direct DFT)
  void* stwS = nullptr;       // stage twiddle table of the length-N FFT (single-CTA plans)
  // Four-step plans: the layout fs of the length-2N real-even DFT. split: the four passes run as
  // a launch each; else as one launch, a cluster of csize CTAs per vector.
  FourStep fs;
  int split = 0;
  bool mix = false;           // N = 16 m, m a product of 2, 3 and 5 (not a power of two): mixed-radix
  unsigned char rad1[12] = {}, rad2[12] = {};   // its radices of N1 and N2
  int nst1 = 0, nst2 = 0;
  int fe = 2;                 // log2 radix of the launch-per-pass kernels
  int csize = 0, cthr = 0;
  size_t csmem = 0;
  int cex = 0, cexY = 0, cexP = 0;   // FP32: offsets of the exchange area's parts in shared memory
  void* guest = nullptr;      // FP32 launch-per-pass plans: scratch lent to one-launch plans of a batch
  size_t guest_bytes = 0;
  void* tpost = nullptr;      // (cos, sin)(pi k / N), k = 0..N/2 (working type; not four-step)
  void* rk = nullptr;         // 1 / (4k), k = 0..N+1 (working type; rk[0] = 0)
  void* scrA = nullptr;       // scratch between passes A and B, fs.a_len() complex per vector (none of these
                              // three in FP32 one-launch plans)
  void* scrY = nullptr;       // stage buffer between the two DCTs, N + 2 per vector (Bluestein N + 1)
  void* scrG = nullptr;       // Bluestein: second-DCT input (stencil output), N + 1 per vector
  void* part = nullptr;       // pass-A shares of R_0, fs.pairs() per vector
  double* t_nodes = nullptr;  // node times t_j (FP64, device)
  double* w64 = nullptr;      // Clenshaw-Curtis weights (FP64, device, tau-domain)
  void* wT = nullptr;         // Clenshaw-Curtis weights in the working type (device)
  size_t bytes = 0;           // device bytes this plan allocated
  // Dense path (N <= 1024): B^a and (B^a)^T, FP32 plans pre-tiled as TF32 hi/lo parts for the
  // tensor cores, FP64 plans column-major FP64 (dA[0], dA[1]); used while `dense` is set.
  bool dense = false;
  void* dA[2] = {nullptr, nullptr};
  int dMp = 0;                // FP64 layout: rows padded to a multiple of 128
  int* derr = nullptr;        // device error word of the dense kernel (0 = no timeout)
  int dtest = 0;              // test mode: every dense FP32 product times out on purpose
  int dMt = 0, dnK = 0;       // 128-row output tiles, 32-wide K chunks
  void* dpart = nullptr;      // split-K partial sums (FP32)
  unsigned* dcnt = nullptr;   // split-K arrival counters, one per output tile (self-resetting)
};

// Grid sizes a plan of this precision supports: powers of two 4..2^24, any other N 4..2^22
// (BK_F64) or 4..2^23 (BK_F32).
bool plan_n_supported(int64_t N, int dtype);
bk_status plan_create(Plan** out, int64_t N, int n_comp, int max_batch, int dtype, double t0,
                      double tf, int64_t pitch, cudaStream_t st);
void plan_destroy(Plan* p);
bk_status plan_apply(const Plan* p, const void* v, void* out, int batch, bool trans,
                     cudaStream_t st);
// b-form product B^b v = B v - (B v)_N 1 (trans: B^bT u = B^T u - s (1 . u) w).
bk_status plan_apply_b(const Plan* p, const void* v, void* out, int batch, bool trans, cudaStream_t st);
// Apply to `nvec` vectors with an explicit scale (s = 1 gives B^a itself).
bk_status plan_apply_n(const Plan* p, const void* v, void* out, int nvec, bool trans, double s,
                       cudaStream_t st);

// Dense tensor-core path (bk_dense.cu).
bool dense_supported(int64_t N);
bk_status dense_build(Plan* p, cudaStream_t st);
bk_status dense_apply(const Plan* p, const void* v, void* out, int nvec, bool trans, double s, cudaStream_t st);
bk_status dense_status(const Plan* p, cudaStream_t st);

}  // namespace bk
