// Dense complex linear algebra of the PT-CN step and ACE:
//   overlap / projection products S = Psi^H (H Psi), Psi S (Alg. 3),
//   M = Psi^H W, xi^H X, xi Y (ACE), Psi^H Psi and Psi L^{-H} (Sec. 3.4),
//   Cholesky factorisations (orthonormalisation, -M of ACE) and L^{-1}.
// GEMM: 16 x 16 output tiles on the CUDA cores; a long reduction is split over blocks
// (split-K) into a workspace and summed in a fixed order, so results are deterministic.
// Hermitian products (Psi^H Psi) compute half the tiles; products with a triangular
// factor stop the reduction at the diagonal.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace pt {

// Output structure the caller promises (skipped work is exactly zero or implied):
//   GEMM_HERM   C = A^H A is Hermitian: only tiles on or below the diagonal are
//               computed; the upper triangle is written as the conjugate mirror.
//   GEMM_TRI_B  op(B) is upper triangular (op(B)[k][j] = 0 for k > j): the
//               reduction for the output columns [n0, n0 + 16) stops at n0 + 16.
//
// One block of 64 threads computes a 16 x 16 tile over its K chunk, 2 x 2 complex values
// per thread; the next K slice is fetched into registers while the current one is
// multiplied from the other of two shared-memory buffers. In FP64 nothing but the
// multiply-adds counts (an SM does two a clock, one warp instruction in 16 clocks), so
// the small tile costs no time and saves the work of padding and of the skipped
// triangle. FP32 (the small products of mixed precision) takes the same kernel: C is the
// complex type of the arithmetic, TI that of A and B in memory.
constexpr int GT = 16, GK = 16;

template <typename C> __device__ __forceinline__ C mk_as(double2 v) { return cvt<C>(v); }
template <typename C> __device__ __forceinline__ C mk_as(float2 v) { return v; }
__device__ __forceinline__ double2 ld_op(const double2* p) { return *p; }
__device__ __forceinline__ float2 ld_op(const float2* p) { return __ldg(p); }

// row and column of tile t = i (i + 1) / 2 + j of the lower triangle
__device__ __forceinline__ void lower_tile(int t, int& i, int& j) {
  i = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while (i * (i + 1) / 2 > t) --i;
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  j = t - i * (i + 1) / 2;
}

// *c = r + beta *c
__device__ __forceinline__ void put_output(double2* c, double2 beta, double2 r) {
  if (beta.x != 0.0 || beta.y != 0.0) {
    const double2 o = *c;
    r.x += beta.x * o.x - beta.y * o.y;
    r.y += beta.x * o.y + beta.y * o.x;
  }
  *c = r;
}

template <typename C, typename TI, int opA, int opB>
__global__ void __launch_bounds__(64) k_gemm(int M, int N, int K, int kchunk, int ksplit, int structure, int swapped,
                                             double2 alpha, const TI* __restrict__ A, long lda,
                                             const TI* __restrict__ B, long ldb, double2 beta,
                                             double2* __restrict__ Cm, long ldc, double2* __restrict__ part) {
  grid_entry();
  constexpr int P = GT * GK / 64;   // operand elements per thread per slice
  __shared__ C As[2][GK][GT + 1];
  __shared__ C Bs[2][GK][GT + 1];
  const int tid = threadIdx.x;
  const int tx = tid & 7, ty = tid >> 3;
  int bi = swapped ? blockIdx.y : blockIdx.x, bj = swapped ? blockIdx.x : blockIdx.y;
  if (structure == GEMM_HERM) lower_tile(blockIdx.x, bi, bj);
  const int m0 = bi * GT, n0 = bj * GT, kz = blockIdx.z;
  const int kbeg = kz * kchunk;
  int kend = min(K, kbeg + kchunk);
  if (structure == GEMM_TRI_B) kend = min(kend, n0 + GT);
  C acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b] = C{};
  // FP32 sums run over kRun terms, then go into FP64 ones: their rounding does not grow with K
  constexpr int kRun = 512;
  double2 sum[2][2] = {};
  auto flush = [&]() {
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const double2 v = to_d(acc[a][b]);
        sum[a][b].x += v.x;
        sum[a][b].y += v.y;
        acc[a][b] = C{};
      }
  };
  // next slice, untouched until it is stored: the loads stay in flight together (a conjugation
  // at the load waited for each in turn: 16.7 us a product of 16 columns by 1,647, 9.4 now)
  TI ra[P], rb[P];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < P; ++q) {
      const int u = tid & 15, w = (tid >> 4) + 4 * q;   // u runs along the contiguous direction
      const int ia = opA == OP_N ? u : w, ka = opA == OP_N ? w : u;
      const int jb = opB == OP_N ? w : u, kb = opB == OP_N ? u : w;
      ra[q] = rb[q] = TI{};
      if (m0 + ia < M && k0 + ka < kend)
        ra[q] = ld_op(opA == OP_N ? A + (m0 + ia) + (long)(k0 + ka) * lda : A + (k0 + ka) + (long)(m0 + ia) * lda);
      if (n0 + jb < N && k0 + kb < kend)
        rb[q] = ld_op(opB == OP_N ? B + (k0 + kb) + (long)(n0 + jb) * ldb : B + (n0 + jb) + (long)(k0 + kb) * ldb);
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int q = 0; q < P; ++q) {
      const int u = tid & 15, w = (tid >> 4) + 4 * q;
      C a = mk_as<C>(ra[q]), b = mk_as<C>(rb[q]);
      if (opA == OP_H) a.y = -a.y;
      if (opB == OP_H) b.y = -b.y;
      if (opA == OP_N) As[buf][w][u] = a; else As[buf][u][w] = a;
      if (opB == OP_N) Bs[buf][u][w] = b; else Bs[buf][w][u] = b;
    }
  };
  int buf = 0;
  if (kbeg < kend) {
    fetch(kbeg);
    stash(0);
  }
  __syncthreads();
  for (int k0 = kbeg; k0 < kend; k0 += GK) {
    const bool more = k0 + GK < kend;
    if (more) fetch(k0 + GK);   // in flight during the products below
    auto one = [&](int k) {
      C av[2], bv[2];
#pragma unroll
      for (int a = 0; a < 2; ++a) av[a] = As[buf][k][tx + 8 * a];
#pragma unroll
      for (int b = 0; b < 2; ++b) bv[b] = Bs[buf][k][ty + 8 * b];
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          acc[a][b].x = fma(av[a].x, bv[b].x, acc[a][b].x);
          acc[a][b].x = fma(-av[a].y, bv[b].y, acc[a][b].x);
          acc[a][b].y = fma(av[a].x, bv[b].y, acc[a][b].y);
          acc[a][b].y = fma(av[a].y, bv[b].x, acc[a][b].y);
        }
    };
    if (kend - k0 >= GK) {
#pragma unroll
      for (int k = 0; k < GK; ++k) one(k);
    } else {
      for (int k = 0; k < kend - k0; ++k) one(k);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
    if (sizeof(C) == sizeof(float2) && (k0 - kbeg) % kRun == kRun - GK) flush();
  }
  if (sizeof(C) == sizeof(float2)) flush();
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int i = m0 + tx + 8 * a, j = n0 + ty + 8 * b;
      if (i >= M || j >= N || (structure == GEMM_HERM && i < j)) continue;   // i < j: mirrored from (j, i)
      const double2 v = sizeof(C) == sizeof(float2) ? sum[a][b] : to_d(acc[a][b]);
      if (ksplit > 1) {
        part[((long)kz * N + j) * (long)M + i] = v;
        continue;
      }
      put_output(Cm + i + (long)j * ldc, beta, make_double2(alpha.x * v.x - alpha.y * v.y, alpha.x * v.y + alpha.y * v.x));
      if (structure == GEMM_HERM && i != j)   // alpha conj(v)
        put_output(Cm + j + (long)i * ldc, beta, make_double2(alpha.x * v.x + alpha.y * v.y, alpha.y * v.x - alpha.x * v.y));
    }
}

// Sums the split-K partials in a fixed order: G groups of a block's threads (32 entries each)
// sum consecutive runs of partials, then add up in shared memory. For GEMM_HERM the partials
// exist on and below the diagonal; an entry above it is the conjugate of its mirror. Bound by
// the partials' read and by FP64 additions; 32 entries side by side read whole lines where
// four a warp read 64 bytes at a time (Si64 step, 42 sums of 152 partials of 128 x 128: 38.85 ->
// 38.6 ms).
template <int G>
__global__ void __launch_bounds__(256) k_splitk_reduce(int M, int N, int ksplit, int structure, double2 alpha,
                                                       const double2* __restrict__ part, double2 beta,
                                                       double2* __restrict__ Cm, long ldc) {
  grid_entry();
  constexpr int E = 256 / G;   // entries of a block
  __shared__ double2 sums[G > 1 ? G - 1 : 1][E];
  const long total = (long)M * N;
  const int g = threadIdx.x / E, at = threadIdx.x % E;
  const int run = (ksplit + G - 1) / G;
  const int z0 = g * run, z1 = min(ksplit, z0 + run);
  const long t = (long)blockIdx.x * E + at;
  const int i = (int)(t % M), j = (int)(t / M);
  const bool in = t < total, mirror = structure == GEMM_HERM && i < j;
  double2 s = make_double2(0.0, 0.0);
  if (in) {
    const double2* p = part + (mirror ? (long)i * M + j : t);
#pragma unroll 8
    for (int kz = z0; kz < z1; ++kz) {
      const double2 v = p[(long)kz * total];
      s.x += v.x;
      s.y += v.y;
    }
  }
  if (G > 1) {
    if (g > 0) sums[g - 1][at] = s;
    __syncthreads();
    if (g > 0) return;
#pragma unroll
    for (int q = 0; q < G - 1; ++q) {
      s.x += sums[q][at].x;
      s.y += sums[q][at].y;
    }
  }
  if (!in) return;
  if (mirror) s.y = -s.y;
  put_output(Cm + i + (long)j * ldc, beta, make_double2(alpha.x * s.x - alpha.y * s.y, alpha.x * s.y + alpha.y * s.x));
}

static cudaError_t reduce_partials(int M, int N, int ksplit, int structure, double2 alpha, const double2* part,
                                   double2 beta, double2* C, long ldc, cudaStream_t s) {
  const long total = (long)M * N;
  // eight groups while one per entry would leave the chip mostly idle
  const int G = ksplit >= 8 && total < 65536 ? 8 : 1;
  const unsigned blocks = (unsigned)((total * G + 255) / 256);
  if (G == 8) launch(blocks, 256, 0, s)(k_splitk_reduce<8>, M, N, ksplit, structure, alpha, part, beta, C, ldc);
  else launch(blocks, 256, 0, s)(k_splitk_reduce<1>, M, N, ksplit, structure, alpha, part, beta, C, ldc);
  launched();
  return cudaGetLastError();
}

int sm_count() {
  static std::atomic<int> count[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
  int sms = count[dev & 63].load(std::memory_order_relaxed);
  if (sms == 0) {
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    sms = std::max(1, sms);
    count[dev & 63].store(sms, std::memory_order_relaxed);
  }
  return sms;
}

// Chunks of the reduction: of those that the workspace allows, the fewest within 3% (FP32: 1%)
// of the least time. FP64: the blocks of an SM share its multiply pipe, so the time goes as the
// blocks of the fullest SM times the chunk length, and chunks of half a slice pay (FP64 step
// of Si8 5.64 ms, 5.74 with whole slices). FP32 (microseconds, small32_us): a block alone on
// its SM waits for its slices, and hides the waits of a few others.
static int choose_split64(long tiles, int K, long out_elems, size_t ws_elems) {
  const long sms = sm_count();
  const long most = std::max<long>(1, std::min<long>({(long)(K / 8), (long)(ws_elems / out_elems), 4 * sms}));
  auto cost = [&](long ks) { return (double)((tiles * ks + sms - 1) / sms) * (double)((K + ks - 1) / ks); };
  double least = cost(1);
  for (long ks = 2; ks <= most; ++ks) least = std::min(least, cost(ks));
  for (long ks = 1; ks <= most; ++ks)
    if (cost(ks) <= 1.03 * least) return (int)ks;
  return 1;
}

// Microseconds that summing ks partials of an output takes: a launch, the wait for the first
// partials of a thread, one after the other, and their bytes.
static double reduce_us(long ks, long out_elems) {
  if (ks <= 1) return 0.0;
  return 2.0 + 0.06 * (double)std::min(ks, 32L) + 1.5e-5 * (double)out_elems + (double)ks * (double)out_elems * 32 / 8e6;
}

// The FP32 kernel on `tiles` tiles of 16 x 16 in ks chunks: a step along the reduction takes a
// block alone on its SM 54 ns, b blocks 16 + 10.3 b (fitted to 33 products, 16 x 16 to 4096 x
// 32 by 300 to 60,000, each in 1 to 1024 chunks; 32 x 300 by 60,000 took 830 us in the four
// chunks that give every SM one block, 191 in 128).
static double small32_us(long tiles, long K, long ks, long out_elems, long sms) {
  const long blocks = (tiles * ks + sms - 1) / sms;
  const long steps = ((K + ks - 1) / ks + GK - 1) / GK * GK;
  return 1e-3 * (double)steps * std::max(54.0, 16.0 + 10.3 * (double)blocks) + reduce_us(ks, out_elems);
}

static int choose_split32(long tiles, int K, long out_elems, size_t ws_elems) {
  constexpr long kMost = 256;
  const long sms = sm_count(), slices = ((long)K + GK - 1) / GK;
  const long most = std::max<long>(1, std::min<long>({slices, (long)(ws_elems / out_elems), kMost}));
  // the fewest chunks of each length: q slices, then q - 1 or the next that leaves fewer chunks
  int chunks[kMost], n = 0;
  double us[kMost], least = 0.0;
  for (long ks = 1; ks <= most;) {
    chunks[n] = (int)ks;
    us[n] = small32_us(tiles, K, ks, out_elems, sms);
    least = n == 0 ? us[0] : std::min(least, us[n]);
    ++n;
    const long q = (slices + ks - 1) / ks;
    if (q <= 1) break;
    ks = (slices + q - 2) / (q - 1);
  }
  for (int i = 0; i < n; ++i)
    if (us[i] <= 1.01 * least) return chunks[i];
  return 1;
}

template <typename C, typename TI>
static cudaError_t gemm_impl(int opA, int opB, int M, int N, int K, double2 alpha, const TI* A, long lda, const TI* B,
                             long ldb, double2 beta, double2* Cm, long ldc, double2* ws, size_t ws_elems,
                             cudaStream_t s, int structure) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (structure == GEMM_HERM && M != N) return cudaErrorInvalidValue;
  const long tm = ((long)M + GT - 1) / GT, tn = ((long)N + GT - 1) / GT;
  const long tiles = structure == GEMM_HERM ? tm * (tm + 1) / 2 : tm * tn;
  // grid axis y takes 65,535 tiles, x any number: a longer row of tiles goes along x
  const int swapped = tn > 65535;
  if (std::min(tm, tn) > 65535 || (structure == GEMM_HERM && tiles > INT_MAX)) return cudaErrorInvalidValue;
  int ksplit = 1;
  if (K > 0 && ws != nullptr)
    ksplit = sizeof(C) == sizeof(double2) ? choose_split64(tiles, K, (long)M * N, ws_elems)
                                          : choose_split32(tiles, K, (long)M * N, ws_elems);
  const int kchunk = std::max(1, (K + ksplit - 1) / ksplit);
  // GEMM_HERM: only the lower triangle's tiles, as blocks that return at once would leave some
  // SMs with seven of the others and some with four (Psi^H Psi of Si216: 41.5 ms, 30.6 so)
  const dim3 grid = structure == GEMM_HERM ? dim3((unsigned)tiles, 1, (unsigned)ksplit)
                    : swapped              ? dim3((unsigned)tn, (unsigned)tm, (unsigned)ksplit)
                                           : dim3((unsigned)tm, (unsigned)tn, (unsigned)ksplit);
#define PT_GEMM(OA, OB) \
  launch(grid, 64, 0, s)(k_gemm<C, TI, OA, OB>, M, N, K, kchunk, ksplit, structure, swapped, alpha, A, lda, B, ldb, beta, Cm, ldc, ws)
  if (opA == OP_N && opB == OP_N) PT_GEMM(OP_N, OP_N);
  else if (opA == OP_N) PT_GEMM(OP_N, OP_H);
  else if (opB == OP_N) PT_GEMM(OP_H, OP_N);
  else PT_GEMM(OP_H, OP_H);
#undef PT_GEMM
  launched();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || ksplit == 1) return e;
  return reduce_partials(M, N, ksplit, structure, alpha, ws, beta, Cm, ldc, s);
}

cudaError_t gemm64(int opA, int opB, int M, int N, int K, double2 alpha, const double2* A, long lda, const double2* B,
                   long ldb, double2 beta, double2* C, long ldc, double2* ws, size_t ws_elems, cudaStream_t s,
                   int structure) {
  return gemm_impl<double2>(opA, opB, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, ws, ws_elems, s, structure);
}

cudaError_t gemm32_small(int opA, int opB, int M, int N, int K, double2 alpha, const float2* A, long lda,
                         const float2* B, long ldb, double2 beta, double2* C, long ldc, double2* ws, size_t ws_elems,
                         cudaStream_t s, int structure) {
  return gemm_impl<float2>(opA, opB, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, ws, ws_elems, s, structure);
}

cudaError_t gemm32_small(int opA, int opB, int M, int N, int K, double2 alpha, const double2* A, long lda,
                         const double2* B, long ldb, double2 beta, double2* C, long ldc, double2* ws, size_t ws_elems,
                         cudaStream_t s, int structure) {
  return gemm_impl<float2>(opA, opB, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, ws, ws_elems, s, structure);
}

cudaError_t splitk_reduce(int M, int N, int ksplit, double2 alpha, const double2* part, double2 beta, double2* C,
                          long ldc, cudaStream_t s) {
  return reduce_partials(M, N, ksplit, GEMM_GENERAL, alpha, part, beta, C, ldc, s);
}

// ---------------------------------------------------------------------------
// Cholesky, right-looking by panels of CB columns: one block factors the diagonal block
// and inverts its factor, the rows below are multiplied by that inverse, and the trailing
// matrix takes the rank-CB update: 3 launches per CB columns. Bound by FP64 (two
// multiply-adds a clock and SM) in the single diagonal block, so only one thread takes
// each pivot's square root and reciprocal.
constexpr int CB = 32;

// Factor of the nb x nb block at (j0, j0), zeros above its diagonal, and the factor's
// inverse into the same block of Linv, both column by column. The last warp keeps the
// diagonal, a lane per entry: it takes the next pivot's square root and reciprocal
// while the others update the entries below the diagonal and the rows of the inverse (32
// columns: 75 us when every thread waited for the pivot, 45 so).
constexpr int kCholUpdate = 224;

__global__ void __launch_bounds__(kCholUpdate + 32) k_chol_diag(double2* __restrict__ A, double2* __restrict__ Linv,
                                                                int n, int j0, int* __restrict__ status) {
  grid_entry();
  constexpr int NT = kCholUpdate + 32;
  __shared__ double2 a[CB][CB + 1], x[CB][CB + 1];
  __shared__ double rinv[CB];
  __shared__ int bad;
  // entries (i, k), k < i < nb, by falling k: those a column j still changes (k > j) come first
  __shared__ unsigned char ent[CB * (CB - 1) / 2][2];
  if (*status != 0) return;
  const int tid = threadIdx.x, nb = min(CB, n - j0), lane = tid - kCholUpdate;
  double2* Ab = A + j0 + (long)j0 * n;
  double2* Xb = Linv + j0 + (long)j0 * n;
  if (tid == 0) bad = 0;
  for (int t = tid; t < nb * nb; t += NT) {
    const int i = t % nb, k = t / nb;
    a[i][k] = i >= k ? Ab[i + (long)k * n] : make_double2(0.0, 0.0);
    x[i][k] = make_double2(i == k ? 1.0 : 0.0, 0.0);
  }
  if (lane > 0 && lane < nb) {
    const int k = nb - 1 - lane;
    int at = lane * (lane - 1) / 2;   // after 1, 2, .. entries of the later columns
    for (int i = k + 1; i < nb; ++i, ++at) {
      ent[at][0] = (unsigned char)i;
      ent[at][1] = (unsigned char)k;
    }
  }
  __syncthreads();
  double diag = lane >= 0 && lane < nb ? a[lane][lane].x : 0.0;
  auto pivot = [&](int j) {   // by the diagonal's warp
    const double d = __shfl_sync(0xffffffffu, diag, j);
    const double s = sqrt(d);
    if (lane == 0) {
      if (d > 0.0) {
        a[j][j] = make_double2(s, 0.0);
        rinv[j] = 1.0 / s;
      } else {
        bad = 1;
      }
    }
  };
  if (lane >= 0) pivot(0);
  __syncthreads();
  for (int j = 0; j < nb; ++j) {
    if (bad) {
      if (tid == 0) *status = 1;
      return;
    }
    const double r = rinv[j];
    if (tid < nb) {   // column j of the factor, row j of the inverse
      double2& v = tid > j ? a[tid][j] : x[j][tid];
      v = make_double2(v.x * r, v.y * r);
    }
    __syncthreads();
    if (j + 1 == nb) break;
    if (lane >= 0) {
      if (lane > j && lane < nb) {
        const double2 u = a[lane][j];
        diag -= u.x * u.x + u.y * u.y;
      }
      pivot(j + 1);
    } else {
      const int m = nb - 1 - j, low = m * (m - 1) / 2;
      for (int t = tid; t < low + m * (j + 1); t += kCholUpdate) {
        if (t < low) {
          const int i = ent[t][0], k = ent[t][1];
          const double2 u = a[i][j], w = a[k][j];
          a[i][k].x -= u.x * w.x + u.y * w.y;
          a[i][k].y -= u.y * w.x - u.x * w.y;
        } else {
          const int k = j + 1 + (t - low) % m, c = (t - low) / m;
          const double2 l = a[k][j], v = x[j][c];
          x[k][c].x -= l.x * v.x - l.y * v.y;
          x[k][c].y -= l.x * v.y + l.y * v.x;
        }
      }
    }
    __syncthreads();
  }
  for (int t = tid; t < nb * nb; t += NT) {
    const int i = t % nb, k = t / nb;
    Ab[i + (long)k * n] = a[i][k];
    Xb[i + (long)k * n] = x[i][k];
  }
}

// Rows below the diagonal block: A21 <- A21 L11^{-H}, eight rows per block; the block's part
// of the columns j0.. above the diagonal (rows of A12) is zeroed.
__global__ void __launch_bounds__(256) k_chol_panel(double2* __restrict__ A, const double2* __restrict__ Linv, int n,
                                                    int j0, const int* __restrict__ status) {
  grid_entry();
  __shared__ double2 a[8][CB + 1], x[CB][CB + 1];
  if (*status != 0) return;
  const int tid = threadIdx.x, i0 = j0 + CB + 8 * blockIdx.x;
  const int r = tid & 7, k = tid >> 3;
  for (int t = tid; t < CB * CB; t += 256) x[t % CB][t / CB] = Linv[j0 + t % CB + (long)(j0 + t / CB) * n];
  const bool in = i0 + r < n;
  double2* p = A + i0 + r + (long)(j0 + k) * n;
  a[r][k] = in ? *p : make_double2(0.0, 0.0);
  __syncthreads();
  double2 s = make_double2(0.0, 0.0);
  for (int m = 0; m <= k; ++m) {
    const double2 u = a[r][m], w = x[k][m];
    s.x += u.x * w.x + u.y * w.y;
    s.y += u.y * w.x - u.x * w.y;
  }
  if (!in) return;
  *p = s;
  A[j0 + k + (long)(i0 + r) * n] = make_double2(0.0, 0.0);
}

// A22 -= L21 L21^H on and below the diagonal, one 16 x 16 tile per block
__global__ void __launch_bounds__(256) k_chol_trail(double2* __restrict__ A, int n, int j0,
                                                    const int* __restrict__ status) {
  grid_entry();
  __shared__ double2 u[CB][17], w[CB][17];
  if (blockIdx.x < blockIdx.y || *status != 0) return;
  const int tid = threadIdx.x, base = j0 + CB;
  const int i0 = base + 16 * blockIdx.x, k0 = base + 16 * blockIdx.y;
  for (int t = tid; t < 16 * CB; t += 256) {
    const int i = t & 15, m = t >> 4;
    const double2 z = make_double2(0.0, 0.0);
    u[m][i] = i0 + i < n ? A[i0 + i + (long)(j0 + m) * n] : z;
    w[m][i] = k0 + i < n ? A[k0 + i + (long)(j0 + m) * n] : z;
  }
  __syncthreads();
  const int i = i0 + (tid & 15), k = k0 + (tid >> 4);
  if (i >= n || k > i) return;
  double2 s = A[i + (long)k * n];
#pragma unroll 8
  for (int m = 0; m < CB; ++m) {
    const double2 a = u[m][tid & 15], b = w[m][tid >> 4];
    s.x -= a.x * b.x + a.y * b.y;
    s.y -= a.y * b.x - a.x * b.y;
  }
  A[i + (long)k * n] = s;
}

// Column c of L^{-1}: solve L x = e_c by forward substitution (one block per column), with the
// pivots' reciprocals taken at the start and the next column of L on its way during a step
// (n = 128: 185 us with a division by every thread in every step, and the column then loaded).
__global__ void __launch_bounds__(128) k_tri_inverse(const double2* __restrict__ L, double2* __restrict__ Li, int n) {
  grid_entry();
  extern __shared__ double2 b[];
  double* rinv = reinterpret_cast<double*>(b + n);
  constexpr int PRE = 4;   // rows of a thread whose entries are fetched a step ahead
  const int c = blockIdx.x, tid = threadIdx.x;
  for (int i = tid; i < n; i += 128) {
    b[i] = make_double2(i == c ? 1.0 : 0.0, 0.0);
    rinv[i] = 1.0 / L[i + (long)i * n].x;   // real and positive
  }
  double2 pre[PRE];
  auto fetch = [&](int i) {
#pragma unroll
    for (int q = 0; q < PRE; ++q) {
      const int k = tid + 128 * q;
      if (i < n && k > i && k < n) pre[q] = L[k + (long)i * n];
    }
  };
  fetch(c);
  __syncthreads();
  for (int i = c; i < n; ++i) {
    const double2 bi = b[i];
    const double r = rinv[i];
    const double2 xi = make_double2(bi.x * r, bi.y * r);
    auto update = [&](int k, double2 l) {
      double2 v = b[k];
      v.x -= l.x * xi.x - l.y * xi.y;
      v.y -= l.x * xi.y + l.y * xi.x;
      b[k] = v;
    };
    double2 now[PRE];
#pragma unroll
    for (int q = 0; q < PRE; ++q) now[q] = pre[q];
    fetch(i + 1);
#pragma unroll
    for (int q = 0; q < PRE; ++q) {
      const int k = tid + 128 * q;
      if (k > i && k < n) update(k, now[q]);
    }
    for (int k = tid + 128 * PRE; k < n; k += 128)
      if (k > i) update(k, L[k + (long)i * n]);
    __syncthreads();
  }
  for (int i = tid; i < n; i += 128)
    Li[i + (long)c * n] = i < c ? make_double2(0.0, 0.0) : make_double2(b[i].x * rinv[i], b[i].y * rinv[i]);
}

cudaError_t cholesky_inverse(double2* A, double2* Linv, int n, int* d_status, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(d_status, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  for (int j0 = 0; j0 < n; j0 += CB) {
    launch(1, kCholUpdate + 32, 0, s)(k_chol_diag, A, Linv, n, j0, d_status); launched();
    const int rest = n - j0 - CB;
    if (rest <= 0) continue;
    launch((rest + 7) / 8, 256, 0, s)(k_chol_panel, A, Linv, n, j0, d_status); launched();
    const unsigned t = (unsigned)((rest + 15) / 16);
    launch(dim3(t, t), 256, 0, s)(k_chol_trail, A, n, j0, d_status); launched();
  }
  if (n > CB) {
    const size_t smem = (sizeof(double2) + sizeof(double)) * n;
    if (smem > 48 * 1024) {
      e = cudaFuncSetAttribute(k_tri_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    launch(n, 128, smem, s)(k_tri_inverse, A, Linv, n); launched();
  }
  return cudaGetLastError();
}

}  // namespace pt
