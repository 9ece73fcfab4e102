// Generic batched 3D transforms between the planewave basis and the real-space
// grid (orbitals, density, local potential of Eq. 2; Sec. 3.2 and 3.4).
// A 3D FFT is three passes over global memory, one per axis:
//   rows   (axis 2, contiguous lines): a block owns whole rows,
//   cols   (axis 1 or 0): a block owns an L x C tile of C consecutive i2
//          columns so that every global access is a run of C elements.
// The axis-0 pass can fuse "inverse, multiply by a real field, forward"
// (local potential times orbital) or "forward, multiply by a reciprocal-space
// factor, inverse" (Hartree solve), so those operations cost no extra pass.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "common.cuh"
#include "fft.cuh"
#include "fft_ct.cuh"
#include "internal.h"

namespace pt {

int twiddle_offset(int L) {
  int off = 0;
  for (int i = 0; i < kNumLengths; ++i) {
    if (kLengths[i] == L) return off;
    off += kLengths[i];
  }
  return -1;
}

void twiddle_host(double2* out) {
  int off = 0;
  for (int i = 0; i < kNumLengths; ++i) {
    const int L = kLengths[i];
    for (int t = 0; t < L; ++t) {
      const double a = 2.0 * M_PI * (double)t / (double)L;
      out[off + t] = make_double2(std::cos(a), -std::sin(a));
    }
    off += L;
  }
}

template <> const void* DevTwiddles::base<double>() const { return d64; }
template <> const void* DevTwiddles::base<float>() const { return d32; }

template <typename T>
static const cplx<T>* tw_for(const DevTwiddles& tw, int L) {
  return reinterpret_cast<const cplx<T>*>(tw.base<T>()) + twiddle_offset(L);
}

static int round_threads(int t) {
  t = ((t + 31) / 32) * 32;
  return std::max(64, std::min(1024, t));
}

// ---------------------------------------------------------------------------
template <typename T, bool INV>
__global__ void k_rows(const cplx<T>* __restrict__ in, cplx<T>* __restrict__ out, long nrows, int L, int rpc,
                       const cplx<T>* __restrict__ tw_g, T scale, const T* __restrict__ mul, long rows_per_vol) {
  grid_entry();
  using C = cplx<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf = tw + L;
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int t = tid; t < L; t += nthr) tw[t] = tw_g[t];
  const long r0 = (long)blockIdx.x * rpc;
  const int nr = (int)min((long)rpc, nrows - r0);
  const int cnt = nr * L;
  const C* src = in + r0 * L;
  for (int e = tid; e < cnt; e += nthr) {
    C v = src[e];
    if (mul != nullptr) {
      const long row = r0 + e / L;
      v = cscale(v, mul[(row % rows_per_vol) * L + (e % L)]);
    }
    buf[e] = v;
  }
  __syncthreads();
  fft_lines<T, INV, true>(buf, L, nr, L, 1, tw, tid, nthr);
  C* dst = out + r0 * L;
  for (int e = tid; e < cnt; e += nthr) dst[e] = cscale(buf[e], scale);
}

template <typename T, bool INV, int MODE>
__global__ void k_cols(cplx<T>* __restrict__ data, int n0, int n1, int n2, int axis, int chunk,
                       const cplx<T>* __restrict__ tw_g, T scale, const T* __restrict__ mul) {
  grid_entry();
  using C = cplx<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int L = axis == 0 ? n0 : n1;
  const long S = axis == 0 ? (long)n1 * n2 : (long)n2;
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf = tw + L;
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int t = tid; t < L; t += nthr) tw[t] = tw_g[t];
  const int i2s = blockIdx.x * chunk;
  const int nc = min(chunk, n2 - i2s);
  const int u = blockIdx.y;
  const long N = (long)n0 * n1 * n2;
  C* base = data + (long)blockIdx.z * N + (axis == 1 ? (long)u * n1 * n2 : (long)u * n2) + i2s;
  const int cnt = L * nc;
  for (int idx = tid; idx < cnt; idx += nthr) {
    const int e = idx / nc, c = idx - e * nc;
    buf[e * chunk + c] = base[e * S + c];
  }
  __syncthreads();
  fft_lines<T, INV, false>(buf, L, nc, 1, chunk, tw, tid, nthr);
  if (MODE != 0) {
    for (int idx = tid; idx < cnt; idx += nthr) {
      const int e = idx / nc, c = idx - e * nc;
      // axis 0 only: point (e, u, i2s + c)
      const long flat = ((long)e * n1 + u) * n2 + i2s + c;
      buf[e * chunk + c] = cscale(buf[e * chunk + c], mul[flat]);
    }
    __syncthreads();
    fft_lines<T, !INV, false>(buf, L, nc, 1, chunk, tw, tid, nthr);
  }
  for (int idx = tid; idx < cnt; idx += nthr) {
    const int e = idx / nc, c = idx - e * nc;
    base[e * S + c] = cscale(buf[e * chunk + c], scale);
  }
}

template <typename T>
cudaError_t fft_rows(const void* in, void* out, long nvol, Grid3 g, int inverse, double scale, const T* mul_real,
                     const DevTwiddles& tw, cudaStream_t s) {
  using C = cplx<T>;
  const int L = g.n2;
  if (!fft_length_supported(L)) return cudaErrorInvalidValue;
  const long nrows = nvol * g.n0 * g.n1;
  // rows per block: aim at ~4-8 KB of data per block
  int rpc = std::max(1, (int)(8192 / (L * (int)sizeof(C))));
  rpc = std::min<long>(rpc, nrows);
  const bool fp64 = sizeof(T) == 8;
  const int nthr = round_threads(fft_threads_needed(L, rpc, fp64));
  const size_t smem = (size_t)(L + rpc * L) * sizeof(C);
  const long nblk = (nrows + rpc - 1) / rpc;
  const T sc = (T)scale;
  const long rpv = (long)g.n0 * g.n1;
  if (inverse)
    launch((unsigned)nblk, nthr, smem, s)(k_rows<T, true>, (const C*)in, (C*)out, nrows, L, rpc, tw_for<T>(tw, L), sc,
                                                      mul_real, rpv);
  else
    launch((unsigned)nblk, nthr, smem, s)(k_rows<T, false>, (const C*)in, (C*)out, nrows, L, rpc, tw_for<T>(tw, L), sc,
                                                       mul_real, rpv);
  launched();
  return cudaGetLastError();
}

template <typename T>
cudaError_t fft_cols(void* data, long nvol, Grid3 g, int axis, int inverse, int mode, double scale, const T* mul_real,
                     const DevTwiddles& tw, cudaStream_t s) {
  using C = cplx<T>;
  const int L = axis == 0 ? g.n0 : g.n1;
  if (!fft_length_supported(L)) return cudaErrorInvalidValue;
  if (mode != 0 && (axis != 0 || mul_real == nullptr)) return cudaErrorInvalidValue;
  int chunk = sizeof(T) == 4 ? 16 : 8;
  chunk = std::min(chunk, g.n2);
  const bool fp64 = sizeof(T) == 8;
  const int nthr = round_threads(fft_threads_needed(L, chunk, fp64));
  const size_t smem = (size_t)(L + L * chunk) * sizeof(C);
  dim3 grid((g.n2 + chunk - 1) / chunk, axis == 0 ? g.n1 : g.n0, (unsigned)nvol);
  const T sc = (T)scale;
  const C* twp = tw_for<T>(tw, L);
#define PT_COLS(INV, MODE) launch(grid, nthr, smem, s)(k_cols<T, INV, MODE>, (C*)data, g.n0, g.n1, g.n2, axis, chunk, twp, sc, mul_real)
  if (mode == 0) {
    if (inverse) PT_COLS(true, 0); else PT_COLS(false, 0);
  } else if (mode == 1) {
    PT_COLS(true, 1);   // inverse, multiply, forward
  } else {
    PT_COLS(false, 2);  // forward, multiply, inverse
  }
#undef PT_COLS
  launched();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Convolution of a real field with an even real reciprocal-space factor (the Hartree solve,
// the Kerker mixing) on cubic grids of 32 to 96 points: a block transforms a whole plane
// (axes 1 and 2) in shared memory, so the solve takes three launches instead of seven, with
// the field's load, the factor and the potential's assembly inside them. FP64 arithmetic and
// latency bound it (one volume is little work), so the transforms use that the field is
// real: two rows share one complex line, and only the frequencies 0..L/2 of axis 2 are kept.
// The three launches at 32^3: 40 us, 48 with complex fields (64^3 with complex fields: 140).
namespace {

template <int L> struct ConvCfg {
  static constexpr int H = L / 2 + 1;                              // columns of the half spectrum
  static constexpr int HS = H | 1;                                 // odd row stride
  static constexpr int NT = L == 32 ? 128 : L == 48 ? 192 : L == 64 ? 256 : 384;   // plane kernels
  // columns of an axis-0 block: at 32, 136 blocks of four instead of 68 of eight
  static constexpr int NC = L == 32 ? 4 : 8;
  static constexpr int NT0 = L == 32 ? 32 : L == 64 ? 64 : 96;
  static constexpr size_t smem_plane = sizeof(double2) * (L + L / 2 * (L + 1) + L * HS);
  static constexpr size_t smem_axis0 = sizeof(double2) * (L + L * (NC + 1));
};

// plane i0 of a (minus b, when given), transformed along axes 2 and 1, frequencies 0..L/2 of
// axis 2; the blocks beyond the planes write the part of the local potential that does not
// wait for the result, on SMs the planes leave idle
template <int L>
__global__ void __launch_bounds__(ConvCfg<L>::NT) k_conv_plane_fwd(const double* __restrict__ a,
                                                                   const double* __restrict__ b,
                                                                   double2* __restrict__ out, ConvSink sink,
                                                                   const double2* __restrict__ tw_g) {
  grid_entry();
  constexpr int NT = ConvCfg<L>::NT, H = ConvCfg<L>::H, HS = ConvCfg<L>::HS, W = L + 1;
  if (blockIdx.x >= L) {
#pragma unroll 2
    for (int p = (blockIdx.x - L) * NT + threadIdx.x; p < L * L * L; p += (gridDim.x - L) * NT)
      sink.vloc[p] = static_potential(sink, p);
    return;
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* tw = reinterpret_cast<double2*>(smem_raw);
  double2* buf = tw + L;             // [row pair][i2]
  double2* half = buf + L / 2 * W;   // [i1][frequency]
  const int tid = threadIdx.x;
  const long off = (long)blockIdx.x * L * L;
  for (int t = tid; t < L; t += NT) tw[t] = tw_g[t];
#pragma unroll 4
  for (int e = tid; e < L / 2 * L; e += NT) {
    const int r = e / L, i2 = e % L;
    const long p = off + 2 * r * L + i2;
    double2 v = make_double2(a[p], a[p + L]);
    if (b != nullptr) v = make_double2(v.x - b[p], v.y - b[p + L]);
    buf[r * W + i2] = v;
  }
  __syncthreads();
  ct_forward<double2, L, L / 2, NT, W, 1>(buf, L / 2, tw, tid);
  // the two rows of a line: (Z_k + conj Z_-k) / 2 and (Z_k - conj Z_-k) / 2i
  for (int e = tid; e < L / 2 * H; e += NT) {
    const int r = e / H, k = e % H;
    const double2 z = buf[r * W + k], c = buf[r * W + (k ? L - k : 0)];
    half[2 * r * HS + k] = make_double2(0.5 * (z.x + c.x), 0.5 * (z.y - c.y));
    half[(2 * r + 1) * HS + k] = make_double2(0.5 * (z.y + c.y), 0.5 * (c.x - z.x));
  }
  __syncthreads();
  ct_forward<double2, L, H, NT, 1, HS>(half, H, tw, tid);
  double2* o = out + (long)blockIdx.x * L * H;
#pragma unroll 4
  for (int e = tid; e < L * H; e += NT) o[e] = half[(e / H) * HS + e % H];
}

// axis 0 of NC columns: forward, times f, inverse, in place
template <int L>
__global__ void __launch_bounds__(ConvCfg<L>::NT0) k_conv_axis0(double2* __restrict__ data,
                                                                const double* __restrict__ f,
                                                                const double2* __restrict__ tw_g) {
  grid_entry();
  constexpr int NT = ConvCfg<L>::NT0, NC = ConvCfg<L>::NC, H = ConvCfg<L>::H;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* tw = reinterpret_cast<double2*>(smem_raw);
  double2* buf = tw + L;
  const int tid = threadIdx.x;
  const int c0 = blockIdx.x * NC, nc = min(NC, L * H - c0);
  for (int t = tid; t < L; t += NT) tw[t] = tw_g[t];
#pragma unroll 4
  for (int e = tid; e < L * NC; e += NT)
    if (e % NC < nc) buf[(e / NC) * (NC + 1) + e % NC] = data[(long)(e / NC) * L * H + c0 + e % NC];
  __syncthreads();
  ct_forward<double2, L, NC, NT, 1, NC + 1>(buf, nc, tw, tid);
  for (int e = tid; e < L * NC; e += NT) {
    if (e % NC >= nc) continue;
    const int col = c0 + e % NC;
    double2& v = buf[(e / NC) * (NC + 1) + e % NC];
    v = cscale(v, f[((long)(e / NC) * L + col / H) * L + col % H]);
  }
  __syncthreads();
  ct_inverse<double2, L, NC, NT, 1, NC + 1>(buf, nc, tw, tid);
#pragma unroll 4
  for (int e = tid; e < L * NC; e += NT)
    if (e % NC < nc) data[(long)(e / NC) * L * H + c0 + e % NC] = buf[(e / NC) * (NC + 1) + e % NC];
}

// plane i0 back along axes 1 and 2 (row pairs as one complex line), the result to the sink
template <int L>
__global__ void __launch_bounds__(ConvCfg<L>::NT) k_conv_plane_inv(const double2* __restrict__ in, ConvSink sink,
                                                                   const double2* __restrict__ tw_g) {
  grid_entry();
  constexpr int NT = ConvCfg<L>::NT, H = ConvCfg<L>::H, HS = ConvCfg<L>::HS, W = L + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* tw = reinterpret_cast<double2*>(smem_raw);
  double2* buf = tw + L;
  double2* half = buf + L / 2 * W;
  const int tid = threadIdx.x;
  const long off = (long)blockIdx.x * L * L;
  for (int t = tid; t < L; t += NT) tw[t] = tw_g[t];
  const double2* src = in + (long)blockIdx.x * L * H;
#pragma unroll 4
  for (int e = tid; e < L * H; e += NT) half[(e / H) * HS + e % H] = src[e];
  __syncthreads();
  ct_inverse<double2, L, H, NT, 1, HS>(half, H, tw, tid);
  for (int e = tid; e < L / 2 * L; e += NT) {   // Z_k = A_k + i B_k, A_-k = conj A_k
    const int r = e / L, k = e % L;
    const bool up = k < H;
    const double2 x = half[2 * r * HS + (up ? k : L - k)], y = half[(2 * r + 1) * HS + (up ? k : L - k)];
    buf[r * W + k] = up ? make_double2(x.x - y.y, x.y + y.x) : make_double2(x.x + y.y, y.x - x.y);
  }
  __syncthreads();
  ct_inverse<double2, L, L / 2, NT, W, 1>(buf, L / 2, tw, tid);
#pragma unroll 4
  for (int e = tid; e < L / 2 * L; e += NT) {
    const int r = e / L, i2 = e % L;
    const long p = off + 2 * r * L + i2;
    const double2 h = buf[r * W + i2];
    sink_result(sink, p, h.x);
    sink_result(sink, p + L, h.y);
  }
}

template <int L>
cudaError_t convolve_t(const double* a, const double* b, const double* f, double2* work, const ConvSink& sink,
                       const double2* tw, cudaStream_t s) {
  using G = ConvCfg<L>;
  static std::atomic<unsigned long long> attr_done{0};
  if (const unsigned long long bit = device_bit_todo(attr_done)) {
    cudaError_t e = cudaFuncSetAttribute(k_conv_plane_fwd<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)G::smem_plane);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_conv_plane_inv<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::smem_plane);
    if (e != cudaSuccess) return e;
    attr_done.fetch_or(bit, std::memory_order_release);
  }
  const int extra = sink.acc == nullptr ? std::max(32, sm_count() - L) : 0;
  launch(L + extra, G::NT, G::smem_plane, s)(k_conv_plane_fwd<L>, a, b, work, sink, tw);
  launch((L * G::H + G::NC - 1) / G::NC, G::NT0, G::smem_axis0, s)(k_conv_axis0<L>, work, f, tw);
  launch(L, G::NT, G::smem_plane, s)(k_conv_plane_inv<L>, work, sink, tw);
  launched(3);
  return cudaGetLastError();
}

}  // namespace

bool convolve_supported(Grid3 g) {
  return g.n0 == g.n1 && g.n1 == g.n2 && (g.n0 == 32 || g.n0 == 48 || g.n0 == 64 || g.n0 == 96);
}

cudaError_t convolve(const double* a, const double* b, const double* f, double2* work, const ConvSink& sink, Grid3 g,
                     const DevTwiddles& tw, cudaStream_t s) {
  const double2* t = tw_for<double>(tw, g.n0);
  switch (g.n0) {
    case 32: return convolve_t<32>(a, b, f, work, sink, t, s);
    case 48: return convolve_t<48>(a, b, f, work, sink, t, s);
    case 64: return convolve_t<64>(a, b, f, work, sink, t, s);
    case 96: return convolve_t<96>(a, b, f, work, sink, t, s);
    default: return cudaErrorInvalidValue;
  }
}

// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_scatter(const double2* __restrict__ in, long in_ld, cplx<T>* __restrict__ out, long N,
                          const int* __restrict__ basis, int npw, double scale) {
  grid_entry();
  const long v = blockIdx.y;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < npw; k += gridDim.x * blockDim.x) {
    const double2 c = in[v * in_ld + k];
    out[v * N + basis[k]] = cvt<cplx<T>>(make_double2(c.x * scale, c.y * scale));
  }
}

template <typename T>
__global__ void k_gather(const cplx<T>* __restrict__ in, double2* __restrict__ out, long out_ld, long N,
                         const int* __restrict__ basis, int npw, double scale, const double* __restrict__ kin,
                         const double2* __restrict__ x, long x_ld, int accumulate) {
  grid_entry();
  const long v = blockIdx.y;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < npw; k += gridDim.x * blockDim.x) {
    const double2 f = to_d(in[v * N + basis[k]]);
    double2 r = make_double2(f.x * scale, f.y * scale);
    if (kin != nullptr) {
      const double2 c = x[v * x_ld + k];
      r.x += kin[k] * c.x;
      r.y += kin[k] * c.y;
    }
    double2* o = out + v * out_ld + k;
    if (accumulate) { r.x += o->x; r.y += o->y; }
    *o = r;
  }
}

template <typename T>
cudaError_t scatter_basis(const double2* in, long in_ld, void* out, long nvol, Grid3 g, const int* basis, int npw,
                          double scale, cudaStream_t s) {
  using C = cplx<T>;
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(C) * g.N() * nvol, s);
  if (e != cudaSuccess) return e;
  dim3 grid((npw + 255) / 256, (unsigned)nvol);
  launch(grid, 256, 0, s)(k_scatter<T>, in, in_ld, (C*)out, g.N(), basis, npw, scale); launched();
  return cudaGetLastError();
}

template <typename T>
cudaError_t gather_basis(const void* in, double2* out, long out_ld, long nvol, Grid3 g, const int* basis, int npw,
                         double scale, const double* kin, const double2* x, long x_ld, int accumulate, cudaStream_t s) {
  using C = cplx<T>;
  dim3 grid((npw + 255) / 256, (unsigned)nvol);
  launch(grid, 256, 0, s)(k_gather<T>, (const C*)in, out, out_ld, g.N(), basis, npw, scale, kin, x, x_ld, accumulate); launched();
  return cudaGetLastError();
}

__global__ void k_c128_to_c64(const double2* __restrict__ in, float2* __restrict__ out, long n) {
  grid_entry();
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    out[i] = make_float2((float)in[i].x, (float)in[i].y);
}

cudaError_t convert_c128_to_c64(const double2* in, float2* out, long n, cudaStream_t s) {
  long blocks = std::min<long>((n + 255) / 256, 152L * 32);
  launch((unsigned)std::max<long>(blocks, 1), 256, 0, s)(k_c128_to_c64, in, out, n); launched();
  return cudaGetLastError();
}

// explicit instantiations
template cudaError_t fft_rows<float>(const void*, void*, long, Grid3, int, double, const float*, const DevTwiddles&, cudaStream_t);
template cudaError_t fft_rows<double>(const void*, void*, long, Grid3, int, double, const double*, const DevTwiddles&, cudaStream_t);
template cudaError_t fft_cols<float>(void*, long, Grid3, int, int, int, double, const float*, const DevTwiddles&, cudaStream_t);
template cudaError_t fft_cols<double>(void*, long, Grid3, int, int, int, double, const double*, const DevTwiddles&, cudaStream_t);
template cudaError_t scatter_basis<float>(const double2*, long, void*, long, Grid3, const int*, int, double, cudaStream_t);
template cudaError_t scatter_basis<double>(const double2*, long, void*, long, Grid3, const int*, int, double, cudaStream_t);
template cudaError_t gather_basis<float>(const void*, double2*, long, long, Grid3, const int*, int, double, const double*, const double2*, long, int, cudaStream_t);
template cudaError_t gather_basis<double>(const void*, double2*, long, long, Grid3, const int*, int, double, const double*, const double2*, long, int, cudaStream_t);

static std::atomic<unsigned long long> g_launches{0};
void launched(int n) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }
unsigned long long launch_count() { return g_launches.load(std::memory_order_relaxed); }

std::string cuda_msg(cudaError_t e) { return std::string(cudaGetErrorName(e)) + ": " + cudaGetErrorString(e); }

}  // namespace pt
