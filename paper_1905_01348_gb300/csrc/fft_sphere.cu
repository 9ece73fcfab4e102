// Transforms (FP32 or FP64) between the planewave sphere and the real-space grid for
// cubic grids of 32, 48, 64 or 96 points (the orbital transforms of the SCF loop,
// Sec. 3.2 and 3.4: real-space orbitals for the density and exchange, and the
// local-potential product of Eq. 2).
//
// The basis is the sphere |G|^2/2 <= ecut, a small part of the grid's
// frequency cube (about 6% at the workloads' cutoff). A 3D transform from the
// sphere therefore starts with few nonzero lines and only the last axis is
// full, and a transform to the sphere needs few outputs after its first axis:
//   to real space:  rows (axis 2) only for the live (i0, i1) rows, the basis
//                   coefficients scattered straight into them; axis 1 only on
//                   the live i0 planes, reading only their live rows; axis 0
//                   on every line, reading only the live planes.
//   to the sphere:  axis 0 on every line (the real-space product with the
//                   local potential fused into the load), storing only the
//                   live planes; axis 1 on the live planes, storing only the
//                   live rows; axis 2 on the live rows, gathering the basis
//                   coefficients straight from them.
// Rows and planes that no basis vector reaches are never read or written, so
// a pass never depends on what they hold. The transforms are exact: the
// skipped inputs are zero and the skipped outputs are not needed.
#include "common.cuh"
#include "fft_ct.cuh"
#include "fft_pk.cuh"
#include "internal.h"

namespace pt {

namespace {

constexpr int SNT = 64;   // threads per block
constexpr int SC = 16;    // lines (rows, or i2 columns) per block
constexpr int SW = SC + 1;

template <int L> constexpr int RW = L + 1;   // row stride of the row kernels

// Row kernels: SC live rows per block, rows of length L at stride L + 1.
template <typename C, int L> constexpr size_t smem_rows() { return sizeof(C) * (size_t)(L + SC * RW<L>); }
// Column kernels: an L x SC block (element e of column c at e * (SC + 1) + c).
template <typename C, int L> constexpr size_t smem_cols() { return sizeof(C) * (size_t)(L + L * SW); }

template <typename C> __device__ __forceinline__ C scaled(double2 a, double s) { return cvt<C>(make_double2(a.x * s, a.y * s)); }

// Inverse along axis 2 of SC live rows, the row's basis coefficients scattered in.
template <typename C, int L>
__global__ void __launch_bounds__(SNT) k_sph_rows_inv(const double2* __restrict__ coef, long ldc,
                                                      C* __restrict__ vol, const SphereTables st,
                                                      const int* __restrict__ basis, double scale,
                                                      const C* __restrict__ tw_g) {
  grid_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf = tw + L;
  const int tid = threadIdx.x;
  const int r0 = blockIdx.x * SC;
  const int nr = min(SC, st.nrows - r0);
  const long v = blockIdx.y;
  for (int t = tid; t < L; t += SNT) tw[t] = tw_g[t];
  for (int e = tid; e < SC * RW<L>; e += SNT) buf[e] = C{};
  __syncthreads();
  const int k0 = st.row_kbeg[r0], k1 = st.row_kbeg[r0 + nr];
  const double2* cv = coef + v * ldc;
  for (int k = k0 + tid; k < k1; k += SNT)
    buf[(st.krow[k] - r0) * RW<L> + basis[k] % L] = scaled<C>(cv[k], scale);
  __syncthreads();
  ct_inverse<C, L, SC, SNT, RW<L>, 1>(buf, nr, tw, tid);
  C* vv = vol + v * (long)L * L * L;
  for (int e = tid; e < nr * L; e += SNT) {
    const int rr = e / L, i2 = e % L;
    vv[(long)st.row_idx[r0 + rr] * L + i2] = buf[rr * RW<L> + i2];
  }
}

// Axis-1 transform of one live plane i0 over SC columns i2. INV: reads only the
// plane's live rows (others are zero), writes the whole plane block. Forward:
// reads the whole plane block, writes only the live rows.
template <typename C, int L, bool INV>
__global__ void __launch_bounds__(SNT) k_sph_axis1(C* __restrict__ vol, const SphereTables st,
                                                   const C* __restrict__ tw_g) {
  grid_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf = tw + L;
  const int tid = threadIdx.x;
  const int i2s = blockIdx.x * SC;
  const int i0 = st.planes[blockIdx.y];
  const long v = blockIdx.z;
  for (int t = tid; t < L; t += SNT) tw[t] = tw_g[t];
  C* base = vol + v * (long)L * L * L + (long)i0 * L * L + i2s;
  const unsigned char* live = st.rowlive + i0 * L;
  for (int idx = tid; idx < L * SC; idx += SNT) {
    const int i1 = idx / SC, c = idx % SC;
    buf[i1 * SW + c] = (!INV || live[i1]) ? base[(long)i1 * L + c] : C{};
  }
  __syncthreads();
  if (INV) ct_inverse<C, L, SC, SNT, 1, SW>(buf, SC, tw, tid);
  else ct_forward<C, L, SC, SNT, 1, SW>(buf, SC, tw, tid);
  for (int idx = tid; idx < L * SC; idx += SNT) {
    const int i1 = idx / SC, c = idx % SC;
    if (INV || live[i1]) base[(long)i1 * L + c] = buf[i1 * SW + c];
  }
}

// Axis-0 transform of the lines (i1, i2s..i2s+SC). INV: reads only the live
// planes, writes every plane. Forward: reads every plane (times the real field
// `mul` when given), writes only the live planes. `dst` may be `src`: a block
// reads all of its lines before it writes them.
template <typename C, int L, bool INV>
__global__ void __launch_bounds__(SNT) k_sph_axis0(const C* src, C* dst, const typename real_of<C>::type* __restrict__ mul,
                                                   const SphereTables st, const C* __restrict__ tw_g) {
  grid_entry();
  using R = typename real_of<C>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf = tw + L;
  const int tid = threadIdx.x;
  const int i2s = blockIdx.x * SC;
  const int i1 = blockIdx.y;
  const long v = blockIdx.z;
  for (int t = tid; t < L; t += SNT) tw[t] = tw_g[t];
  const long off = (long)i1 * L + i2s;
  const C* sb = src + v * (long)L * L * L + off;
  C* db = dst + v * (long)L * L * L + off;
  for (int idx = tid; idx < L * SC; idx += SNT) {
    const int i0 = idx / SC, c = idx % SC;
    C x{};
    if (!INV || st.planelive[i0]) {
      x = sb[(long)i0 * L * L + c];
      if (!INV && mul != nullptr) x = cscale(x, (R)__ldg(mul + (long)i0 * L * L + off + c));
    }
    buf[i0 * SW + c] = x;
  }
  __syncthreads();
  if (INV) ct_inverse<C, L, SC, SNT, 1, SW>(buf, SC, tw, tid);
  else ct_forward<C, L, SC, SNT, 1, SW>(buf, SC, tw, tid);
  for (int idx = tid; idx < L * SC; idx += SNT) {
    const int i0 = idx / SC, c = idx % SC;
    if (INV || st.planelive[i0]) db[(long)i0 * L * L + c] = buf[i0 * SW + c];
  }
}

// Forward along axis 2 of SC live rows, then out[k] = scale * F[k]
// (+ kin[k] x[k]) (+ out[k]) for the rows' basis vectors.
template <typename C, int L>
__global__ void __launch_bounds__(SNT) k_sph_rows_fwd(const C* __restrict__ vol, const SphereTables st,
                                                      const int* __restrict__ basis, double scale,
                                                      const double* __restrict__ kin, const double2* __restrict__ x,
                                                      long ldx, double2* __restrict__ out, long ldo, int accumulate,
                                                      const C* __restrict__ tw_g) {
  grid_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf = tw + L;
  const int tid = threadIdx.x;
  const int r0 = blockIdx.x * SC;
  const int nr = min(SC, st.nrows - r0);
  const long v = blockIdx.y;
  for (int t = tid; t < L; t += SNT) tw[t] = tw_g[t];
  const C* vv = vol + v * (long)L * L * L;
  for (int e = tid; e < nr * L; e += SNT) {
    const int rr = e / L, i2 = e % L;
    buf[rr * RW<L> + i2] = vv[(long)st.row_idx[r0 + rr] * L + i2];
  }
  __syncthreads();
  ct_forward<C, L, SC, SNT, RW<L>, 1>(buf, nr, tw, tid);
  const int k0 = st.row_kbeg[r0], k1 = st.row_kbeg[r0 + nr];
  double2* ov = out + v * ldo;
  const double2* xv = x != nullptr ? x + v * ldx : nullptr;
  for (int k = k0 + tid; k < k1; k += SNT) {
    const double2 f = to_d(buf[(st.krow[k] - r0) * RW<L> + basis[k] % L]);
    double2 r = make_double2(f.x * scale, f.y * scale);
    if (kin != nullptr) {
      const double2 c = xv[k];
      r.x += kin[k] * c.x;
      r.y += kin[k] * c.y;
    }
    if (accumulate) {
      const double2 o = ov[k];
      r.x += o.x;
      r.y += o.y;
    }
    ov[k] = r;
  }
}

// ---- FP32: packed pairs of lines (fft_pk.cuh) --------------------------------------
// The FP32 passes are bound by memory traffic once their transforms are cheap: a pk2 holds
// two neighbouring lines (i2, i2 + 1 in the column passes, two live rows in the row
// passes), loads and stores go straight between global memory and registers, and a value
// crosses shared memory once per pass, between the 8-point and the M-point DFTs (L = 8 M).
constexpr int CPB = 8;    // column pairs per block (16 columns)
constexpr int RPB = 8;    // row pairs per block

template <int L> struct Pk {
  static constexpr int M = L / 8;
  static constexpr int NT = 8 * (M > 8 ? M : 8);
  static constexpr int LS = L + 1;   // odd: neighbouring pairs on distinct banks
};

// twiddles W_L^(n1 k2) = c - i s as (c, c, s, s) at [k2][n1]
template <int L> __device__ __forceinline__ void load_tw(pk2* tw, const float2* __restrict__ tw_g, int tid) {
  for (int t = tid; t < L; t += Pk<L>::NT) {
    const float2 w = tw_g[(t / Pk<L>::M) * (t % Pk<L>::M)];
    tw[t] = {f2(w.x), f2(-w.y)};
  }
}

__device__ __forceinline__ pk2 pk_load(const float2* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {make_float2(v.x, v.z), make_float2(v.y, v.w)};
}
__device__ __forceinline__ void pk_store(float2* p, pk2 v) {
  *reinterpret_cast<float4*>(p) = make_float4(v.re.x, v.im.x, v.re.y, v.im.y);
}

// Axis-0 (AXIS 0: lines (i1, i2), blockIdx.y = i1) or axis-1 (blockIdx.y = live plane) pass over
// 16 columns i2. INV: reads only the live planes / the plane's live rows (others are
// zero), writes every element. Forward: reads every element (times `mul` when given),
// writes only the live ones. `dst` may be `src`.
template <int L, bool INV, int AXIS>
__global__ void __launch_bounds__(Pk<L>::NT) k_sphp_cols(const float2* src, float2* dst, const float* __restrict__ mul,
                                                         const SphereTables st, const float2* __restrict__ tw_g) {
  grid_entry();
  constexpr int M = Pk<L>::M, NT = Pk<L>::NT, LS = Pk<L>::LS;
  constexpr long S = AXIS == 0 ? (long)L * L : L;
  __shared__ pk2 tw[L];
  __shared__ pk2 ex[CPB * LS];
  __shared__ unsigned char live[L];
  const int tid = threadIdx.x, cp = tid % CPB, u = tid / CPB;
  const int line = AXIS == 0 ? (int)blockIdx.y : st.planes[blockIdx.y];
  const unsigned char* lv = AXIS == 0 ? st.planelive : st.rowlive + line * L;
  for (int t = tid; t < L; t += NT) live[t] = lv[t];
  load_tw<L>(tw, tw_g, tid);
  const long off = (AXIS == 0 ? (long)line * L : (long)line * L * L) + blockIdx.x * (2 * CPB) + 2 * cp;
  const long vol = (long)blockIdx.z * L * L * L;
  const float2* s = src + vol + off;
  float2* d = dst + vol + off;
  if (INV) {
    __syncthreads();   // live flags and twiddles
    if (u < 8) {
      pk2 v[M];
#pragma unroll
      for (int k1 = 0; k1 < M; ++k1)
        v[k1] = live[u + 8 * k1] ? pk_load(s + (u + 8 * k1) * S) : pk2{f2(0.f), f2(0.f)};
      pk_dft<M, true>(v);
      ex[cp * LS + u * M] = v[0];
#pragma unroll
      for (int m = 1; m < M; ++m) ex[cp * LS + u * M + m] = ptwiddle<true>(v[m], tw[u * M + m]);
    }
    __syncthreads();
    if (u < M) {
      pk2 v[8];
#pragma unroll
      for (int k2 = 0; k2 < 8; ++k2) v[k2] = ex[cp * LS + k2 * M + u];
      pk_dft<8, true>(v);
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) pk_store(d + (u + M * n2) * S, v[n2]);
    }
  } else {
    pk2 v[8];
    if (u < M) {
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) v[n2] = pk_load(s + (u + M * n2) * S);
      if (mul != nullptr) {
#pragma unroll
        for (int n2 = 0; n2 < 8; ++n2) {
          const float2 f = __ldg(reinterpret_cast<const float2*>(mul + off + (u + M * n2) * S));
          v[n2] = {vmul(v[n2].re, f), vmul(v[n2].im, f)};
        }
      }
      pk_dft<8, false>(v);
    }
    __syncthreads();
    if (u < M) {
      ex[cp * LS + u] = v[0];
#pragma unroll
      for (int k2 = 1; k2 < 8; ++k2) ex[cp * LS + k2 * M + u] = ptwiddle<false>(v[k2], tw[k2 * M + u]);
    }
    __syncthreads();
    if (u < 8) {
      pk2 w[M];
#pragma unroll
      for (int m = 0; m < M; ++m) w[m] = ex[cp * LS + u * M + m];
      pk_dft<M, false>(w);
#pragma unroll
      for (int k1 = 0; k1 < M; ++k1)
        if (live[u + 8 * k1]) pk_store(d + (u + 8 * k1) * S, w[k1]);
    }
  }
}

// Inverse along axis 2 of 16 live rows, the rows' basis coefficients scattered in.
template <int L>
__global__ void __launch_bounds__(Pk<L>::NT) k_sphp_rows_inv(const double2* __restrict__ coef, long ldc,
                                                             float2* __restrict__ vol, const SphereTables st,
                                                             const int* __restrict__ basis, double scale,
                                                             const float2* __restrict__ tw_g) {
  grid_entry();
  constexpr int M = Pk<L>::M, NT = Pk<L>::NT, LS = Pk<L>::LS;
  __shared__ pk2 tw[L];
  __shared__ pk2 buf[RPB * LS];
  const int tid = threadIdx.x, rp = tid % RPB, u = tid / RPB;
  const int r0 = blockIdx.x * (2 * RPB), nr = min(2 * RPB, st.nrows - r0);
  load_tw<L>(tw, tw_g, tid);
  for (int e = tid; e < RPB * LS; e += NT) buf[e] = pk2{f2(0.f), f2(0.f)};
  __syncthreads();
  const int kb = st.row_kbeg[r0], ke = st.row_kbeg[r0 + nr];
  const double2* cv = coef + blockIdx.y * ldc;
  for (int k = kb + tid; k < ke; k += NT) {
    const int r = st.krow[k] - r0;
    float* p = reinterpret_cast<float*>(buf + (r >> 1) * LS + basis[k] % L) + (r & 1);
    const double2 c = cv[k];
    p[0] = (float)(c.x * scale);
    p[2] = (float)(c.y * scale);
  }
  __syncthreads();
  pk2* mine = buf + rp * LS;
  if (u < 8) {   // element u + 8 k1 -> m of k2 = u, in place
    pk2 v[M];
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) v[k1] = mine[u + 8 * k1];
    pk_dft<M, true>(v);
    mine[u] = v[0];
#pragma unroll
    for (int m = 1; m < M; ++m) mine[u + 8 * m] = ptwiddle<true>(v[m], tw[u * M + m]);
  }
  __syncthreads();
  if (u < M) {
    pk2 v[8];
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) v[k2] = mine[8 * u + k2];
    pk_dft<8, true>(v);
    float2* vv = vol + (long)blockIdx.y * L * L * L + u;
    if (2 * rp < nr) {
      float2* d = vv + (long)st.row_idx[r0 + 2 * rp] * L;
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) d[M * n2] = make_float2(v[n2].re.x, v[n2].im.x);
    }
    if (2 * rp + 1 < nr) {
      float2* d = vv + (long)st.row_idx[r0 + 2 * rp + 1] * L;
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) d[M * n2] = make_float2(v[n2].re.y, v[n2].im.y);
    }
  }
}

// Forward along axis 2 of 16 live rows, then out[k] = scale * F[k] (+ kin[k] x[k]) (+ out[k])
// for the rows' basis vectors.
template <int L>
__global__ void __launch_bounds__(Pk<L>::NT) k_sphp_rows_fwd(const float2* __restrict__ vol, const SphereTables st,
                                                             const int* __restrict__ basis, double scale,
                                                             const double* __restrict__ kin,
                                                             const double2* __restrict__ x, long ldx,
                                                             double2* __restrict__ out, long ldo, int accumulate,
                                                             const float2* __restrict__ tw_g) {
  grid_entry();
  constexpr int M = Pk<L>::M, NT = Pk<L>::NT, LS = Pk<L>::LS;
  __shared__ pk2 tw[L];
  __shared__ pk2 buf[RPB * LS];
  const int tid = threadIdx.x, rp = tid % RPB, u = tid / RPB;
  const int r0 = blockIdx.x * (2 * RPB), nr = min(2 * RPB, st.nrows - r0);
  load_tw<L>(tw, tw_g, tid);
  __syncthreads();
  pk2* mine = buf + rp * LS;
  if (u < M) {
    const float2* vv = vol + (long)blockIdx.y * L * L * L + u;
    const float2* p = vv + (long)st.row_idx[r0 + min(2 * rp, nr - 1)] * L;
    const float2* q = vv + (long)st.row_idx[r0 + min(2 * rp + 1, nr - 1)] * L;   // past the last row: any live one
    pk2 v[8];
#pragma unroll
    for (int n2 = 0; n2 < 8; ++n2) {
      const float2 a = p[M * n2], b = q[M * n2];
      v[n2] = {make_float2(a.x, b.x), make_float2(a.y, b.y)};
    }
    pk_dft<8, false>(v);
    mine[8 * u] = v[0];
#pragma unroll
    for (int k2 = 1; k2 < 8; ++k2) mine[8 * u + k2] = ptwiddle<false>(v[k2], tw[k2 * M + u]);
  }
  __syncthreads();
  if (u < 8) {
    pk2 v[M];
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = mine[u + 8 * m];
    pk_dft<M, false>(v);
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) mine[u + 8 * k1] = v[k1];
  }
  __syncthreads();
  const int kb = st.row_kbeg[r0], ke = st.row_kbeg[r0 + nr];
  double2* ov = out + blockIdx.y * ldo;
  const double2* xv = x != nullptr ? x + blockIdx.y * ldx : nullptr;
  for (int k = kb + tid; k < ke; k += NT) {
    const int r = st.krow[k] - r0;
    const float* f = reinterpret_cast<const float*>(buf + (r >> 1) * LS + basis[k] % L) + (r & 1);
    double2 t = make_double2((double)f[0] * scale, (double)f[2] * scale);
    if (kin != nullptr) {
      const double2 c = xv[k];
      t.x += kin[k] * c.x;
      t.y += kin[k] * c.y;
    }
    if (accumulate) {
      const double2 o = ov[k];
      t.x += o.x;
      t.y += o.y;
    }
    ov[k] = t;
  }
}

template <int L>
cudaError_t to_real_t(const double2* coef, long ldc, float2* vol, long nvol, const SphereTables& st, const int* basis,
                      double scale, const float2* tw, cudaStream_t s) {
  if (st.nrows == 0) return cudaMemsetAsync(vol, 0, sizeof(float2) * (size_t)L * L * L * nvol, s);
  constexpr int NT = Pk<L>::NT;
  launch(dim3((unsigned)((st.nrows + 2 * RPB - 1) / (2 * RPB)), (unsigned)nvol), NT, 0, s)(k_sphp_rows_inv<L>, coef, ldc, vol, st, basis, scale, tw);
  launch(dim3(L / (2 * CPB), (unsigned)st.nplanes, (unsigned)nvol), NT, 0, s)(k_sphp_cols<L, true, 1>, vol, vol, nullptr, st, tw);
  launch(dim3(L / (2 * CPB), L, (unsigned)nvol), NT, 0, s)(k_sphp_cols<L, true, 0>, vol, vol, nullptr, st, tw);
  launched(3);
  return cudaGetLastError();
}

template <int L>
cudaError_t to_sphere_t(const float2* vol, const float* mul, float2* work, long nvol, const SphereTables& st,
                        const int* basis, double scale, const double* kin, const double2* x, long ldx, double2* out,
                        long ldo, int accumulate, const float2* tw, cudaStream_t s) {
  if (st.nrows == 0) return cudaSuccess;
  constexpr int NT = Pk<L>::NT;
  launch(dim3(L / (2 * CPB), L, (unsigned)nvol), NT, 0, s)(k_sphp_cols<L, false, 0>, vol, work, mul, st, tw);
  launch(dim3(L / (2 * CPB), (unsigned)st.nplanes, (unsigned)nvol), NT, 0, s)(k_sphp_cols<L, false, 1>, work, work, nullptr, st, tw);
  launch(dim3((unsigned)((st.nrows + 2 * RPB - 1) / (2 * RPB)), (unsigned)nvol), NT, 0, s)(k_sphp_rows_fwd<L>, work, st, basis, scale, kin, x, ldx, out, ldo, accumulate, tw);
  launched(3);
  return cudaGetLastError();
}

// ---- FP64 ---------------------------------------------------------------------------
template <int L, typename C>
cudaError_t to_real_t(const double2* coef, long ldc, C* vol, long nvol, const SphereTables& st, const int* basis,
                      double scale, const C* tw, cudaStream_t s) {
  if (st.nrows == 0) return cudaMemsetAsync(vol, 0, sizeof(C) * (size_t)L * L * L * nvol, s);
  const dim3 gr((unsigned)((st.nrows + SC - 1) / SC), (unsigned)nvol);
  launch(gr, SNT, smem_rows<C, L>(), s)(k_sph_rows_inv<C, L>, coef, ldc, vol, st, basis, scale, tw);
  const dim3 g1((unsigned)(L / SC), (unsigned)st.nplanes, (unsigned)nvol);
  launch(g1, SNT, smem_cols<C, L>(), s)(k_sph_axis1<C, L, true>, vol, st, tw);
  const dim3 g0((unsigned)(L / SC), (unsigned)L, (unsigned)nvol);
  launch(g0, SNT, smem_cols<C, L>(), s)(k_sph_axis0<C, L, true>, vol, vol, nullptr, st, tw);
  launched(3);
  return cudaGetLastError();
}

template <int L, typename C>
cudaError_t to_sphere_t(const C* vol, const typename real_of<C>::type* mul, C* work, long nvol,
                        const SphereTables& st, const int* basis, double scale, const double* kin, const double2* x,
                        long ldx, double2* out, long ldo, int accumulate, const C* tw, cudaStream_t s) {
  if (st.nrows == 0) return cudaSuccess;
  const dim3 g0((unsigned)(L / SC), (unsigned)L, (unsigned)nvol);
  launch(g0, SNT, smem_cols<C, L>(), s)(k_sph_axis0<C, L, false>, vol, work, mul, st, tw);
  const dim3 g1((unsigned)(L / SC), (unsigned)st.nplanes, (unsigned)nvol);
  launch(g1, SNT, smem_cols<C, L>(), s)(k_sph_axis1<C, L, false>, work, st, tw);
  const dim3 gr((unsigned)((st.nrows + SC - 1) / SC), (unsigned)nvol);
  launch(gr, SNT, smem_rows<C, L>(), s)(k_sph_rows_fwd<C, L>, work, st, basis, scale, kin, x, ldx, out, ldo, accumulate,
                                                          tw);
  launched(3);
  return cudaGetLastError();
}

}  // namespace

bool sphere_fast_supported(Grid3 g) {
  return g.n0 == g.n1 && g.n1 == g.n2 && (g.n0 == 32 || g.n0 == 48 || g.n0 == 64 || g.n0 == 96);
}

template <typename C>
static cudaError_t to_real_any(const double2* coef, long ldc, C* vol, long nvol, Grid3 g, const SphereTables& st,
                               const int* basis, double scale, const C* tw_L, cudaStream_t s) {
  if (nvol <= 0) return cudaSuccess;
  if (nvol > 65535) return cudaErrorInvalidValue;
  switch (g.n0) {
    case 32: return to_real_t<32>(coef, ldc, vol, nvol, st, basis, scale, tw_L, s);
    case 48: return to_real_t<48>(coef, ldc, vol, nvol, st, basis, scale, tw_L, s);
    case 64: return to_real_t<64>(coef, ldc, vol, nvol, st, basis, scale, tw_L, s);
    case 96: return to_real_t<96>(coef, ldc, vol, nvol, st, basis, scale, tw_L, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename C>
static cudaError_t from_real_any(const C* vol, const typename real_of<C>::type* mul, C* work, long nvol, Grid3 g,
                                 const SphereTables& st, const int* basis, double scale, const double* kin,
                                 const double2* x, long ldx, double2* out, long ldo, int accumulate, const C* tw_L,
                                 cudaStream_t s) {
  if (nvol <= 0) return cudaSuccess;
  if (nvol > 65535) return cudaErrorInvalidValue;
  switch (g.n0) {
    case 32: return to_sphere_t<32>(vol, mul, work, nvol, st, basis, scale, kin, x, ldx, out, ldo, accumulate, tw_L, s);
    case 48: return to_sphere_t<48>(vol, mul, work, nvol, st, basis, scale, kin, x, ldx, out, ldo, accumulate, tw_L, s);
    case 64: return to_sphere_t<64>(vol, mul, work, nvol, st, basis, scale, kin, x, ldx, out, ldo, accumulate, tw_L, s);
    case 96: return to_sphere_t<96>(vol, mul, work, nvol, st, basis, scale, kin, x, ldx, out, ldo, accumulate, tw_L, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t sphere_to_real(const double2* coef, long ldc, float2* vol, long nvol, Grid3 g, const SphereTables& st,
                           const int* basis, double scale, const float2* tw_L, cudaStream_t s) {
  return to_real_any(coef, ldc, vol, nvol, g, st, basis, scale, tw_L, s);
}
cudaError_t sphere_to_real(const double2* coef, long ldc, double2* vol, long nvol, Grid3 g, const SphereTables& st,
                           const int* basis, double scale, const double2* tw_L, cudaStream_t s) {
  return to_real_any(coef, ldc, vol, nvol, g, st, basis, scale, tw_L, s);
}
cudaError_t sphere_from_real(const float2* vol, const float* mul, float2* work, long nvol, Grid3 g,
                             const SphereTables& st, const int* basis, double scale, const double* kin,
                             const double2* x, long ldx, double2* out, long ldo, int accumulate, const float2* tw_L,
                             cudaStream_t s) {
  return from_real_any(vol, mul, work, nvol, g, st, basis, scale, kin, x, ldx, out, ldo, accumulate, tw_L, s);
}
cudaError_t sphere_from_real(const double2* vol, const double* mul, double2* work, long nvol, Grid3 g,
                             const SphereTables& st, const int* basis, double scale, const double* kin,
                             const double2* x, long ldx, double2* out, long ldo, int accumulate, const double2* tw_L,
                             cudaStream_t s) {
  return from_real_any(vol, mul, work, nvol, g, st, basis, scale, kin, x, ldx, out, ldo, accumulate, tw_L, s);
}

}  // namespace pt
