// Elementwise and reduction kernels of the PT-CN step (Alg. 1, Alg. 3,
// Sec. 3.4) and of the local part of the Hamiltonian (Eq. 2).
// Reductions are two-level (block partials, then one block sums the
// partials in order), so every sum is deterministic.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "kernels.h"

namespace pt {

static inline unsigned nblk(long n, int thr, long cap = 152L * 16) {
  return (unsigned)std::max<long>(1, std::min<long>((n + thr - 1) / thr, cap));
}

// ---- block reduction helper (fixed order) ----------------------------------
template <int NS>
__device__ __forceinline__ void block_sums(double (&v)[NS], double* part) {
  __shared__ double sh[NS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    double x = v[s];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) sh[s][warp] = x;
  }
  __syncthreads();
  if (threadIdx.x < NS) {
    const int nw = blockDim.x >> 5;
    double t = 0.0;
    for (int w = 0; w < nw; ++w) t += sh[threadIdx.x][w];
    part[blockIdx.x * NS + threadIdx.x] = t;
  }
}

// out[q] = sum of part[b ns + q] over the nblocks partials, in an order that depends on
// nblocks alone: one warp per sum, lane l adding partials l, l + 32, ... first.
__global__ void k_finalize(const double* __restrict__ part, int nblocks, int ns, double* __restrict__ out) {
  grid_entry();
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q >= ns) return;
  double t = 0.0;
#pragma unroll 4
  for (int b = lane; b < nblocks; b += 32) t += part[b * ns + q];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if (lane == 0) out[q] = t;
}

static void finalize(const double* part, int nblocks, int ns, double* out, cudaStream_t s) {
  launch(1, 32 * ns, 0, s)(k_finalize, part, nblocks, ns, out); launched();
}

// ---- density ------------------------------------------------------------------
__global__ void k_density(const double2* __restrict__ psi_r, long N, int ne, double* __restrict__ rho) {
  grid_entry();
  for (long r = blockIdx.x * (long)blockDim.x + threadIdx.x; r < N; r += (long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int k = 0; k < ne; ++k) {
      const double2 v = psi_r[(long)k * N + r];
      s += v.x * v.x + v.y * v.y;
    }
    rho[r] = 2.0 * s;
  }
}

cudaError_t density(const double2* psi_r, long N, int ne, double* rho, cudaStream_t s) {
  launch(nblk(N, 256, 152L * 64), 256, 0, s)(k_density, psi_r, N, ne, rho); launched();
  return cudaGetLastError();
}

// FP32 squares summed in FP32 over groups of 16 bands (eight loads in flight
// per thread), the group sums accumulated in FP64: FP64 work drops 16-fold.
__global__ void k_density32(const float2* __restrict__ psi_r, long N, int ne, double* __restrict__ rho) {
  grid_entry();
  constexpr int G = 16;
  for (long r = blockIdx.x * (long)blockDim.x + threadIdx.x; r < N; r += (long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int k0 = 0; k0 < ne; k0 += G) {
      const int kn = min(G, ne - k0);
      float g = 0.f;
#pragma unroll 8
      for (int k = 0; k < kn; ++k) {
        const float2 v = __ldg(psi_r + (long)(k0 + k) * N + r);
        g = fmaf(v.x, v.x, fmaf(v.y, v.y, g));
      }
      s += (double)g;
    }
    rho[r] = 2.0 * s;
  }
}

cudaError_t density32(const float2* psi_r, long N, int ne, double* rho, cudaStream_t s) {
  launch(nblk(N, 256, 152L * 64), 256, 0, s)(k_density32, psi_r, N, ne, rho); launched();
  return cudaGetLastError();
}

// ---- local potential -----------------------------------------------------------
__global__ void k_rho_to_complex(const double* __restrict__ rho, double2* __restrict__ buf, long N) {
  grid_entry();
  for (long r = blockIdx.x * (long)blockDim.x + threadIdx.x; r < N; r += (long)gridDim.x * blockDim.x)
    buf[r] = make_double2(rho[r], 0.0);
}

__global__ void k_vloc(const double2* __restrict__ vh_c, ConvSink sink, long N) {
  grid_entry();
  for (long r = blockIdx.x * (long)blockDim.x + threadIdx.x; r < N; r += (long)gridDim.x * blockDim.x) {
    double v = static_potential(sink, r);
    if (vh_c != nullptr) {
      const double h = vh_c[r].x;
      sink.vh[r] = h;
      v += h;
    }
    sink.vloc[r] = v;
    if (sink.vloc32 != nullptr) sink.vloc32[r] = (float)v;
  }
}

cudaError_t rho_to_complex(const double* rho, double2* buf, long N, cudaStream_t s) {
  launch(nblk(N, 256), 256, 0, s)(k_rho_to_complex, rho, buf, N); launched();
  return cudaGetLastError();
}

cudaError_t assemble_vloc(const double2* vh_c, const ConvSink& sink, long N, cudaStream_t s) {
  launch(nblk(N, 256), 256, 0, s)(k_vloc, vh_c, sink, N); launched();
  return cudaGetLastError();
}

// Gaussian wells summed over atoms and periodic images in real space.
__global__ void k_vion(double* __restrict__ v, int n0, int n1, int n2, double a0, double a1, double a2,
                       const double* __restrict__ atoms, int na, double depth, double sigma, double rcut) {
  grid_entry();
  const long N = (long)n0 * n1 * n2;
  const double inv2s2 = 1.0 / (2.0 * sigma * sigma);
  const int m0 = (int)ceil(rcut / a0), m1 = (int)ceil(rcut / a1), m2 = (int)ceil(rcut / a2);
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < N; t += (long)gridDim.x * blockDim.x) {
    const int i2 = (int)(t % n2);
    const int i1 = (int)((t / n2) % n1);
    const int i0 = (int)(t / ((long)n1 * n2));
    const double x = a0 * i0 / n0, y = a1 * i1 / n1, z = a2 * i2 / n2;
    double s = 0.0;
    for (int a = 0; a < na; ++a) {
      const double ax = atoms[3 * a] * a0, ay = atoms[3 * a + 1] * a1, az = atoms[3 * a + 2] * a2;
      for (int p = -m0; p <= m0; ++p) {
        const double dx = x - ax - p * a0;
        if (fabs(dx) > rcut) continue;
        for (int q = -m1; q <= m1; ++q) {
          const double dy = y - ay - q * a1;
          if (fabs(dy) > rcut) continue;
          for (int w = -m2; w <= m2; ++w) {
            const double dz = z - az - w * a2;
            const double d2 = dx * dx + dy * dy + dz * dz;
            if (d2 <= rcut * rcut) s += exp(-d2 * inv2s2);
          }
        }
      }
    }
    v[t] = -depth * s;
  }
}

cudaError_t ion_potential(double* v, Grid3 g, const double* cell, const double* d_atoms, int na, double depth,
                          double sigma, cudaStream_t s) {
  // exp(-d^2 / (2 sigma^2)) < 1e-20 beyond rcut
  const double rcut = sigma * std::sqrt(2.0 * 46.0);
  launch(nblk(g.N(), 128, 152L * 64), 128, 0, s)(k_vion, v, g.n0, g.n1, g.n2, cell[0], cell[1], cell[2], d_atoms, na,
                                                     depth, sigma, rcut); launched();
  return cudaGetLastError();
}

// ---- PT residual (Alg. 1 and Alg. 3) ---------------------------------------------
// psi_half = psi - i dt/2 R
__global__ void k_half_step(const double2* __restrict__ psi, const double2* __restrict__ R, double hdt,
                            double2* __restrict__ out, long n) {
  grid_entry();
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x) {
    const double2 p = psi[t], r = R[t];
    // -i hdt (rx + i ry) = hdt ry - i hdt rx
    out[t] = make_double2(p.x + hdt * r.y, p.y - hdt * r.x);
  }
}

cudaError_t half_step(const double2* psi, const double2* R, double hdt, double2* out, long n, cudaStream_t s) {
  launch(nblk(n, 256), 256, 0, s)(k_half_step, psi, R, hdt, out, n); launched();
  return cudaGetLastError();
}

// y = x - tau * P * R, P = 1 / (1 + kin) per basis vector (start-state relaxation)
__global__ void k_precond_step(double2* __restrict__ x, const double2* __restrict__ R, const double* __restrict__ kin,
                               int npw, long n, double tau) {
  grid_entry();
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x) {
    const double p = tau / (1.0 + kin[t % npw]);
    const double2 r = R[t];
    double2 v = x[t];
    v.x -= p * r.x;
    v.y -= p * r.y;
    x[t] = v;
  }
}

cudaError_t precond_step(double2* x, const double2* R, const double* kin, int npw, long n, double tau, cudaStream_t s) {
  launch(nblk(n, 256), 256, 0, s)(k_precond_step, x, R, kin, npw, n, tau); launched();
  return cudaGetLastError();
}

// ---- Anderson mixing (Sec. 3.4), per band -------------------------------------------
// r = -(x + i dt/2 T - psi_half) (the fixed-point residual, Alg. 1 and 3) and the history
// entries dX[slot] = x - x_prev, dR[slot] = r - r_prev when there is a previous iterate. r
// overwrites r_prev: one pass over the orbitals instead of three. Bound by memory: 128 bands x
// 13,133 in 46 us (4.1 TB/s); the norm of r, needed once a step, made it 62.
// History entries are stored as H: complex128, or complex64 in mixed precision
// (the differences of successive iterates and residuals, whose rounding to FP32
// only perturbs the least-squares extrapolation, not the fixed point).
template <typename H>
__global__ void __launch_bounds__(256) k_resid_push(const double2* __restrict__ x, const double2* __restrict__ T,
                                                    const double2* __restrict__ ph, double hdt,
                                                    const double2* __restrict__ xp, double2* __restrict__ r,
                                                    H* __restrict__ dx, H* __restrict__ dr, long n, int have_prev) {
  grid_entry();
  using A = decltype(H::x);
#pragma unroll 2
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x) {
    const double2 p = x[t], q = T[t], h = ph[t];
    // i hdt (qx + i qy) = -hdt qy + i hdt qx
    const double2 v = make_double2(-(p.x - hdt * q.y - h.x), -(p.y + hdt * q.x - h.y));
    if (have_prev) {
      const double2 c = xp[t], d = r[t];
      dx[t] = {(A)(p.x - c.x), (A)(p.y - c.y)};
      dr[t] = {(A)(v.x - d.x), (A)(v.y - d.y)};
    }
    r[t] = v;
  }
}

cudaError_t residual_push(const double2* x, const double2* T, const double2* ph, double hdt, const double2* xp,
                          double2* r, void* dx, void* dr, long n, int have_prev, int f32, cudaStream_t s) {
  const unsigned b = nblk(n, 256);
  if (f32)
    launch(b, 256, 0, s)(k_resid_push<float2>, x, T, ph, hdt, xp, r, (float2*)dx, (float2*)dr, n, have_prev);
  else
    launch(b, 256, 0, s)(k_resid_push<double2>, x, T, ph, hdt, xp, r, (double2*)dx, (double2*)dr, n, have_prev);
  launched();
  return cudaGetLastError();
}

// out = sum |r|^2 (once per step, of its last residual); part: 1024 doubles
__global__ void k_norm2(const double2* __restrict__ r, long n, double* __restrict__ part) {
  grid_entry();
  double acc[1] = {0.0};
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x) {
    const double2 v = r[t];
    acc[0] += v.x * v.x + v.y * v.y;
  }
  block_sums<1>(acc, part);
}

cudaError_t norm2(const double2* r, long n, double* part, double* out, cudaStream_t s) {
  const unsigned b = nblk(n, 256, 1024);
  launch(b, 256, 0, s)(k_norm2, r, n, part); launched();
  finalize(part, (int)b, 1, out, s);
  return cudaGetLastError();
}

// Partial sums over one of gridDim.x chunks of the basis of <dR_q, dR_new> and <dR_q, r> for
// band blockIdx.y and every slot q: a thread reads dR_new and r of its coefficients once and
// carries four sums per slot in registers (KM >= k slots), so each entry of the history is
// read once, coalesced, with k loads in flight. One warp per slot re-read dR_new and r from L1
// for each slot: 92 us on average over a step at 128 bands x 13,133, 59 so.
// Complex64 history (mixed precision): the products are formed in FP32 and
// summed in FP32 over each thread's share of the basis (at most npw / 256 terms);
// the threads' sums are reduced in FP64. FP64 otherwise. The Gram matrix and
// right-hand side feed the FP64 solve either way. The reduction halves the values a lane
// carries with every exchange, 78 FP64 additions a lane where a tree per value takes 400.
constexpr int kDotThreads = 128, kDotChunksMax = 8;

// Sums x over the warp's lanes, HAVE values: lanes whose bit O is set keep the upper half, the
// others the lower; the lane ends with the n values from `base` on in x[0..n).
template <int HAVE, int O>
__device__ __forceinline__ void fold_lanes(double* x, int lane, int& base, int& n) {
  constexpr int HALF = (HAVE + 1) / 2;
  const bool up = (lane & O) != 0;
#pragma unroll
  for (int i = 0; i < HALF; ++i) {
    const double hi = i + HALF < HAVE ? x[i + HALF < HAVE ? i + HALF : 0] : 0.0;
    const double send = up ? x[i] : hi, keep = up ? hi : x[i];
    x[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
  }
  if (up) {
    base += HALF;
    n -= HALF;
  } else {
    n = min(n, HALF);
  }
  if constexpr (O > 1) fold_lanes<HALF, O / 2>(x, lane, base, n);
}

template <typename H, int KM>
__global__ void __launch_bounds__(kDotThreads) k_anderson_dots(const H* __restrict__ dR, long slot_stride, SlotList sl,
                                                               int newslot, const double2* __restrict__ r, int npw,
                                                               double* __restrict__ part) {
  grid_entry();
  using A = decltype(H::x);
  constexpr int NV = 4 * KM;
  __shared__ double sh[kDotThreads / 32][NV];
  const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, k = sl.k;
  const int len = (npw + gridDim.x - 1) / gridDim.x;
  const int g0 = blockIdx.x * len, g1 = min(npw, g0 + len);
  const long boff = (long)b * npw;
  const H* dn = dR + (long)newslot * slot_stride + boff;
  const double2* rb = r + boff;
  A acc[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) acc[c] = 0;
  for (int g = g0 + tid; g < g1; g += kDotThreads) {
    const H v = dn[g];
    const double2 w = rb[g];
    H u[KM];
#pragma unroll
    for (int q = 0; q < KM; ++q) {
      u[q] = H{};
      if (q < k) u[q] = dR[(long)sl.s[q] * slot_stride + boff + g];
    }
    const A wx = (A)w.x, wy = (A)w.y;
#pragma unroll
    for (int q = 0; q < KM; ++q) {
      acc[4 * q + 0] += u[q].x * v.x + u[q].y * v.y;
      acc[4 * q + 1] += u[q].x * v.y - u[q].y * v.x;
      acc[4 * q + 2] += u[q].x * wx + u[q].y * wy;
      acc[4 * q + 3] += u[q].x * wy - u[q].y * wx;
    }
  }
  double x[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) x[c] = (double)acc[c];
  int base = 0, n = NV;
  fold_lanes<NV, 16>(x, lane, base, n);
#pragma unroll
  for (int i = 0; i < (NV + 31) / 32; ++i)
    if (i < n) sh[tid >> 5][base + i] = x[i];
  __syncthreads();
  if (tid < NV && tid < 4 * k) {
    double t = sh[0][tid];
#pragma unroll
    for (int w = 1; w < kDotThreads / 32; ++w) t += sh[w][tid];
    part[(((long)b * k + tid / 4) * gridDim.x + blockIdx.x) * 4 + tid % 4] = t;
  }
}

// Gathers the sums into gram[b][slot_q][new] (and its conjugate at [new][slot_q]) and the
// right-hand side <dR_q, r> (slots in order, oldest first), then solves
// (G + 1e-14 tr(G) I) gamma = rhs per band by L D L^H; gamma = 0 when the trace is zero
// or a pivot is not positive. One block per band, the matrix in shared memory with the
// right-hand side as its last row (so the forward substitution is part of the
// factorisation). Latency bounds it: k dependent pivots. One warp keeps the diagonal, a lane per
// entry, and inverts the next pivot while the others update the entries below the
// diagonal; columns stay unscaled, so a column costs one barrier (a step's average, up to 20
// entries: 20.0 us with a scaled column per pivot, 17.5 so).
constexpr int kSolveUpdate = 128, kSolveThreads = kSolveUpdate + 32;

__global__ void __launch_bounds__(kSolveThreads) k_anderson_solve(const double4_16a* __restrict__ part, SlotList sl,
                                                                  int newslot, int chunks, int mdim,
                                                                  double2* __restrict__ gram,
                                                                  double2* __restrict__ gamma) {
  grid_entry();
  __shared__ double2 V[kSlotMax + 1][kSlotMax + 1];   // below the diagonal: column j of L times the pivot D_j
  __shared__ double inv[kSlotMax];                    // 1 / D_j, or 0 when it is not positive
  // entries (i, p), p < i <= k, by falling p: those a column j still changes (p > j) come first
  __shared__ unsigned char ent[kSlotMax * (kSlotMax + 1) / 2][2];
  const int b = blockIdx.x, tid = threadIdx.x, k = sl.k;
  double2* G = gram + (long)b * mdim * mdim;
  // A[i][j] = G[s_i][s_j]  (G[s][t] = <dR_s, dR_t>); older entries
#pragma unroll 4
  for (int t = tid; t < k * k; t += kSolveThreads) {
    const int i = t / k, j = t % k;
    if (j <= i && sl.s[i] != newslot && sl.s[j] != newslot) V[i][j] = G[(long)sl.s[i] * mdim + sl.s[j]];
  }
  if (tid >= kSolveUpdate && tid - kSolveUpdate < k) {
    const int c = tid - kSolveUpdate, p = k - 1 - c;   // rows p + 1 .. k after the sum of 1, 2, .. c earlier entries
    int at = c * (c + 1) / 2;
    for (int i = p + 1; i <= k; ++i, ++at) {
      ent[at][0] = (unsigned char)i;
      ent[at][1] = (unsigned char)p;
    }
  }
  if (tid < k) {
    const int q = tid, mine = sl.s[q];
    const double4_16a* p = part + ((long)b * k + q) * chunks;
    double4_16a t = p[0];
#pragma unroll 4
    for (int c = 1; c < chunks; ++c) {
      t.x += p[c].x;
      t.y += p[c].y;
      t.z += p[c].z;
      t.w += p[c].w;
    }
    int at = 0;   // the new slot's place in the list
    while (sl.s[at] != newslot) ++at;
    const double2 fwd = make_double2(t.x, q == at ? 0.0 : t.y), rev = make_double2(t.x, q == at ? 0.0 : -t.y);
    G[(long)mine * mdim + newslot] = fwd;
    G[(long)newslot * mdim + mine] = rev;
    if (q >= at) V[q][at] = fwd;
    if (q <= at) V[at][q] = rev;
    V[k][q] = make_double2(t.z, -t.w);   // conj(rhs): row k becomes w^H, L w = rhs
  }
  __syncthreads();
  const int lane = tid - kSolveUpdate;
  double diag = 0.0;
  auto pivot = [&](int j) {   // by the diagonal's warp
    const double d = __shfl_sync(0xffffffffu, diag, j);
    const double r = d > 0.0 ? 1.0 / d : 0.0;
    if (lane == 0) inv[j] = r;
  };
  if (lane >= 0) {
    diag = lane < k ? V[lane][lane].x : 0.0;
    double tr = diag;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    diag += 1e-14 * tr;
    if (!(tr > 0.0)) diag = 0.0;
    pivot(0);
  }
  __syncthreads();
  bool ok = true;
  for (int j = 0; j < k; ++j) {
    const double r = inv[j];
    if (!(r > 0.0)) { ok = false; break; }
    if (j + 1 == k) break;
    if (lane >= 0) {
      if (lane > j && lane < k) {
        const double2 u = V[lane][j];
        diag -= r * (u.x * u.x + u.y * u.y);
      }
      pivot(j + 1);
    } else {
      const int m = k - j;   // A[i][p] -= V[i][j] conj(V[p][j]) / D_j for j < p < i <= k
      for (int t = tid; t < m * (m - 1) / 2; t += kSolveUpdate) {
        const int i = ent[t][0], p = ent[t][1];
        const double2 u = V[i][j], w = V[p][j];
        V[i][p].x -= r * (u.x * w.x + u.y * w.y);
        V[i][p].y -= r * (u.y * w.x - u.x * w.y);
      }
    }
    __syncthreads();
  }
  if (tid >= 32) return;
  if (!ok) {
    if (tid < k) gamma[(long)b * mdim + tid] = make_double2(0.0, 0.0);
    return;
  }
  double2 y = tid < k ? make_double2(V[k][tid].x, -V[k][tid].y) : make_double2(0.0, 0.0);
  const double di = tid < k ? inv[tid] : 0.0;
  for (int i = k - 1; i >= 0; --i) {   // D L^H gamma = w
    if (tid == i) { y.x *= di; y.y *= di; }
    const double yx = __shfl_sync(0xffffffffu, y.x, i), yy = __shfl_sync(0xffffffffu, y.y, i);
    if (tid < i) {
      const double2 l = V[i][tid];
      y.x -= l.x * yx + l.y * yy;
      y.y -= l.x * yy - l.y * yx;
    }
  }
  if (tid < k) gamma[(long)b * mdim + tid] = y;
}

template <typename H>
static void dots_any(const H* dR, long slot_stride, const SlotList& sl, int newslot, const double2* r, int npw, int ne,
                     int chunks, double* part, cudaStream_t s) {
  launch to(dim3((unsigned)chunks, (unsigned)ne), kDotThreads, 0, s);
  switch ((sl.k + 3) / 4) {
    case 1: to(k_anderson_dots<H, 4>, dR, slot_stride, sl, newslot, r, npw, part); break;
    case 2: to(k_anderson_dots<H, 8>, dR, slot_stride, sl, newslot, r, npw, part); break;
    case 3: to(k_anderson_dots<H, 12>, dR, slot_stride, sl, newslot, r, npw, part); break;
    case 4: to(k_anderson_dots<H, 16>, dR, slot_stride, sl, newslot, r, npw, part); break;
    default: to(k_anderson_dots<H, kSlotMax>, dR, slot_stride, sl, newslot, r, npw, part); break;
  }
}

cudaError_t anderson_gamma(const void* dR, long slot_stride, const SlotList& sl, int newslot, const double2* r,
                           int npw, int ne, int mdim, double2* gram, double2* gamma, void* part, int f32,
                           cudaStream_t s) {
  if (sl.k < 1 || sl.k > kSlotMax) return cudaErrorInvalidValue;
  if (ne > 65535) return cudaErrorInvalidValue;
  // two chunks of 128 threads each (256 threads' sums per band) once the bands fill the chip
  const int chunks = std::max(2, std::min(kDotChunksMax, 2 * sm_count() / ne));
  if (f32) dots_any<float2>((const float2*)dR, slot_stride, sl, newslot, r, npw, ne, chunks, (double*)part, s);
  else dots_any<double2>((const double2*)dR, slot_stride, sl, newslot, r, npw, ne, chunks, (double*)part, s);
  launch(ne, kSolveThreads, 0, s)(k_anderson_solve, (const double4_16a*)part, sl, newslot, chunks, mdim, gram, gamma);
  launched(2);
  return cudaGetLastError();
}

// out = x + beta r - sum_q gamma_q (dX_q + beta dR_q). One block row per band (no
// division per element). With complex64 history the correction sum is formed
// in FP32 and added to the FP64 iterate once.
template <typename H>
__global__ void __launch_bounds__(256) k_anderson_update(const double2* __restrict__ x, const double2* __restrict__ r,
                                                         const H* __restrict__ dX, const H* __restrict__ dR,
                                                         long slot_stride, SlotList sl,
                                                         const double2* __restrict__ gamma, int mdim, int npw,
                                                         double beta, double2* __restrict__ out) {
  grid_entry();
  using A = decltype(H::x);
  const int k = sl.k;
  const int b = blockIdx.y;
  const long boff = (long)b * npw;
  __shared__ A gs[2 * kSlotMax];
  // the slots' places: looked up in the parameters, each held up its loads (128 bands x 13,133, 16 to
  // 20 entries: 134 us a launch, 85 so)
  __shared__ long at[kSlotMax];
  if (threadIdx.x < k) {
    const double2 g = gamma[(long)b * mdim + threadIdx.x];
    gs[2 * threadIdx.x] = (A)g.x;
    gs[2 * threadIdx.x + 1] = (A)g.y;
    at[threadIdx.x] = (long)sl.s[threadIdx.x] * slot_stride + boff;
  }
  __syncthreads();
  const A bt = (A)beta;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < npw; i += gridDim.x * blockDim.x) {
    const long t = boff + i;
    A cx = 0, cy = 0;
#pragma unroll 4
    for (int q = 0; q < k; ++q) {
      const long sq = at[q] + i;
      const H a = dX[sq], c = dR[sq];
      const A ux = a.x + bt * c.x, uy = a.y + bt * c.y;
      const A gx = gs[2 * q], gy = gs[2 * q + 1];
      cx += ux * gx - uy * gy;
      cy += ux * gy + uy * gx;
    }
    const double2 v = x[t], rr = r[t];
    out[t] = make_double2(v.x + (beta * rr.x - (double)cx), v.y + (beta * rr.y - (double)cy));
  }
}

cudaError_t anderson_update(const double2* x, const double2* r, const void* dX, const void* dR, long slot_stride,
                            const SlotList& sl, const double2* gamma, int mdim, int npw, long n, double beta, int f32,
                            double2* out, cudaStream_t s) {
  if (sl.k > kSlotMax) return cudaErrorInvalidValue;
  const int ne = npw > 0 ? (int)(n / npw) : 0;
  if (ne == 0) return cudaSuccess;
  const dim3 grid((unsigned)std::min(32, (npw + 255) / 256), (unsigned)ne);
  if (f32)
    launch(grid, 256, 0, s)(k_anderson_update<float2>, x, r, (const float2*)dX, (const float2*)dR, slot_stride, sl, gamma,
                                                   mdim, npw, beta, out);
  else
    launch(grid, 256, 0, s)(k_anderson_update<double2>, x, r, (const double2*)dX, (const double2*)dR, slot_stride, sl,
                                                    gamma, mdim, npw, beta, out);
  launched();
  return cudaGetLastError();
}

// kin[k] = |gk[k] + a|^2 / 2 with gk the basis vectors G + kick (three arrays of npw)
__global__ void k_kinetic_shifted(const double* __restrict__ gk3, int npw, double ax, double ay, double az,
                                  double* __restrict__ kin) {
  grid_entry();
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < npw; k += gridDim.x * blockDim.x) {
    const double x = gk3[k] + ax, y = gk3[npw + k] + ay, z = gk3[2 * (long)npw + k] + az;
    kin[k] = 0.5 * (x * x + y * y + z * z);
  }
}

cudaError_t kinetic_shifted(const double* gk3, int npw, double ax, double ay, double az, double* kin, cudaStream_t s) {
  launch(nblk(npw, 256), 256, 0, s)(k_kinetic_shifted, gk3, npw, ax, ay, az, kin); launched();
  return cudaGetLastError();
}

// ---- density change, energy, dipole ---------------------------------------------------
__global__ void k_drho(const double* __restrict__ a, const double* __restrict__ b, long N, double* __restrict__ part) {
  grid_entry();
  double acc[1] = {0.0};
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < N; t += (long)gridDim.x * blockDim.x)
    acc[0] += fabs(a[t] - b[t]);
  block_sums<1>(acc, part);
}

cudaError_t rho_change(const double* a, const double* b, long N, double* part, double* out, cudaStream_t s) {
  const unsigned nb = nblk(N, 256, 1024);
  launch(nb, 256, 0, s)(k_drho, a, b, N, part); launched();
  finalize(part, nb, 1, out, s);
  return cudaGetLastError();
}

// grid sums: [0] vion*rho, [1] vh*rho, [2] rho^{4/3}, [3..5] r*rho
__global__ void k_grid_sums(const double* __restrict__ rho, const double* __restrict__ vion,
                            const double* __restrict__ vh, int use_h, int n0, int n1, int n2, double a0, double a1,
                            double a2, double* __restrict__ part) {
  grid_entry();
  const long N = (long)n0 * n1 * n2;
  double acc[6] = {0, 0, 0, 0, 0, 0};
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < N; t += (long)gridDim.x * blockDim.x) {
    const int i2 = (int)(t % n2);
    const int i1 = (int)((t / n2) % n1);
    const int i0 = (int)(t / ((long)n1 * n2));
    const double p = rho[t];
    acc[0] += vion[t] * p;
    if (use_h) acc[1] += vh[t] * p;
    acc[2] += cbrt_pos(p) * p;
    acc[3] += (a0 * i0 / n0) * p;
    acc[4] += (a1 * i1 / n1) * p;
    acc[5] += (a2 * i2 / n2) * p;
  }
  block_sums<6>(acc, part);
}

// [0] sum kin |c|^2
__global__ void k_kin_sum(const double2* __restrict__ c, const double* __restrict__ kin, int npw, long n,
                          double* __restrict__ part) {
  grid_entry();
  double acc[1] = {0.0};
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x) {
    const double2 v = c[t];
    acc[0] += kin[t % npw] * (v.x * v.x + v.y * v.y);
  }
  block_sums<1>(acc, part);
}

__global__ void k_trace_real(const double2* __restrict__ M, int n, double* __restrict__ out) {
  grid_entry();
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < n; ++i) t += M[i + (long)i * n].x;
    *out = t;
  }
}

cudaError_t energy_sums(const double* rho, const double* vion, const double* vh, int use_h, Grid3 g, const double* cell,
                        const double2* c, const double* kin, int npw, int ne, const double2* negM, double* part,
                        double* out8, cudaStream_t s) {
  const unsigned nb = nblk(g.N(), 256, 1024);
  launch(nb, 256, 0, s)(k_grid_sums, rho, vion, vh, use_h, g.n0, g.n1, g.n2, cell[0], cell[1], cell[2], part); launched();
  finalize(part, nb, 6, out8, s);
  const long n = (long)npw * ne;
  const unsigned nb2 = nblk(n, 256, 1024);
  launch(nb2, 256, 0, s)(k_kin_sum, c, kin, npw, n, part + 6 * 1024); launched();
  finalize(part + 6 * 1024, nb2, 1, out8 + 6, s);
  if (negM != nullptr) { launch(1, 32, 0, s)(k_trace_real, negM, ne, out8 + 7); launched(); }
  return cudaGetLastError();
}

__global__ void k_hartree_factor(double* __restrict__ f, int n0, int n1, int n2, double a0, double a1, double a2) {
  grid_entry();
  const long N = (long)n0 * n1 * n2;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < N; t += (long)gridDim.x * blockDim.x) {
    const int i2 = (int)(t % n2);
    const int i1 = (int)((t / n2) % n1);
    const int i0 = (int)(t / ((long)n1 * n2));
    const int m0 = i0 < (n0 + 1) / 2 ? i0 : i0 - n0;
    const int m1 = i1 < (n1 + 1) / 2 ? i1 : i1 - n1;
    const int m2 = i2 < (n2 + 1) / 2 ? i2 : i2 - n2;
    const double g0 = 2.0 * M_PI * m0 / a0, g1 = 2.0 * M_PI * m1 / a1, g2 = 2.0 * M_PI * m2 / a2;
    const double gg = g0 * g0 + g1 * g1 + g2 * g2;
    f[t] = gg > 0.0 ? 4.0 * M_PI / (gg * (double)N) : 0.0;
  }
}

cudaError_t hartree_factor(double* f, Grid3 g, const double* cell, cudaStream_t s) {
  launch(nblk(g.N(), 256), 256, 0, s)(k_hartree_factor, f, g.n0, g.n1, g.n2, cell[0], cell[1], cell[2]); launched();
  return cudaGetLastError();
}

}  // namespace pt

namespace pt {

__global__ void k_axpy(double2 a, const double2* __restrict__ x, double2* __restrict__ y, long n) {
  grid_entry();
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n; t += (long)gridDim.x * blockDim.x) {
    const double2 v = x[t];
    double2 w = y[t];
    w.x += a.x * v.x - a.y * v.y;
    w.y += a.x * v.y + a.y * v.x;
    y[t] = w;
  }
}

cudaError_t axpy(double2 a, const double2* x, double2* y, long n, cudaStream_t s) {
  launch(nblk(n, 256), 256, 0, s)(k_axpy, a, x, y, n); launched();
  return cudaGetLastError();
}

}  // namespace pt

namespace pt {

__global__ void k_diff_to_complex(const double* __restrict__ a, const double* __restrict__ b, double2* __restrict__ buf,
                                  long N) {
  grid_entry();
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < N; t += (long)gridDim.x * blockDim.x)
    buf[t] = make_double2(a[t] - b[t], 0.0);
}

__global__ void k_add_real(const double2* __restrict__ buf, double* __restrict__ a, long N) {
  grid_entry();
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < N; t += (long)gridDim.x * blockDim.x)
    a[t] += buf[t].x;
}

cudaError_t diff_to_complex(const double* a, const double* b, double2* buf, long N, cudaStream_t s) {
  launch(nblk(N, 256), 256, 0, s)(k_diff_to_complex, a, b, buf, N); launched();
  return cudaGetLastError();
}

cudaError_t add_real(const double2* buf, double* a, long N, cudaStream_t s) {
  launch(nblk(N, 256), 256, 0, s)(k_add_real, buf, a, N); launched();
  return cudaGetLastError();
}

// b |G|^2 / (|G|^2 + q0^2) / N  (Kerker weight with the inverse-FFT normalisation)
__global__ void k_kerker_factor(double* __restrict__ f, int n0, int n1, int n2, double a0, double a1, double a2,
                                double b, double q2) {
  grid_entry();
  const long N = (long)n0 * n1 * n2;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < N; t += (long)gridDim.x * blockDim.x) {
    const int i2 = (int)(t % n2);
    const int i1 = (int)((t / n2) % n1);
    const int i0 = (int)(t / ((long)n1 * n2));
    const int m0 = i0 < (n0 + 1) / 2 ? i0 : i0 - n0;
    const int m1 = i1 < (n1 + 1) / 2 ? i1 : i1 - n1;
    const int m2 = i2 < (n2 + 1) / 2 ? i2 : i2 - n2;
    const double g0 = 2.0 * M_PI * m0 / a0, g1 = 2.0 * M_PI * m1 / a1, g2 = 2.0 * M_PI * m2 / a2;
    const double gg = g0 * g0 + g1 * g1 + g2 * g2;
    f[t] = b * gg / (gg + q2) / (double)N;
  }
}

cudaError_t kerker_factor(double* f, Grid3 g, const double* cell, double b, double q0, cudaStream_t s) {
  launch(nblk(g.N(), 256), 256, 0, s)(k_kerker_factor, f, g.n0, g.n1, g.n2, cell[0], cell[1], cell[2], b, q0 * q0);
  launched();
  return cudaGetLastError();
}

}  // namespace pt
