// Fock exchange by orbital pairs (Eq. 3; the pair loop of Alg. 2).
//
// For every pair (i, j) the pair density rho_ij = conj(psi_i) psi_j goes
// through a forward 3D FFT, is multiplied by the screened kernel
// Khat(G) = 4 pi (1 - exp(-G^2 / (4 w^2))) / G^2 (scaled by -alpha / N), goes
// back through an inverse FFT and is multiplied by psi_i and accumulated
// into W_j. Because Khat is real and even, v_ji = conj(v_ij): one solve per
// unordered pair also feeds W_i += psi_j conj(v_ij) ("sym" mode).
//
// Pairs are grouped into tiles (up to kTileMax orbitals on each side) and a
// launch holds tiles whose output orbitals are all distinct, so every W
// element has a single writer per launch (deterministic, no atomics). One
// launch is three kernels over an intermediate X in global memory:
//   F1  rows: product of two orbitals' rows, FFT along axis 2; the block owns
//       `rr` rows of all pairs of its tile and stores X[pair][i2][i0][i1]
//       (axis 1 fastest, so F2 reads a contiguous slab);
//   F2  slab (pair, i2): FFT along axis 1 and axis 0, multiply by Khat,
//       inverse along axis 0 and axis 1, all in shared memory;
//   F3  rows: inverse FFT along axis 2 of all pairs of the tile, then each
//       output orbital sums its pair contributions in a fixed order and
//       updates its W row once.
// X traffic is four passes of the pair volume (write, read+write, read).
//
// These kernels serve every grid in FP64 and the non-cubic ones in FP32. FP64 arithmetic
// bounds them (an SM does two FP64 multiply-adds a clock), so they save operations: a
// line takes at most two steps of large codelets (fft_pk.cuh) with the fewest twiddles,
// and the slabs (axis 2) and columns (axis 1) of frequencies that products of the basis
// cannot reach are neither transformed nor stored. 27 orbitals on 24 x 48 x 32 points, an
// exchange in FP64: 3.63 ms with lines of three small codelets, 3.46 pruned with the large
// ones, 3.29 with coprime factors; the FP64 pipe is then busy 3/4 of the time.
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "fft_pk.cuh"
#include "internal.h"

namespace pt {

template <typename T>
static const cplx<T>* twp(const DevTwiddles& tw, int L) {
  return reinterpret_cast<const cplx<T>*>(tw.base<T>()) + twiddle_offset(L);
}

// ---------------------------------------------------------------------------
// Lines in shared memory, L = R M, take two in-place steps: A, R-point DFTs, and B, M-point
// DFTs. For M = 3 (24 = 8 x 3, 48 = 16 x 3, 12 = 4 x 3: coprime factors) element 3 q + R m (mod
// L) has index q in step A and m in step B, without twiddles; otherwise element m + M q has,
// and step A applies W_L^(m q). place_of(k) is where frequency k ends: (R + 3) k mod L, or
// M (k mod R) + k / R. The inverse starts from there.
//
// Few lines (FEW, FP64): a codelet per line of 8 to 16 points leaves most of a warp idle when
// there are fewer than 32 lines, and the FP64 pipe, which bounds the kernels, is as long busy with
// a part of a warp as with all of it. Such lines take R = 4 (F2 of slabs of two short axes, a
// launch of 32 pairs on 16 x 16 x 64 points: 133 us with 16-point codelets, 55 so).
template <typename T> struct value_of;
template <> struct value_of<float> { using type = cf; };
template <> struct value_of<double> { using type = cd; };

template <bool FEW> __host__ __device__ constexpr int first_radix(int L) {
  return FEW ? 4 : L == 12 ? 12 : L == 16 || L == 48 ? 16 : 8;
}
template <bool FEW> __host__ __device__ constexpr bool coprime(int L) { return L == 3 * first_radix<FEW>(L); }
template <bool FEW = false> __device__ __forceinline__ int place_of(int k, int L) {
  const int R = first_radix<FEW>(L), M = L / R;
  return coprime<FEW>(L) ? (R + 3) * k % L : M * (k % R) + k / R;
}
// (the inverses of 7 mod 12, 11 mod 24 and 19 mod 48)
template <bool FEW = false> __device__ __forceinline__ int freq_at(int place, int L) {
  const int R = first_radix<FEW>(L), M = L / R;
  return coprime<FEW>(L) ? (L == 12 ? 7 : L == 24 ? 11 : 43) * place % L : place / M + R * (place % M);
}

// Transforms `nlines` lines: element e of line i at buf[lines(i) + e es].
template <int L, bool INV, bool FEW, typename V, class Lines>
__device__ __forceinline__ void line_pass(V* buf, int nlines, int es, const V* tw, int tid, int nthr, Lines lines) {
  constexpr int R = first_radix<FEW>(L), M = L / R;
  constexpr bool twiddled = M > 1 && !coprime<FEW>(L);
  // element q of the DFT number m of step A (b = false), element m of DFT q of step B
  auto at = [](int q, int m) {
    if (!coprime<FEW>(L)) return m + M * q;
    const int e = 3 * q + R * m;
    return e >= L ? e - L : e;
  };
  auto step_a = [&]() {
    for (int b = tid; b < nlines * M; b += nthr) {
      const int m = b / nlines;
      V* p = buf + lines(b - m * nlines);
      V v[R];
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = p[at(q, m) * es];
      if (INV && twiddled) {
#pragma unroll
        for (int q = 1; q < R; ++q) v[q] = ptwiddle<true>(v[q], tw[q * m]);
      }
      pk_dft<R, INV>(v);
      if (!INV && twiddled) {
#pragma unroll
        for (int q = 1; q < R; ++q) v[q] = ptwiddle<false>(v[q], tw[q * m]);
      }
#pragma unroll
      for (int q = 0; q < R; ++q) p[at(q, m) * es] = v[q];
    }
    __syncthreads();
  };
  auto step_b = [&]() {
    for (int b = tid; b < nlines * R; b += nthr) {
      const int q = b / nlines;
      V* p = buf + lines(b - q * nlines);
      V v[M];
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] = p[at(q, m) * es];
      pk_dft<M, INV>(v);
#pragma unroll
      for (int m = 0; m < M; ++m) p[at(q, m) * es] = v[m];
    }
    __syncthreads();
  };
  if constexpr (M == 1) {
    step_a();
  } else if constexpr (!INV) {
    step_a();
    step_b();
  } else {
    step_b();
    step_a();
  }
}

template <bool INV, bool FEW = false, typename V, class Lines>
__device__ __forceinline__ void line_pass_any(V* buf, int L, int nlines, int es, const V* tw, int tid, int nthr,
                                              Lines lines) {
  switch (L) {
    case 8: line_pass<8, INV, FEW>(buf, nlines, es, tw, tid, nthr, lines); return;
    case 12: line_pass<12, INV, FEW>(buf, nlines, es, tw, tid, nthr, lines); return;
    case 16: line_pass<16, INV, FEW>(buf, nlines, es, tw, tid, nthr, lines); return;
    default: break;
  }
  if constexpr (!FEW) {
    switch (L) {
      case 24: line_pass<24, INV, FEW>(buf, nlines, es, tw, tid, nthr, lines); break;
      case 32: line_pass<32, INV, FEW>(buf, nlines, es, tw, tid, nthr, lines); break;
      case 48: line_pass<48, INV, FEW>(buf, nlines, es, tw, tid, nthr, lines); break;
      case 64: line_pass<64, INV, FEW>(buf, nlines, es, tw, tid, nthr, lines); break;
      case 96: line_pass<96, INV, FEW>(buf, nlines, es, tw, tid, nthr, lines); break;
      default: break;
    }
  }
}

// whether F1 and F3 take the transforms of few lines for a tile's lines
template <typename T> __device__ __forceinline__ bool few_lines(int L, int nlines) {
  return sizeof(T) == 8 && L <= 16 && nlines < 32;
}

// where the frequencies of a line are, by the transforms of many and (FP64) of few lines: a
// table, as the divisions for a length known at run time took F1 and F3 a tenth of their time
// (FP32, 33 orbitals on 32 x 32 x 64 points: 1640 us an exchange without, 1495 so)
template <typename T, int L>
__device__ __forceinline__ void load_places_of(unsigned char (&places)[2][kMaxLength], int tid, int nthr) {
  for (int t = tid; t < L; t += nthr) {
    places[0][t] = (unsigned char)place_of(t, L);
    if (sizeof(T) == 8 && L <= 16) places[1][t] = (unsigned char)place_of<true>(t, L);
  }
}
template <typename T>
__device__ __forceinline__ void load_places(unsigned char (&places)[2][kMaxLength], int L, int tid, int nthr) {
  switch (L) {
    case 8: load_places_of<T, 8>(places, tid, nthr); break;
    case 12: load_places_of<T, 12>(places, tid, nthr); break;
    case 16: load_places_of<T, 16>(places, tid, nthr); break;
    case 24: load_places_of<T, 24>(places, tid, nthr); break;
    case 32: load_places_of<T, 32>(places, tid, nthr); break;
    case 48: load_places_of<T, 48>(places, tid, nthr); break;
    case 64: load_places_of<T, 64>(places, tid, nthr); break;
    case 96: load_places_of<T, 96>(places, tid, nthr); break;
    default: break;
  }
}

// twiddles c - i s as (c, s)
template <typename V, typename C> __device__ __forceinline__ void load_tw(V* tw, const C* tw_g, int L, int tid, int nthr) {
  for (int t = tid; t < L; t += nthr) tw[t] = V{tw_g[t].x, -tw_g[t].y};
}

// Largest frequency along axis 1 of the pair products in the axis-2 slab of frequency +-g2,
// and the axis-2 reach (n1, n2 or more: every one is reached).
struct PairReach {
  int g2;
  unsigned char g1[kMaxLength / 2 + 1];
};

__device__ __forceinline__ bool live(int k, int n, int reach) { return k <= reach || k >= n - reach; }

// Blocks of 256 threads that share an SM's registers. FP64 needs those of two. FP32 is bound by
// latency and memory, and four of 64 registers fit without a spill (16 orbitals on 96 x 64 x 64
// points: 2026 us an exchange with the 72 to 80 registers the compiler would take, 1878 so).
template <typename T> struct PairBlocks { static constexpr int value = sizeof(T) == 8 ? 2 : 4; };

template <typename T>
__global__ void __launch_bounds__(256, PairBlocks<T>::value) k_fock_f1(const PairTile* __restrict__ tiles, int tile0,
                                                    cplx<T>* __restrict__ Xc, int n0, int n1, int n2, int rr,
                                                    int reach2, const cplx<T>* __restrict__ tw_g) {
  grid_entry();
  using V = typename value_of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ PairTile tl;
  __shared__ unsigned char places[2][kMaxLength];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int rowlen = rr * n2, ls = n2 + 1;
  V* X = reinterpret_cast<V*>(Xc);
  V* tw = reinterpret_cast<V*>(smem_raw);
  V* orb = tw + n2;
  V* work = orb + 2 * kTileMax * rowlen;
  for (int t = tid; t < (int)(sizeof(PairTile) / 4); t += nthr)
    reinterpret_cast<unsigned*>(&tl)[t] = reinterpret_cast<const unsigned*>(tiles + tile0 + blockIdx.y)[t];
  load_tw(tw, tw_g, n2, tid, nthr);
  load_places<T>(places, n2, tid, nthr);
  __syncthreads();
  const int nb1 = n1 / rr;
  const int i0 = blockIdx.x / nb1;
  const int i1s = (blockIdx.x - i0 * nb1) * rr;
  const long roff = ((long)i0 * n1 + i1s) * n2;
  const bool few = few_lines<T>(n2, tl.n_pairs * rr);
  for (int o = 0; o < tl.n_orb; ++o) {
    const V* src = (const V*)tl.in[o] + roff;
    for (int e = tid; e < rowlen; e += nthr) orb[o * rowlen + e] = src[e];
  }
  __syncthreads();
  const int np = tl.n_pairs;
  for (int idx = tid; idx < np * rowlen; idx += nthr) {
    const int l = idx / n2, p = l / rr, e = idx - p * rowlen;
    const V a = orb[tl.pi[p] * rowlen + e], b = orb[tl.pj[p] * rowlen + e];
    work[l * ls + idx - l * n2] = V{vfma(a.re, b.re, vmul(a.im, b.im)), vdet(a.re, b.im, a.im, b.re)};   // conj(a) b
  }
  __syncthreads();
  auto rows = [ls](int l) { return l * ls; };
  if (few) line_pass_any<false, true>(work, n2, np * rr, 1, tw, tid, nthr, rows);
  else line_pass_any<false>(work, n2, np * rr, 1, tw, tid, nthr, rows);
  // store X[slot][i2][i0][i1s + r]; consecutive threads take consecutive r
  const long slot0 = (long)blockIdx.y * kTileMax * kTileMax;
  for (int idx = tid; idx < np * rowlen; idx += nthr) {
    const int r = idx % rr, rest = idx / rr;
    const int i2 = rest % n2, p = rest / n2;
    if (live(i2, n2, reach2))
      X[(((slot0 + p) * n2 + i2) * n0 + i0) * n1 + i1s + r] = work[(p * rr + r) * ls + places[few][i2]];
  }
}

template <typename T, bool FEW>
__global__ void __launch_bounds__(sizeof(T) == 8 && !FEW ? 512 : 256, FEW ? 4 : sizeof(T) == 8 ? 1 : PairBlocks<T>::value)
    k_fock_f2(cplx<T>* __restrict__ Xc, const PairTile* __restrict__ tiles, int tile0, int n0, int n1, int n2,
              const __grid_constant__ PairReach reach, const T* __restrict__ khat_t, const cplx<T>* __restrict__ tw0_g,
              const cplx<T>* __restrict__ tw1_g) {
  grid_entry();
  using V = typename value_of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int n_cols;
  __shared__ unsigned char cols[kMaxLength], dead[kMaxLength];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int slot = blockIdx.y;
  const int p = slot % (kTileMax * kTileMax);
  if (p >= tiles[tile0 + slot / (kTileMax * kTileMax)].n_pairs) return;
  // live slabs only: blockIdx.x in [0, n_live) maps to frequencies 0..R, then -R..-1
  const int i2 = (int)blockIdx.x <= reach.g2 ? (int)blockIdx.x : (int)blockIdx.x + (n2 - (int)gridDim.x);
  const int reach1 = reach.g1[min(i2, n2 - i2)];
  const int ls = n1 + 1, cnt = n0 * n1;
  V* tw0 = reinterpret_cast<V*>(smem_raw);
  V* tw1 = tw0 + n0;
  V* buf = tw1 + n1;
  load_tw(tw0, tw0_g, n0, tid, nthr);
  load_tw(tw1, tw1_g, n1, tid, nthr);
  if (tid < 32) {   // places of the live axis-1 frequencies, then of the dead ones
    int nl = 0, nd = 0;
    for (int c0 = 0; c0 < n1; c0 += 32) {
      const int c = c0 + tid;
      const bool in = c < n1, lv = in && live(freq_at<FEW>(c, n1), n1, reach1);
      const unsigned ml = __ballot_sync(0xffffffffu, lv), md = __ballot_sync(0xffffffffu, in && !lv);
      const unsigned below = (1u << tid) - 1u;
      if (lv) cols[nl + __popc(ml & below)] = (unsigned char)c;
      else if (in) dead[nd + __popc(md & below)] = (unsigned char)c;
      nl += __popc(ml);
      nd += __popc(md);
    }
    if (tid == 0) n_cols = nl;
  }
  V* X = reinterpret_cast<V*>(Xc) + (long)slot * n2 * cnt;
#pragma unroll 4
  for (int e = tid; e < cnt; e += nthr) buf[e / n1 * ls + e % n1] = X[(long)i2 * cnt + e];
  __syncthreads();
  const int nc = n_cols;
  auto rows = [ls](int l) { return l * ls; };
  auto live_cols = [](int l) { return (int)cols[l]; };
  line_pass_any<false, FEW>(buf, n1, n0, 1, tw1, tid, nthr, rows);           // axis 1
  line_pass_any<false, FEW>(buf, n0, nc, ls, tw0, tid, nthr, live_cols);     // axis 0, live columns
  const T* kt = khat_t + (long)i2 * cnt;
  for (int e = tid; e < nc * n0; e += nthr) {
    const int r = e / nc, c = cols[e - r * nc];
    V& v = buf[r * ls + c];
    const T k = kt[freq_at<FEW>(r, n0) * n1 + freq_at<FEW>(c, n1)];
    v = V{v.re * k, v.im * k};
  }
  for (int e = tid; e < (n1 - nc) * n0; e += nthr) buf[e / (n1 - nc) * ls + dead[e % (n1 - nc)]] = V{(T)0, (T)0};
  __syncthreads();
  line_pass_any<true, FEW>(buf, n0, nc, ls, tw0, tid, nthr, live_cols);
  line_pass_any<true, FEW>(buf, n1, n0, 1, tw1, tid, nthr, rows);
  for (int e = tid; e < cnt; e += nthr) X[(long)i2 * cnt + e] = buf[e / n1 * ls + e % n1];
}

template <typename T>
__global__ void __launch_bounds__(256, PairBlocks<T>::value) k_fock_f3(const PairTile* __restrict__ tiles, int tile0,
                                                    const cplx<T>* __restrict__ Xc, int n0, int n1, int n2, int rr,
                                                    int reach2, const cplx<T>* __restrict__ tw_g) {
  grid_entry();
  using V = typename value_of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ PairTile tl;
  __shared__ unsigned char places[2][kMaxLength];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int rowlen = rr * n2, ls = n2 + 1;
  const V* X = reinterpret_cast<const V*>(Xc);
  V* tw = reinterpret_cast<V*>(smem_raw);
  V* orb = tw + n2;
  V* work = orb + 2 * kTileMax * rowlen;
  for (int t = tid; t < (int)(sizeof(PairTile) / 4); t += nthr)
    reinterpret_cast<unsigned*>(&tl)[t] = reinterpret_cast<const unsigned*>(tiles + tile0 + blockIdx.y)[t];
  load_tw(tw, tw_g, n2, tid, nthr);
  load_places<T>(places, n2, tid, nthr);
  __syncthreads();
  const int nb1 = n1 / rr;
  const int i0 = blockIdx.x / nb1;
  const int i1s = (blockIdx.x - i0 * nb1) * rr;
  const long roff = ((long)i0 * n1 + i1s) * n2;
  const int np = tl.n_pairs;
  const long slot0 = (long)blockIdx.y * kTileMax * kTileMax;
  const bool few = few_lines<T>(n2, np * rr);
#pragma unroll 4
  for (int idx = tid; idx < np * rowlen; idx += nthr) {
    const int r = idx % rr, rest = idx / rr;
    const int i2 = rest % n2, p = rest / n2;
    work[(p * rr + r) * ls + places[few][i2]] =
        live(i2, n2, reach2) ? X[(((slot0 + p) * n2 + i2) * n0 + i0) * n1 + i1s + r] : V{(T)0, (T)0};
  }
  for (int o = 0; o < tl.n_orb; ++o) {
    const V* src = (const V*)tl.in[o] + roff;
    for (int e = tid; e < rowlen; e += nthr) orb[o * rowlen + e] = src[e];
  }
  __syncthreads();
  auto rows = [ls](int l) { return l * ls; };
  if (few) line_pass_any<true, true>(work, n2, np * rr, 1, tw, tid, nthr, rows);
  else line_pass_any<true>(work, n2, np * rr, 1, tw, tid, nthr, rows);
  // each output orbital: fixed-order sum over the tile's pairs, one RMW of its row
  for (int o = 0; o < tl.n_orb; ++o) {
    if (!tl.is_out[o]) continue;
    V* dst = (V*)tl.out[o] + roff;
    for (int e = tid; e < rowlen; e += nthr) {
      const int r = e / n2;
      V acc = {(T)0, (T)0};
      for (int c = 0; c < tl.out_n[o]; ++c) {
        const V v = work[(tl.out_pair[o][c] * rr + r) * ls + e - r * n2], a = orb[tl.out_other[o][c] * rowlen + e];
        if (tl.out_conj[o][c]) acc = padd(acc, V{vfma(a.re, v.re, vmul(a.im, v.im)), vdet(a.im, v.re, a.re, v.im)});
        else acc = padd(acc, V{vdet(a.re, v.re, a.im, v.im), vfma(a.re, v.im, vmul(a.im, v.re))});
      }
      dst[e] = padd(dst[e], acc);
    }
  }
}

// ---------------------------------------------------------------------------
static int rows_per_block(int n1, bool fp64) {
  const int want = fp64 ? 2 : 4;
  for (int r = want; r >= 1; r /= 2)
    if (n1 % r == 0) return r;
  return 1;
}

template <typename T>
cudaError_t fock_pairs(const FockPlan& plan, Grid3 g, const T* khat_t, void* scratch, const DevTwiddles& tw,
                       cudaStream_t s) {
  using C = cplx<T>;
  if constexpr (sizeof(T) == 4) {
    if (fock_fast_supported(g)) return fock_pairs_fast(plan, g, khat_t, scratch, twp<float>(tw, g.n0), s);
  }
  const bool fp64 = sizeof(T) == 8;
  const int rr = rows_per_block(g.n1, fp64);
  const size_t smem13 = (size_t)(g.n2 + 2 * kTileMax * rr * g.n2 + kTileMax * kTileMax * rr * (g.n2 + 1)) * sizeof(C);
  const size_t smem2 = (size_t)(g.n0 + g.n1 + g.n0 * (g.n1 + 1)) * sizeof(C);
  cudaError_t e;
  static std::atomic<unsigned long long> attr_done{0};
  if (const unsigned long long bit = device_bit_todo(attr_done)) {
    e = cudaFuncSetAttribute(k_fock_f1<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_fock_f2<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_fock_f3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    attr_done.fetch_or(bit, std::memory_order_release);
  }
  if (smem13 > 200 * 1024 || smem2 > 200 * 1024) return cudaErrorInvalidConfiguration;
  // Threads. FP64: four blocks per SM keep its pipe busy across barriers, large tiles take wider
  // blocks. Lines of up to 16 points (one codelet each) fill 64 threads, which pays once there
  // are more blocks than four per SM (16 orbitals on 64 x 48 x 16 points: 1605 us an exchange
  // with 128, 1346 so; on 24 x 8 x 16: 249 and 263). FP32: lines of 48 and more points fill 256
  // (16 orbitals on 64 x 48 x 64: 1105 us with 128, 947 so; on 64 x 48 x 32: 514 and 592).
  const bool few = fp64 && g.n0 <= 16 && g.n1 <= 16;
  const int thr13 = g.n2 >= (fp64 ? 96 : 48) ? 256 : 128;
  const int thr2 = few ? 64 : smem2 > 50 * 1024 ? 256 : 128;
  const C* tw0 = twp<T>(tw, g.n0);
  const C* tw1 = twp<T>(tw, g.n1);
  const C* tw2 = twp<T>(tw, g.n2);
  C* X = (C*)scratch;
  auto f2 = k_fock_f2<T, false>;
  if constexpr (sizeof(T) == 8) f2 = few ? k_fock_f2<T, true> : f2;
  // frequencies of pair products; with aliasing along axis 1 or 2 any may hold one
  PairReach reach;
  const bool free2 = 2 * plan.g2_reach + 1 <= g.n2, free1 = 2 * plan.g1_reach[0] + 1 <= g.n1;
  reach.g2 = free2 ? plan.g2_reach : g.n2;
  for (int k = 0; k <= kMaxLength / 2; ++k)
    reach.g1[k] = (unsigned char)(free1 && free2 && k <= plan.g2_reach ? plan.g1_reach[k] : g.n1);
  const unsigned n_live = free2 ? 2 * plan.g2_reach + 1 : g.n2;
  for (int l = 0; l < plan.n_launch; ++l) {
    const int t0 = plan.launch_first[l], nt = plan.launch_count[l];
    dim3 g13((unsigned)(g.n0 * (g.n1 / rr)), (unsigned)nt);
    const int t13 = fp64 && g.n2 <= 16 && (long)g13.x * nt > 4L * sm_count() ? 64 : thr13;
    launch(g13, t13, smem13, s)(k_fock_f1<T>, plan.d_tiles, t0, X, g.n0, g.n1, g.n2, rr, reach.g2, tw2); launched();
    dim3 g2(n_live, (unsigned)(nt * kTileMax * kTileMax));
    // FP64, large slabs: 512 threads (the registers of an SM) where no second block shares the
    // SM, for its shared memory or because there are no more slabs (5 orbitals on 64 x 96 x 12
    // points: 641 us an exchange with 256, 526 so)
    const bool alone = fp64 && smem2 > 50 * 1024 &&
                       (2 * smem2 > 220 * 1024 || (long)n_live * nt * kTileMax * kTileMax <= 2L * sm_count());
    launch(g2, alone ? 512 : thr2, smem2, s)(f2, X, plan.d_tiles, t0, g.n0, g.n1, g.n2, reach, khat_t, tw0, tw1); launched();
    launch(g13, t13, smem13, s)(k_fock_f3<T>, plan.d_tiles, t0, X, g.n0, g.n1, g.n2, rr, reach.g2, tw2); launched();
  }
  return cudaGetLastError();
}

template cudaError_t fock_pairs<float>(const FockPlan&, Grid3, const float*, void*, const DevTwiddles&,
                                       cudaStream_t);
template cudaError_t fock_pairs<double>(const FockPlan&, Grid3, const double*, void*, const DevTwiddles&,
                                        cudaStream_t);

void fock_bind_tiles(PairTile* tiles, int n, const void* psi_r, const void* x_r, void* w_occ, void* w_x, long N,
                     size_t cs) {
  for (int t = 0; t < n; ++t) {
    PairTile& tl = tiles[t];
    for (int o = 0; o < 2 * kTileMax; ++o) {
      tl.in[o] = nullptr;
      tl.out[o] = nullptr;
      if (o >= tl.n_orb) continue;
      const size_t off = (size_t)tl.orb[o] * (size_t)N * cs;
      tl.in[o] = (const unsigned char*)(tl.src[o] == 0 ? psi_r : x_r) + off;
      if (tl.is_out[o]) tl.out[o] = (unsigned char*)(tl.src[o] == 0 ? w_occ : w_x) + off;
    }
  }
}

// ---------------------------------------------------------------------------
// Tile schedule. Symmetric: blocks of `tile` orbitals; rounds of a
// round-robin tournament pair the blocks so each block appears once per
// round (off-diagonal tiles: all |A| x |B| pairs), then one round of the
// diagonal tiles (pairs a <= b inside a block). Non-symmetric (V_X applied to
// other vectors): round r pairs X-block b with occupied block (b + r) mod nbo.
// Paired order: blocks go two by two, (A, A') and (B, B'), through the tournament, and each
// meeting is the tiles A B, A' B', then A B', A' B; the diagonal ones are A A, A' A', then A A'.
long fock_max_tiles(int n_occ, int tile) {
  const long nb = (n_occ + tile - 1) / tile, np = (nb + 1) / 2;
  return 2 * np * (np + 1);
}

int fock_build_tiles(int n_occ, int n_x, int tile, int sym, int order, int tiles_per_launch, PairTile** tiles_out,
                     int** launch_first, int** launch_count, int* n_launch) {
  if (tile < 1 || tile > kTileMax || n_occ < 1 || tiles_per_launch < (order == TILE_GROUPED ? 4 : 1)) return -1;
  std::vector<PairTile> tiles;
  std::vector<std::vector<int>> rounds;   // tile indices per round
  auto block_range = [&](int b, int n, int* lo) { *lo = b * tile; return std::min(n, (b + 1) * tile) - b * tile; };
  auto make_tile = [&](int a_lo, int a_n, int a_src, int b_lo, int b_n, int b_src, bool diag, int out_a,
                       int out_b) {
    PairTile t;
    std::memset(&t, 0, sizeof(t));
    for (int i = 0; i < a_n; ++i) { t.orb[t.n_orb] = a_lo + i; t.src[t.n_orb] = (signed char)a_src; t.is_out[t.n_orb] = (signed char)out_a; ++t.n_orb; }
    if (!diag)
      for (int i = 0; i < b_n; ++i) { t.orb[t.n_orb] = b_lo + i; t.src[t.n_orb] = (signed char)b_src; t.is_out[t.n_orb] = (signed char)out_b; ++t.n_orb; }
    if (diag) {
      for (int a = 0; a < a_n; ++a)
        for (int b = a; b < a_n; ++b) { t.pi[t.n_pairs] = (signed char)a; t.pj[t.n_pairs] = (signed char)b; ++t.n_pairs; }
    } else {
      for (int a = 0; a < a_n; ++a)
        for (int b = 0; b < b_n; ++b) { t.pi[t.n_pairs] = (signed char)a; t.pj[t.n_pairs] = (signed char)(a_n + b); ++t.n_pairs; }
    }
    for (int o = 0; o < t.n_orb; ++o) {
      if (!t.is_out[o]) continue;
      int c = 0;
      for (int q = 0; q < t.n_pairs; ++q) {
        if (t.pj[q] == o) { t.out_pair[o][c] = (signed char)q; t.out_other[o][c] = t.pi[q]; t.out_conj[o][c] = 0; ++c; }
        if (sym && t.pi[q] == o && t.pi[q] != t.pj[q]) {
          t.out_pair[o][c] = (signed char)q; t.out_other[o][c] = t.pj[q]; t.out_conj[o][c] = 1; ++c;
        }
      }
      t.out_n[o] = (signed char)c;
    }
    tiles.push_back(t);
    return (int)tiles.size() - 1;
  };
  if (sym && order != TILE_ROUNDS) {
    const int nb = (n_occ + tile - 1) / tile, np = (nb + 1) / 2, npp = np + (np & 1);
    auto pair_tile = [&](int a, int b) {
      int alo, blo;
      const int an = block_range(a, n_occ, &alo), bn = block_range(b, n_occ, &blo);
      return make_tile(alo, an, 0, blo, bn, 0, a == b, 1, 1);
    };
    // a meeting's tiles, the first `apart` of them without a common block; the rest likewise
    auto add = [&](std::vector<int>* first, std::vector<int>* second, const std::vector<int>& t, size_t apart) {
      for (size_t k = 0; k < t.size(); ++k) (order == TILE_GROUPED || k < apart ? first : second)->push_back(t[k]);
      if (order == TILE_GROUPED) first->resize((first->size() + 3) / 4 * 4, -1);
    };
    auto end_round = [&](std::vector<int>* rd) {
      if (!rd->empty()) rounds.push_back(*rd);
      rd->clear();
    };
    std::vector<int> one, two;
    for (int r = 0; r < npp - 1; ++r) {
      for (int i = 0; i < npp / 2; ++i) {
        int a = i == 0 ? r : (r + i) % (npp - 1), b = i == 0 ? npp - 1 : (r - i + npp - 1) % (npp - 1);
        if (a >= np || b >= np) continue;
        if (a > b) std::swap(a, b);
        if (2 * b + 1 < nb)
          add(&one, &two, {pair_tile(2 * a, 2 * b), pair_tile(2 * a + 1, 2 * b + 1), pair_tile(2 * a, 2 * b + 1),
                           pair_tile(2 * a + 1, 2 * b)}, 2);
        else
          add(&one, &two, {pair_tile(2 * a, 2 * b), pair_tile(2 * a + 1, 2 * b)}, 1);
      }
      end_round(&one);
      end_round(&two);
    }
    for (int a = 0; a < np; ++a) {
      if (2 * a + 1 < nb) add(&one, &two, {pair_tile(2 * a, 2 * a), pair_tile(2 * a + 1, 2 * a + 1), pair_tile(2 * a, 2 * a + 1)}, 2);
      else add(&one, &two, {pair_tile(2 * a, 2 * a)}, 1);
    }
    end_round(&one);
    end_round(&two);
    if (order == TILE_GROUPED) tiles_per_launch -= tiles_per_launch % 4;
  } else if (sym) {
    const int nb = (n_occ + tile - 1) / tile;
    const int nbp = nb + (nb & 1);
    for (int r = 0; r < nbp - 1; ++r) {
      std::vector<int> rd;
      for (int i = 0; i < nbp / 2; ++i) {
        int a, b;
        if (i == 0) { a = r; b = nbp - 1; }
        else { a = (r + i) % (nbp - 1); b = (r - i + nbp - 1) % (nbp - 1); }
        if (a >= nb || b >= nb) continue;
        if (a > b) std::swap(a, b);
        int alo, blo;
        const int an = block_range(a, n_occ, &alo), bn = block_range(b, n_occ, &blo);
        rd.push_back(make_tile(alo, an, 0, blo, bn, 0, false, 1, 1));
      }
      if (!rd.empty()) rounds.push_back(rd);
    }
    std::vector<int> rd;
    for (int b = 0; b < nb; ++b) {
      int lo;
      const int bn = block_range(b, n_occ, &lo);
      rd.push_back(make_tile(lo, bn, 0, 0, 0, 0, true, 1, 0));
    }
    rounds.push_back(rd);
  } else {
    const int nbo = (n_occ + tile - 1) / tile, nbx = (n_x + tile - 1) / tile;
    for (int r = 0; r < nbo; ++r) {
      std::vector<int> rd;
      for (int bx = 0; bx < nbx; ++bx) {
        const int bo = (bx + r) % nbo;
        int alo, blo;
        const int an = block_range(bo, n_occ, &alo), bn = block_range(bx, n_x, &blo);
        rd.push_back(make_tile(alo, an, 0, blo, bn, 1, false, 0, 1));
      }
      rounds.push_back(rd);
    }
  }
  // order tiles by round and split rounds into launches of at most tiles_per_launch
  std::vector<PairTile> ordered;
  std::vector<int> lf, lc;
  for (auto& rd : rounds) {
    for (size_t k = 0; k < rd.size(); k += tiles_per_launch) {
      const int cnt = (int)std::min<size_t>(tiles_per_launch, rd.size() - k);
      lf.push_back((int)ordered.size());
      lc.push_back(cnt);
      for (int q = 0; q < cnt; ++q) ordered.push_back(rd[k + q] < 0 ? PairTile{} : tiles[rd[k + q]]);
    }
  }
  *tiles_out = (PairTile*)std::malloc(sizeof(PairTile) * ordered.size());
  std::memcpy(*tiles_out, ordered.data(), sizeof(PairTile) * ordered.size());
  *launch_first = (int*)std::malloc(sizeof(int) * lf.size());
  *launch_count = (int*)std::malloc(sizeof(int) * lc.size());
  std::memcpy(*launch_first, lf.data(), sizeof(int) * lf.size());
  std::memcpy(*launch_count, lc.data(), sizeof(int) * lc.size());
  *n_launch = (int)lf.size();
  return (int)ordered.size();
}

}  // namespace pt
