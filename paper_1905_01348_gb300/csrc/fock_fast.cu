// FP32 pair pipeline for cubic grids of 32, 48, 64 or 96 points per edge (the
// Si8 / Si64 / Si216 workloads, and 48 for the Si216 wavefunction grid): the same three
// passes as fock.cu (Eq. 3, pair loop of Alg. 2) on packed pairs of lines (fft_pk.cuh):
// every value in registers and shared memory is a pk2, the same element of two
// neighbouring grid rows, so that one packed FP32 instruction, one 16-byte shared access
// and one address serve two lines.
//
// Pair intermediate X: [pair slot][i2][i0][i1 / 2] of pk2, a pk2 holding i1 and i1 + 1
// (the byte count and position of two complex64 values); only the axis-2 slabs that
// pair products can reach are written or read.
// Kernel table (fast_khat_index): [i2][i1 / 2][i0] pairs of K(i1), K(i1 + 1), i1 even: the two
// frequencies one pk2 of F2's inner step holds, in the order its threads read.
#include <algorithm>

#include "common.cuh"
#include "fft_pk.cuh"
#include "internal.h"

namespace pt {

namespace {

constexpr int TT = kTileMax;      // orbitals per tile edge
constexpr int NPAIR = TT * TT;
constexpr int RP = 4;             // row pairs per block in F1 / F3
constexpr int RR = 2 * RP;        // grid rows per block
constexpr int QB = 4;             // pairs of a tile worked on together in F1 / F3

template <int L> struct Sizes {
  static constexpr int M = L / 8;                       // second radix of the axis-2 lines
  static constexpr int MP = M + 1;                      // odd: spreads (row pair, k2) over the banks
  static constexpr int QS = 8 * RP * MP + 2;            // one pair's part of the exchange buffer; 2 mod 8
  static constexpr int NT = 16 * (M > 8 ? M : 8);       // threads of F1 / F3
  static constexpr int RS = L == 48 ? L + 2 : L + (M == 12 ? 6 : M == 8 ? 4 : 2);   // orbital row stride
  // orbital stride: the same elements of four orbitals lie 32 bytes apart in the banks. With the
  // twiddles MP apart, a quarter of F1's and F3's shared accesses waited for a bank without
  // (128 orbitals at 64^3: 18.0 -> 17.2 ms)
  static constexpr int OS = RR * RS + 4;
  static constexpr size_t tw_bytes = sizeof(pk2) * 8 * MP;
  static constexpr size_t orb_bytes = sizeof(float2) * 2 * TT * OS;
  static constexpr size_t smem13 = tw_bytes + orb_bytes + sizeof(pk2) * QB * QS;
  static constexpr int CP = L / 2;                      // pk2 values of a row of X
  // F2: L = 4 Q, Q / 2 column pairs of 16 Q values each
  static constexpr int Q = L / 4;
  static constexpr int CPQ = Q / 2;
  static constexpr int SC = 16 * Q + 1;
  static constexpr int ROT = Q == 16 ? 0 : Q == 12 ? 6 : 4;   // rotation of k2 at odd u: spreads (c', p) over the banks
  static constexpr size_t smem2 = sizeof(pk2) * (4 * Q + 4 * CPQ + CPQ * SC);
  // 96: two blocks of 192 threads (one round of steps A and C) beat three of 96 or 128 by 4 to
  // 5%, and by 12% three of 192, whose 96 registers spill
  static constexpr int NT2 = L == 96 ? 192 : L == 64 ? 128 : L == 48 ? 96 : 64;
  static constexpr int MINB2 = L == 96 ? 2 : L == 64 ? 4 : 6;
  // F2 brings the slab of the block that will take its place into L2: with two blocks an SM
  // their loads are not hidden (96: 334.3 -> 331.1 ms, 288 orbitals); with four and more they are
  // (64: 18.2 ms without, 18.4 with)
  static constexpr bool AHEAD2 = L == 96;
  static constexpr int RG = L * (L / RR);               // row groups of a tile
  static constexpr int RES1 = L == 96 ? 2 : 4;          // resident F1 and F3 blocks per SM
  static constexpr int RES3 = L == 96 ? 2 : 3;
};

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// waits until at most N of the thread's newest groups are in flight
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Axis-2 slab i2 is dead when its frequency lies beyond the pair reach R:
// the pair products have no component there (the slab stays unwritten in X).
template <int L> __device__ __forceinline__ bool dead_slab(int i2, int reach) { return i2 > reach && i2 < L - reach; }

// bit k1: slab k2 + 8 k1 is live
template <int L> __device__ __forceinline__ unsigned live_mask(int k2, int reach) {
  unsigned m = 0;
  for (int k1 = 0; k1 < L / 8; ++k1) m |= dead_slab<L>(k2 + 8 * k1, reach) ? 0u : 1u << k1;
  return m;
}

// An off-diagonal tile of two full orbital blocks: orbitals 0..3 and 4..7,
// pair 4a + b = (a, 4 + b).
__device__ __forceinline__ bool full_tile(const PairTile& tl) { return tl.n_orb == 2 * TT && tl.n_pairs == NPAIR; }

// The walk of an F1 or F3 block: an item is a row group of a group of 1 << glog tiles,
// which the block takes one after another, so that the orbital rows (and W rows) they share
// come from L2 the second time. Unit u is tile u % (1 << glog) of the block's item u >> glog.
template <int L> struct Walk {
  int first, stride, glog, units;
  __device__ __forceinline__ Walk(int n_items, int glog_)
      : first(blockIdx.x), stride(gridDim.x), glog(glog_),
        units(((n_items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1) << glog_) {}
  __device__ __forceinline__ int item(int u) const { return first + (u >> glog) * stride; }
  __device__ __forceinline__ int tile(int u) const { return ((item(u) / Sizes<L>::RG) << glog) + (u & ((1 << glog) - 1)); }
  __device__ __forceinline__ int rows(int u) const { return item(u) % Sizes<L>::RG; }   // row group
};

// the tile record into shared memory, asynchronously
__device__ __forceinline__ void copy_tile(PairTile* dst, const PairTile* src, int tid) {
  static_assert(sizeof(PairTile) % 16 == 0, "copied by 16 bytes");
  if (tid < (int)(sizeof(PairTile) / 16))
    cp_async16(reinterpret_cast<unsigned char*>(dst) + 16 * tid, reinterpret_cast<const unsigned char*>(src) + 16 * tid);
}

// twiddles W_L^(n1 k2) = c - i s as (c, c, s, s) at [k2][n1], MP apart
template <int L> __device__ __forceinline__ void load_twiddles(pk2* tw, const float2* __restrict__ tw_g, int tid, int nt) {
  constexpr int M = Sizes<L>::M;
  for (int t = tid; t < L; t += nt) {
    const float2 w = tw_g[(t / M) * (t % M)];
    tw[t / M * Sizes<L>::MP + t % M] = {f2(w.x), f2(-w.y)};
  }
}

// RR rows (from element roff) of the tile's orbitals o0 .. o1 - 1 into shared memory by
// 16-byte asynchronous copies
template <int L>
__device__ __forceinline__ void load_orbitals(float2* orb, const PairTile& tl, int o0, int o1, long roff, int tid) {
  using S = Sizes<L>;
  constexpr int CH = RR * L / 2, PER = (CH + S::NT - 1) / S::NT;   // 16-byte chunks per orbital and per thread
  const int end = min(tl.n_orb, o1);
  for (int o = o0; o < end; ++o) {
    const float2* src = static_cast<const float2*>(tl.in[o]) + roff;
    float2* dst = orb + o * S::OS;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int e = tid + q * S::NT;
      if (CH % S::NT == 0 || e < CH) cp_async16(dst + (e / (L / 2)) * S::RS + 2 * (e % (L / 2)), src + 2 * e);
    }
  }
}

// element n of rows 2 rp and 2 rp + 1 of orbital o
template <int L> __device__ __forceinline__ pk2 orb_at(const float2* orb, int o, int rp, int n) {
  const float2* p = orb + o * Sizes<L>::OS + 2 * rp * Sizes<L>::RS + n;
  const float2 u = p[0], v = p[Sizes<L>::RS];
  return {make_float2(u.x, v.x), make_float2(u.y, v.y)};
}

// a load that stays where it is written: the compiler would move it down to its use,
// past the barrier, and its latency with it
__device__ __forceinline__ pk2 load_now(const pk2* p) {
  pk2 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n"
               : "=f"(v.re.x), "=f"(v.re.y), "=f"(v.im.x), "=f"(v.im.y)
               : "l"(p)
               : "memory");
  return v;
}

// adds v to a row pair in global memory without waiting for the old values; every element
// has one writer per launch, so the sums keep their order
__device__ __forceinline__ void red_add(float2* p, float x, float y) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};\n" ::"l"(p), "f"(x), "f"(y) : "memory");
}
template <int L> __device__ __forceinline__ void add_rows(float2* p, pk2 v) {
  red_add(p, v.re.x, v.im.x);
  red_add(p + L, v.re.y, v.im.y);
}

__device__ __forceinline__ pk2 pk_select(bool first, pk2 a, pk2 b) {
  return {make_float2(first ? a.re.x : b.re.x, first ? a.re.y : b.re.y),
          make_float2(first ? a.im.x : b.im.x, first ? a.im.y : b.im.y)};
}
__device__ __forceinline__ pk2 pk_shfl_xor(pk2 a, int m) {
  return {make_float2(__shfl_xor_sync(0xffffffffu, a.re.x, m), __shfl_xor_sync(0xffffffffu, a.re.y, m)),
          make_float2(__shfl_xor_sync(0xffffffffu, a.im.x, m), __shfl_xor_sync(0xffffffffu, a.im.y, m))};
}

// the largest |k0| that pair products hold at axis-2 frequency |k2| (L: all)
struct RowReach {
  unsigned char at[kMaxLength / 2 + 1];
};

// asks for `bytes` (a multiple of 16) at p, 16-byte aligned, in L2
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}

}  // namespace

// F1: pair products of RR grid rows for every pair of the tile, forward FFT along axis 2,
// store of the live slabs. Resident blocks walk the (tile, row group) items; the next item's
// orbital rows arrive by asynchronous copies, each orbital's as soon as the current item
// is done with its place, so no item waits for memory. The pairs are worked on four at a
// time: (row pair, n1, pair) threads form the products and run the 8-point DFTs, the values
// cross shared memory once, and (row pair, k2, pair) threads run the M-point DFTs and store
// from registers (64 contiguous bytes per pair and slab). The pair is the fastest thread
// index of the first step, so one read of a left orbital serves four pairs; a full tile
// keeps the right orbitals' values in registers for all of its left ones.
template <int L>
__global__ void __launch_bounds__(Sizes<L>::NT, Sizes<L>::RES1) k_fast_f1(const PairTile* __restrict__ tiles, int n_items, int glog,
                                                          pk2* __restrict__ X, const float2* __restrict__ tw_g,
                                                          int reach) {
  grid_entry();
  using S = Sizes<L>;
  constexpr int M = S::M, MP = S::MP, QS = S::QS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(16) PairTile ring[3];   // the tiles of this item, the next and the one after
  pk2* tw = reinterpret_cast<pk2*>(smem_raw);
  float2* orb = reinterpret_cast<float2*>(smem_raw + S::tw_bytes);
  pk2* ex = reinterpret_cast<pk2*>(smem_raw + S::tw_bytes + S::orb_bytes);
  const int tid = threadIdx.x;
  const Walk<L> walk(n_items, glog);
  copy_tile(&ring[0], tiles + walk.tile(0), tid);
  if (walk.units > 1) copy_tile(&ring[1], tiles + walk.tile(1), tid);
  load_twiddles<L>(tw, tw_g, tid, S::NT);
  cp_async_wait_all();
  __syncthreads();
  load_orbitals<L>(orb, ring[0], 0, 2 * TT, (long)walk.rows(0) * (RR * L), tid);
  const int qa = tid % QB, n1 = (tid / QB) % M, rpa = tid / (QB * M);
  const int rpb = tid % RP, k2b = (tid / RP) % 8, qb = tid / (8 * RP);
  const bool first = rpa < RP;   // M < 8: the last threads only take part in the second step
  const unsigned live = live_mask<L>(k2b, reach);
  pk2 wk[8];   // this thread's twiddles (288 orbitals at 96^3: 330.4 -> 329.3 ms)
#pragma unroll
  for (int k2 = 1; k2 < 8; ++k2) wk[k2] = tw[k2 * MP + n1];
  int cur = 0;
  bool was_full = false;
  for (int u = 0; u < walk.units; ++u) {
    // After a full item four groups are in flight, orbitals (0, right), 1, 2, 3; a full item
    // waits for each as it comes to it.
    const bool piped = was_full && full_tile(ring[cur]);
    if (piped) cp_async_wait<3>(); else cp_async_wait_all();
    __syncthreads();
    const int nxt = cur == 2 ? 0 : cur + 1, far = cur == 0 ? 2 : cur - 1;
    const PairTile& tl = ring[cur];
    const bool more = u + 1 < walk.units;
    const long noff = (long)walk.rows(u + 1) * (RR * L);
    if (u + 2 < walk.units) copy_tile(&ring[far], tiles + walk.tile(u + 2), tid);
    const int np = tl.n_pairs;
    const bool full = full_tile(tl);
    pk2* xb = X + (((long)walk.tile(u) * NPAIR + qb) * L + k2b) * (L * S::CP) + walk.rows(u) * RP + rpb;
    if (np == 0 && more) load_orbitals<L>(orb, ring[nxt], 0, 2 * TT, noff, tid);   // an empty tile
    pk2 b[8];
    if (full && first) {
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) b[n2] = orb_at<L>(orb, TT + qa, rpa, n1 + M * n2);
    }
    for (int p0 = 0; p0 < np; p0 += QB, xb += (long)QB * L * L * S::CP) {
      if (first && p0 + qa < np) {
        if (!full) {
          const int oj = tl.pj[p0 + qa];
#pragma unroll
          for (int n2 = 0; n2 < 8; ++n2) b[n2] = orb_at<L>(orb, oj, rpa, n1 + M * n2);
        }
        const int oi = tl.pi[p0 + qa];
        pk2 v[8];
#pragma unroll
        for (int n2 = 0; n2 < 8; ++n2) {
          const pk2 a = orb_at<L>(orb, oi, rpa, n1 + M * n2);
          v[n2] = {vfma(a.re, b[n2].re, vmul(a.im, b[n2].im)), vdet(a.re, b[n2].im, a.im, b[n2].re)};
        }
        pk_dft<8, false>(v);   // of conj(a) b
        pk2* dst = ex + qa * QS + rpa * MP + n1;
        dst[0] = v[0];
#pragma unroll
        for (int k2 = 1; k2 < 8; ++k2) dst[k2 * RP * MP] = ptwiddle<false>(v[k2], wk[k2]);
      }
      __syncthreads();
      if (more) {   // places of orbitals this item no longer reads
        if (full) {
          load_orbitals<L>(orb, ring[nxt], p0 / QB, p0 / QB + 1, noff, tid);
          if (p0 == 0) load_orbitals<L>(orb, ring[nxt], TT, 2 * TT, noff, tid);
        } else if (p0 + QB >= np) {
          load_orbitals<L>(orb, ring[nxt], 0, 2 * TT, noff, tid);
        }
      }
      cp_async_commit();
      if (qb < QB && p0 + qb < np) {
        pk2 v[M];
        const pk2* src = ex + qb * QS + (k2b * RP + rpb) * MP;
#pragma unroll
        for (int m = 0; m < M; ++m) v[m] = src[m];
        pk_dft<M, false>(v);
#pragma unroll
        for (int k1 = 0; k1 < M; ++k1)
          if (live & (1u << k1)) xb[(long)k1 * 8 * L * S::CP] = v[k1];
      }
      if (piped) cp_async_wait<3>();
      __syncthreads();
    }
    cur = nxt;
    was_full = full;
  }
}

// F2: one live (pair, i2) slab per block: FFT along both of its axes, kernel multiply,
// inverse FFTs, in place. Shared-memory bandwidth bounds it (every value crosses at 16
// bytes per pair of lines), so the 2D transform takes three steps instead of two per axis:
// with L = 4 Q,
//   A  Q-point DFTs along axis 0 over i0 = n1 + 4 n2 (packed over neighbouring columns i1,
//      as X stores them), straight from global memory;
//   B  both radix-4 steps at once, 4 x 4 values per thread: axis 0 over n1 (rows k0 = k2 +
//      Q k1) and axis 1 over i1 = c + Q p (outputs q, twiddle W_L^(c q)), then a 2 x 2
//      transpose in registers packs over (q, q + 1) instead of (c, c + 1);
//   C  Q-point DFTs along axis 1 over c (frequency 4 m + q), kernel multiply, and back;
// then B and A backwards, storing from registers. Values stay at fixed places (a step's
// outputs overwrite its own inputs): place (c', u, k2) = c' SC + u Q + k2 with c' = c / 2 and
// u = (n1, p) before and (k1, c & 1, q / 2) after B; at odd u, k2 is rotated by ROT. Threads
// of neighbouring c' (A) and of neighbouring k2 (B, C) touch distinct banks.
// Rows k0 outside the ball that holds the pair products (a quarter of a live slab's) are not
// stored by B and not taken by C, whose threads share the rest (288 orbitals at 96^3: 335.6 ->
// 331.1 ms an exchange).
template <int L>
__global__ void __launch_bounds__(Sizes<L>::NT2, Sizes<L>::MINB2)
    k_fast_f2(pk2* __restrict__ X, const PairTile* __restrict__ tiles, const float2* __restrict__ kt2,
              const float2* __restrict__ tw_g, int reach, const __grid_constant__ RowReach rows, int ahead) {
  grid_entry();
  using S = Sizes<L>;
  constexpr int Q = S::Q, CP = S::CP, CPQ = S::CPQ, SC = S::SC, ROT = S::ROT, NT = S::NT2;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int tid = threadIdx.x;
  const int slot = blockIdx.y;
  if (slot % NPAIR >= tiles[slot / NPAIR].n_pairs) return;
  // live slabs only: blockIdx.x in [0, n_live) maps to frequencies 0..R, then -R..-1
  const int i2 = (int)blockIdx.x <= reach ? (int)blockIdx.x : (int)blockIdx.x + (L - (int)gridDim.x);
  pk2* twa = reinterpret_cast<pk2*>(smem_raw);   // W_L^(n1 k2) at [n1][k2]
  pk2* twb = twa + 4 * Q;                        // W_L^(c q), c = 2 c' and 2 c' + 1, at [q][c']
  pk2* buf = twb + 4 * CPQ;
  for (int t = tid; t < 4 * Q; t += NT) {
    const float2 w = tw_g[(t / Q) * (t % Q)];
    twa[t] = {f2(w.x), f2(-w.y)};
  }
  for (int t = tid; t < 4 * CPQ; t += NT) {
    const int q = t / CPQ, c = 2 * (t % CPQ);
    const float2 w = tw_g[q * c], z = tw_g[q * (c + 1)];
    twb[t] = {make_float2(w.x, z.x), make_float2(-w.y, -z.y)};
  }
  pk2* slab = X + ((long)slot * L + i2) * (L * CP);
  // the slab of the block that takes this one's place, into L2
  if (tid == 0 && ahead > 0) {
    const unsigned next = blockIdx.y * gridDim.x + blockIdx.x + ahead, y = next / gridDim.x, x = next % gridDim.x;
    if (y < gridDim.y && y % NPAIR < (unsigned)tiles[y / NPAIR].n_pairs) {
      const int j2 = (int)x <= reach ? (int)x : (int)x + (L - (int)gridDim.x);
      prefetch_l2(X + ((long)y * L + j2) * (L * CP), L * CP * sizeof(pk2));
    }
  }
  const int r0 = rows.at[min(i2, L - i2)];   // rows (frequencies k0) that hold pair products
  auto live0 = [&](int k0) { return k0 <= r0 || k0 >= L - r0; };
  __syncthreads();
#pragma unroll 1
  for (int t = tid; t < 8 * Q; t += NT) {
    const int c2 = t % CP, n1 = t / CP;
    const pk2* src = slab + n1 * CP + c2;
    pk2 v[Q];
#pragma unroll
    for (int n2 = 0; n2 < Q; ++n2) v[n2] = src[n2 * 4 * CP];
    pk_dft<Q, false>(v);
    const int odd = (c2 / CPQ) & 1;
    pk2* dst = buf + (c2 % CPQ) * SC + (4 * n1 + c2 / CPQ) * Q + odd * ROT;
    pk2* wrap = dst - odd * Q;   // of the last ROT values
    dst[0] = v[0];
#pragma unroll
    for (int k2 = 1; k2 < Q; ++k2) (k2 < Q - ROT ? dst : wrap)[k2] = ptwiddle<false>(v[k2], twa[n1 * Q + k2]);
  }
  __syncthreads();
#pragma unroll 1
  for (int t = tid; t < CPQ * Q; t += NT) {
    const int c1 = t / Q;
    pk2* p = buf + c1 * SC + t % Q;                    // even u
    pk2* r = buf + c1 * SC + (t % Q + ROT) % Q;        // odd u
    pk2 v[4][4];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u / 4][u % 4] = (u % 2 ? r : p)[u * Q];
#pragma unroll
    for (int h = 0; h < 4; ++h) pk_dft4(v[0][h], v[1][h], v[2][h], v[3][h]);
#pragma unroll
    for (int h = 0; h < 4; ++h) pk_dft4(v[h][0], v[h][1], v[h][2], v[h][3]);
#pragma unroll
    for (int q = 1; q < 4; ++q) {
      const pk2 w = twb[q * CPQ + c1];
#pragma unroll
      for (int h = 0; h < 4; ++h) v[h][q] = ptwiddle<false>(v[h][q], w);
    }
#pragma unroll
    for (int h = 0; h < 4; ++h)
      if (live0(t % Q + Q * h)) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const pk2 a = v[h][2 * g], b = v[h][2 * g + 1];
          (g ? r : p)[(4 * h + g) * Q] = {make_float2(a.re.x, b.re.x), make_float2(a.im.x, b.im.x)};
          (g ? r : p)[(4 * h + 2 + g) * Q] = {make_float2(a.re.y, b.re.y), make_float2(a.im.y, b.im.y)};
        }
      }
  }
  __syncthreads();
  const float2* kt = kt2 + (long)i2 * (L * CP);
  const int n0 = min(L, 2 * r0 + 1);
#pragma unroll 1
  for (int t = tid; t < 2 * n0; t += NT) {
    const int g = t >= n0, j = t - g * n0, k0 = j <= r0 ? j : j + L - n0;
    const int k2 = k0 % Q, k1 = k0 / Q;
    pk2* p = buf + (4 * k1 + g) * Q + (k2 + g * ROT) % Q;
    pk2 v[Q];
#pragma unroll
    for (int c = 0; c < Q; ++c) v[c] = p[(c >> 1) * SC + 2 * Q * (c & 1)];
    pk_dft<Q, false>(v);
#pragma unroll
    for (int m = 0; m < Q; ++m) {
      const float2 kk = __ldg(kt + (2 * m + g) * L + k0);
      v[m] = {vmul(v[m].re, kk), vmul(v[m].im, kk)};
    }
    pk_dft<Q, true>(v);
#pragma unroll
    for (int c = 0; c < Q; ++c) p[(c >> 1) * SC + 2 * Q * (c & 1)] = v[c];
  }
  __syncthreads();
#pragma unroll 1
  for (int t = tid; t < CPQ * Q; t += NT) {
    const int c1 = t / Q;
    pk2* p = buf + c1 * SC + t % Q;                    // even u
    pk2* r = buf + c1 * SC + (t % Q + ROT) % Q;        // odd u
    pk2 v[4][4];
#pragma unroll
    for (int h = 0; h < 4; ++h)
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        pk2 a = {f2(0.f), f2(0.f)}, b = a;
        if (live0(t % Q + Q * h)) {
          a = (g ? r : p)[(4 * h + g) * Q];
          b = (g ? r : p)[(4 * h + 2 + g) * Q];
        }
        v[h][2 * g] = {make_float2(a.re.x, b.re.x), make_float2(a.im.x, b.im.x)};
        v[h][2 * g + 1] = {make_float2(a.re.y, b.re.y), make_float2(a.im.y, b.im.y)};
      }
#pragma unroll
    for (int q = 1; q < 4; ++q) {
      const pk2 w = twb[q * CPQ + c1];
#pragma unroll
      for (int h = 0; h < 4; ++h) v[h][q] = ptwiddle<true>(v[h][q], w);
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) pk_dft<4, true>(v[h]);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      pk2 z[4] = {v[0][h], v[1][h], v[2][h], v[3][h]};
      pk_dft<4, true>(z);
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) (h % 2 ? r : p)[(4 * n1 + h) * Q] = z[n1];
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int t = tid; t < 8 * Q; t += NT) {
    const int c2 = t % CP, n1 = t / CP;
    const int odd = (c2 / CPQ) & 1;
    const pk2* p = buf + (c2 % CPQ) * SC + (4 * n1 + c2 / CPQ) * Q + odd * ROT;
    const pk2* wrap = p - odd * Q;
    pk2 v[Q];
    v[0] = p[0];
#pragma unroll
    for (int k2 = 1; k2 < Q; ++k2) v[k2] = ptwiddle<true>((k2 < Q - ROT ? p : wrap)[k2], twa[n1 * Q + k2]);
    pk_dft<Q, true>(v);
    pk2* dst = slab + n1 * CP + c2;
#pragma unroll
    for (int n2 = 0; n2 < Q; ++n2) dst[n2 * 4 * CP] = v[n2];
  }
}

// F3: inverse FFT along axis 2 for four pairs of the tile at a time, the steps of F1
// backwards, then the accumulation into the W rows (one writer per row). In an
// off-diagonal tile of two full blocks the four pairs share orbital a: each thread
// adds psi_a v_ab to its registers' sums for W_b (added to W once, after the last a), and the
// products psi_b conj(v_ab) of an element's four threads, neighbouring lanes, are summed
// by two exchanges that leave a quarter of the elements to each, which adds them to W_a.
// Any other tile adds its contributions output by output. Resident blocks walk the items
// as in F1: X values are loaded into registers one group of pairs (or item) ahead,
// orbital rows refill their places asynchronously, and the additions to W do not wait.
template <int L>
__global__ void __launch_bounds__(Sizes<L>::NT, Sizes<L>::RES3) k_fast_f3(const PairTile* __restrict__ tiles, int n_items, int glog,
                                                          const pk2* __restrict__ X,
                                                          const float2* __restrict__ tw_g, int reach) {
  grid_entry();
  using S = Sizes<L>;
  constexpr int M = S::M, MP = S::MP, QS = S::QS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(16) PairTile ring[3];
  pk2* tw = reinterpret_cast<pk2*>(smem_raw);
  float2* orb = reinterpret_cast<float2*>(smem_raw + S::tw_bytes);
  pk2* ex = reinterpret_cast<pk2*>(smem_raw + S::tw_bytes + S::orb_bytes);
  const int tid = threadIdx.x;
  const Walk<L> walk(n_items, glog);
  copy_tile(&ring[0], tiles + walk.tile(0), tid);
  if (walk.units > 1) copy_tile(&ring[1], tiles + walk.tile(1), tid);
  load_twiddles<L>(tw, tw_g, tid, S::NT);
  cp_async_wait_all();
  __syncthreads();
  load_orbitals<L>(orb, ring[0], 0, 2 * TT, (long)walk.rows(0) * (RR * L), tid);
  const int qa = tid % QB, n1 = (tid / QB) % M, rpa = tid / (QB * M);
  const int rpb = tid % RP, k2b = (tid / RP) % 8, qb = tid / (8 * RP);
  const bool second = rpa < RP;   // M < 8: the last threads only take part in the first step
  const unsigned live = live_mask<L>(k2b, reach);
  const pk2 zero = {f2(0.f), f2(0.f)};
  pk2 x[M];
  // X values of pairs p0.. of a unit into registers
  auto load_x = [&](int u, int p0, int np) {
    if (qb < QB && p0 + qb < np) {
      const pk2* src = X + (((long)walk.tile(u) * NPAIR + p0 + qb) * L + k2b) * (L * S::CP) + walk.rows(u) * RP + rpb;
#pragma unroll
      for (int k1 = 0; k1 < M; ++k1)
        x[k1] = live & (1u << k1) ? load_now(src + (long)k1 * 8 * L * S::CP) : zero;
    }
  };
  load_x(0, 0, ring[0].n_pairs);
  int cur = 0;
  bool was_full = false;
  for (int u = 0; u < walk.units; ++u) {
    // After a full item five groups are in flight: the right orbitals, 0, 1, 2, 3.
    const bool piped = was_full && full_tile(ring[cur]);
    if (piped) cp_async_wait<4>(); else cp_async_wait_all();
    __syncthreads();
    const int nxt = cur == 2 ? 0 : cur + 1, far = cur == 0 ? 2 : cur - 1;
    const PairTile& tl = ring[cur];
    const bool more = u + 1 < walk.units;
    const long noff = (long)walk.rows(u + 1) * (RR * L);
    if (u + 2 < walk.units) copy_tile(&ring[far], tiles + walk.tile(u + 2), tid);
    const int np = tl.n_pairs;
    const bool full = full_tile(tl);
    const long roff = (long)walk.rows(u) * (RR * L), aoff = roff + (long)2 * rpa * L + n1;
    if (np == 0 && more) {   // an empty tile
      load_x(u + 1, 0, ring[nxt].n_pairs);
      load_orbitals<L>(orb, ring[nxt], 0, 2 * TT, noff, tid);
    }
    pk2 b[8], wb[8];
    if (full && second) {
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) {
        b[n2] = orb_at<L>(orb, TT + qa, rpa, n1 + M * n2);
        wb[n2] = zero;
      }
    }
    for (int p0 = 0; p0 < np; p0 += QB) {
      if (qb < QB && p0 + qb < np) {
        pk_dft<M, true>(x);
        pk2* dst = ex + qb * QS + (k2b * RP + rpb) * MP;
        dst[0] = x[0];
#pragma unroll
        for (int m = 1; m < M; ++m) dst[m] = ptwiddle<true>(x[m], tw[k2b * MP + m]);
      }
      if (p0 + QB < np) load_x(u, p0 + QB, np);
      else if (more) load_x(u + 1, 0, ring[nxt].n_pairs);
      if (piped) {
        if (p0 == 0) cp_async_wait<3>(); else cp_async_wait<4>();
      }
      __syncthreads();
      if (p0 == 0) {
        if (full && more) load_orbitals<L>(orb, ring[nxt], TT, 2 * TT, noff, tid);
        cp_async_commit();
      }
      pk2* mine = ex + qa * QS + rpa * MP + n1;
      if (full) {
        if (second) {
          const int a = p0 / QB;
          pk2 v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = mine[q * RP * MP];
          pk_dft<8, true>(v);
#pragma unroll
          for (int n2 = 0; n2 < 8; ++n2) {
            const pk2 pa = orb_at<L>(orb, a, rpa, n1 + M * n2), y = v[n2];
            wb[n2].re = vminus(vfma(pa.re, y.re, wb[n2].re), vmul(pa.im, y.im));
            wb[n2].im = vfma(pa.im, y.re, vfma(pa.re, y.im, wb[n2].im));
            v[n2] = {vfma(b[n2].re, y.re, vmul(b[n2].im, y.im)), vdet(b[n2].im, y.re, b[n2].re, y.im)};
          }
          const bool lo1 = (qa & 1) == 0, lo2 = (qa & 2) == 0;
          pk2 s[4];
#pragma unroll
          for (int h = 0; h < 4; ++h)
            s[h] = padd(pk_select(lo1, v[h], v[4 + h]), pk_shfl_xor(pk_select(lo1, v[4 + h], v[h]), 1));
          const int n2a = 4 * (qa & 1) + (qa & 2);   // this thread's elements of W_a: n2a and n2a + 1
          float2* w = static_cast<float2*>(tl.out[a]) + aoff + M * n2a;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const pk2 r = padd(pk_select(lo2, s[h], s[2 + h]), pk_shfl_xor(pk_select(lo2, s[2 + h], s[h]), 2));
            if (tl.is_out[a]) add_rows<L>(w + M * h, r);
          }
        }
      } else {
        if (second && p0 + qa < np) {
          pk2 v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = mine[q * RP * MP];
          pk_dft<8, true>(v);
#pragma unroll
          for (int n2 = 0; n2 < 8; ++n2) mine[n2 * RP * MP] = v[n2];
        }
        __syncthreads();
        for (int o = 0; o < tl.n_orb; ++o) {
          if (!tl.is_out[o]) continue;
          for (int e = tid; e < RP * L; e += S::NT) {
            const int rp = e / L, n = e % L;
            pk2 s = zero;
            bool any = false;
            for (int c = 0; c < tl.out_n[o]; ++c) {
              const int p = tl.out_pair[o][c];
              if (p < p0 || p >= p0 + QB) continue;
              any = true;
              const pk2 y = ex[(p - p0) * QS + ((n / M) * RP + rp) * MP + n % M];
              const pk2 a = orb_at<L>(orb, tl.out_other[o][c], rp, n);
              if (tl.out_conj[o][c]) {
                s.re = vfma(a.im, y.im, vfma(a.re, y.re, s.re));
                s.im = vminus(vfma(a.im, y.re, s.im), vmul(a.re, y.im));
              } else {
                s.re = vminus(vfma(a.re, y.re, s.re), vmul(a.im, y.im));
                s.im = vfma(a.im, y.re, vfma(a.re, y.im, s.im));
              }
            }
            if (any) add_rows<L>(static_cast<float2*>(tl.out[o]) + roff + (long)2 * rp * L + n, s);
          }
        }
      }
      __syncthreads();
      if (more) {   // places of orbitals this item no longer reads
        if (full) load_orbitals<L>(orb, ring[nxt], p0 / QB, p0 / QB + 1, noff, tid);
        else if (p0 + QB >= np) load_orbitals<L>(orb, ring[nxt], 0, 2 * TT, noff, tid);
      }
      cp_async_commit();
    }
    if (full && second && tl.is_out[TT + qa]) {
      float2* w = static_cast<float2*>(tl.out[TT + qa]) + aoff;
#pragma unroll
      for (int n2 = 0; n2 < 8; ++n2) add_rows<L>(w + M * n2, wb[n2]);
    }
    cur = nxt;
    was_full = full;
  }
}

template <int L>
static cudaError_t launch_fast(const FockPlan& plan, const float* khat_t, void* scratch, const float2* tw,
                               cudaStream_t s) {
  using S = Sizes<L>;
  static std::atomic<unsigned long long> attr_done{0};
  if (const unsigned long long bit = device_bit_todo(attr_done)) {
    cudaError_t e = cudaFuncSetAttribute(k_fast_f1<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem13);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_fast_f3<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem13);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_fast_f2<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem2);
    if (e != cudaSuccess) return e;
    attr_done.fetch_or(bit, std::memory_order_release);
  }
  pk2* X = (pk2*)scratch;
  const float2* kt2 = reinterpret_cast<const float2*>(khat_t);
  const int reach = 2 * plan.g2_reach + 1 < L ? plan.g2_reach : L;
  const int n_live = reach >= L ? L : 2 * reach + 1;
  RowReach rows;
  const bool free0 = reach < L && 2 * plan.g0_reach[0] + 1 <= L;
  for (int k = 0; k <= kMaxLength / 2; ++k)
    rows.at[k] = (unsigned char)(free0 && k <= plan.g2_reach ? plan.g0_reach[k] : L);
  const int sms = sm_count();   // F1 and F3 run the blocks the chip holds at once
  const int glog = plan.group == 4 ? 2 : 0;
  for (int l = 0; l < plan.n_launch; ++l) {
    const PairTile* tiles = plan.d_tiles + plan.launch_first[l];
    const int nt = plan.launch_count[l], items = (nt >> glog) * S::RG;
    const unsigned g1 = (unsigned)std::min(items, S::RES1 * sms), g3 = (unsigned)std::min(items, S::RES3 * sms);
    launch(g1, S::NT, S::smem13, s)(k_fast_f1<L>, tiles, items, glog, X, tw, reach);
    dim3 g2((unsigned)n_live, (unsigned)(nt * NPAIR));
    launch(g2, S::NT2, S::smem2, s)(k_fast_f2<L>, X, tiles, kt2, tw, reach, rows, S::AHEAD2 ? S::MINB2 * sms : 0);
    launch(g3, S::NT, S::smem13, s)(k_fast_f3<L>, tiles, items, glog, X, tw, reach);
    launched(3);
  }
  return cudaGetLastError();
}

bool fock_fast_supported(Grid3 g) {
  return g.n0 == g.n1 && g.n1 == g.n2 && (g.n0 == 32 || g.n0 == 48 || g.n0 == 64 || g.n0 == 96);
}

// Paired tiles on the fast path once the orbitals and their sums (16 bytes a point) leave L2:
// four tiles of two pairs of blocks then read 16 orbitals' rows from memory instead of 32.
// The order depends on the system alone, so its sums are the same in a batch, for any
// tiles_per_launch and in the static entry. Grouped from six rounds of resident blocks on, where
// the last, partly filled one matters little (128 orbitals at 64^3: 18.98 -> 18.44 ms, 288
// at 96^3: 333.2 -> 331.1).
int fock_tile_order(Grid3 g, bool mixed, int n_occ, int tile, int tiles_per_launch, bool may_group) {
  if (!mixed || !fock_fast_supported(g) || 16.0 * g.N() * n_occ < 64e6) return TILE_ROUNDS;
  const long nb = (n_occ + tile - 1) / tile, meetings = std::min<long>((nb + 1) / 4, tiles_per_launch / 4);
  const int L = g.n0, res = L == 96 ? Sizes<96>::RES1 : Sizes<32>::RES1;
  return may_group && meetings * (L * (L / RR)) >= 6L * res * sm_count() ? TILE_GROUPED : TILE_PAIRED;
}

cudaError_t fock_pairs_fast(const FockPlan& plan, Grid3 g, const float* khat_t, void* scratch, const float2* tw_L,
                            cudaStream_t s) {
  switch (g.n0) {
    case 32: return launch_fast<32>(plan, khat_t, scratch, tw_L, s);
    case 48: return launch_fast<48>(plan, khat_t, scratch, tw_L, s);
    case 64: return launch_fast<64>(plan, khat_t, scratch, tw_L, s);
    case 96: return launch_fast<96>(plan, khat_t, scratch, tw_L, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pt
