// pair_tma.cuh -- two time steps of a periodic D2Q9 lattice in one pass over memory.
//
// The single-step update moves every population through HBM once per step and
// runs at the copy rate, so only fewer passes can make it faster.  Here a block
// owns a strip of at most X columns and a chunk of rows [ya, yb) and marches up
// the rows: the first step of row r is computed from a stage of the bulk-copy
// ring (the producer and window rules of k_step_tma, tma.cuh), its
// post-collision values stay on the chip, and the second step of row r - 1
// follows from rows r - 2, r - 1 and r.  Per pair of steps a node is read and
// written once.  What is computed twice is the first step of one node column
// on each side of a strip (one extra consumer warp, one lane of it) and of one
// row above and below a chunk.
//
// On-chip rows: the six planes with an x component go through shared memory
// (row slots of X + 8 elements, node j of the strip at j + 4).  A row of a plane with
// e_y = -1, 0, +1 is read 0, 1, 2 rows after it was written; with one block
// barrier per row a warp may be one row ahead of another, so these planes keep
// 2, 3 and 4 row slots.  The three planes without an x component stay in the
// registers of the thread that computes both steps of the column.
//
// Bound by HBM again at large sizes: 4096^2 FP32 takes 99 us a step (0.90 of the
// measured copy rate at 36 B per node and step) where the fastest single-step
// variant takes 183 us; the same with a ring of 3 or 4 stages, 107 us with
// strips of 256.
//
// Any row length from 32 bytes on: bulk copies move whole 16-byte words, so at a
// row end that is not a multiple of 16 bytes the wrapped nodes land `pad`
// elements further out than their column says (the padding of the row lies
// between), and the threads beside the ends read them there.
//
// Both steps run the collision of the single-step kernel in the same order and
// round the intermediate state to the storage type, so the results are the
// same bits as two single steps of the pipelined kernel (up to the sign of a zero those
// of the register kernels, which add a zero force where there is none).
//
// Every wait is bounded as in k_step_tma.  A warp whose wait ran out stays in
// the row loop and only arrives at the block barriers, so no warp is left
// waiting there.
#pragma once
#include "tma.cuh"

namespace lbm {

template <typename R>
struct PairArgs {
  Geo g;
  CoefV<R> c;
  const void* src;
  void* dst;
  unsigned int* flag;
  int* err;
  unsigned int step;  // index of the first of the two steps
  int stages;         // ring depth
  int sw;             // strip width: a multiple of 64, at most X
  int nstrips;        // ceil(nx / sw)
  int nchunks;        // row chunks per strip; grid = nstrips * nchunks
  long long timeout_ns;
  int extra_tx;  // test hook: extra bytes every stage waits for (never delivered)
};

// Consumer warps: X / 64 for the strip's node pairs (j, j + sw / 2), one for
// the two columns beside it.
template <int X>
struct PairShape {
  static constexpr int kMainWarps = X / 64;
  static constexpr int kConsumerWarps = kMainWarps + 1;
  static constexpr int kThreads = 32 * (1 + kConsumerWarps);
  static constexpr int kSlot = X + 8;
};

// Barriers, ring (rows of X elements and two 16-byte words on either side), and
// 2 (2 + 3 + 4) on-chip rows.
inline constexpr size_t pair_smem(int esize, int X, int stages) {
  return 128 * ((2 * (size_t)stages * 8 + 4 + 127) / 128) +
         (size_t)stages * 9 * (size_t)(X + 4 * (16 / esize)) * (size_t)esize +
         (size_t)18 * (size_t)(X + 8) * (size_t)esize;
}

// First of plane i's (|e_x| = 1) on-chip row slots, and their number.
template <class L>
constexpr int pair_depth(int i) {
  return 3 + L::cy(i);
}
template <class L>
constexpr int pair_slot0(int i) {
  int s = 0;
  for (int k = 0; k < i; ++k)
    if (L::cx(k) != 0) s += pair_depth<L>(k);
  return s;
}

// Stores a node pair: one aligned word where the two are neighbours.
template <class S, bool ADJ, typename T>
__device__ __forceinline__ void pair_put(T* p0, T* p1, bool act0, bool act1, bool apart, F2 v) {
  if constexpr (ADJ) {
    if (act1 && !apart) {
      *reinterpret_cast<uint32_t*>(p0) = S::enc2(v.x, v.y);
      return;
    }
  }
  if (act0) *p0 = S::enc(v.x);
  if (act1) *p1 = S::enc(v.y);
}

template <class L, int COLL, class S, bool FORCE, int XT>
__global__ void __launch_bounds__(PairShape<XT>::kThreads, XT == 512 ? 2 : 4) k_step_pair(PairArgs<typename S::R> a) {
  using T = typename S::T;
  using R = typename S::R;
  using Sh = PairShape<XT>;
  static_assert(L::Q == 9 && sizeof(T) <= 4, "D2Q9 with packed arithmetic");
  constexpr int HT = 16 / (int)sizeof(T);
  constexpr int HL = 2 * HT;  // slot[HL + j] holds node j of the strip
  constexpr int SLOT = XT + 2 * HL;
  // 16-bit storage: a thread's nodes are neighbours (2 ct, 2 ct + 1) and are stored
  // as one word; 32-bit storage: (ct, ct + sw / 2), as in k_step_tma
  constexpr bool ADJ = sizeof(T) == 2;
  extern __shared__ __align__(128) unsigned char smem[];
  const Geo& G = a.g;
  const int ST = a.stages;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);
  uint64_t* empty = full + ST;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + ST);
  T* ring = reinterpret_cast<T*>(smem + 128 * ((2 * ST * 8 + 4 + 127) / 128));
  T* mid = ring + ST * L::Q * SLOT;  // the on-chip rows

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) {
      mbar_init(smem_addr(full + s), 1);
      mbar_init(smem_addr(empty + s), Sh::kConsumerWarps);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T* src = static_cast<const T*>(chain_wait(a.src));
  T* dst = static_cast<T*>(a.dst);

  const int strip = blockIdx.x % a.nstrips, chunk = blockIdx.x / a.nstrips;
  const int x0 = strip * a.sw;
  const int w = min(a.sw, G.nx - x0);
  const int ya = (int)((long long)G.ny * chunk / a.nchunks);
  const int yb = (int)((long long)G.ny * (chunk + 1) / a.nchunks);
  const int nrows = yb - ya + 2;  // first-step rows ya - 1 .. yb

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    const int nxr = (G.nx + HT - 1) / HT * HT;  // row end, whole words (within the pitch)
    const bool lwrap = x0 == 0, rwrap = x0 + w == G.nx;
    const int lo = lwrap ? 0 : x0 - HT, hi = rwrap ? nxr : x0 + w + HT;
    const uint32_t main_bytes = (uint32_t)(hi - lo) * sizeof(T);
    constexpr uint32_t word = (uint32_t)HT * sizeof(T);
    const uint32_t row_bytes = main_bytes + (lwrap ? 2 * word : 0u) + (rwrap ? word : 0u);
    int ey = 0;
#pragma unroll
    for (int k = 0; k < L::Q; ++k)
      if (k == lane) ey = L::cy(k);
    int y = ya - 1 - ey;  // source row of this lane's plane
    if (y < 0) y += G.ny;
    if (y < 0) y += G.ny;  // (ny == 1: two rows below row 0)
    if (y >= G.ny) y -= G.ny;
    int k = 0, s = 0;
    uint32_t u = 0;
    bool ok = true;
    for (; k < nrows; ++k) {
      if (u > 0 && !mbar_wait_warp(smem_addr(empty + s), (u - 1) & 1u, abort_flag, a.err,
                                   a.timeout_ns)) {
        ok = false;
        break;
      }
      const uint32_t fb = smem_addr(full + s);
      if (lane == 0) mbar_arrive_expect_tx(fb, row_bytes * L::Q + (uint32_t)a.extra_tx);
      __syncwarp();
      if (lane < L::Q) {
        T* slot = ring + (s * L::Q + lane) * SLOT + HL;
        const T* rowp = src + lane * G.plane + (long long)y * G.pitch;
        bulk_g2s(smem_addr(slot + (lo - x0)), rowp + lo, main_bytes, fb);
        if (lwrap) bulk_g2s(smem_addr(slot - HL), rowp + nxr - HL, 2 * word, fb);
        if (rwrap) bulk_g2s(smem_addr(slot + (nxr - x0)), rowp, word, fb);
      }
      if (++y == G.ny) y = 0;
      if (++s == ST) {
        s = 0;
        ++u;
      }
    }
    if (!ok && lane == 0) {
      // let every issued copy land before the block's shared memory is released
      for (int kk = (k > ST ? k - ST : 0); kk < k; ++kk)
        mbar_wait(smem_addr(full + kk % ST), (uint32_t)((kk / ST) & 1), abort_flag, a.err,
                  a.timeout_ns, false);
    }
    return;
  }

  // -------------------------------------------------------------- consumers
  const bool edge = warp == Sh::kConsumerWarps;  // the columns x0 - 1 and x0 + w
  const int ct = threadIdx.x - 32;
  const int nmain = a.sw >> 1;  // threads with a node pair of a full strip
  const int j0 = edge ? -1 : (ADJ ? 2 * ct : ct), j1 = edge ? w : (ADJ ? 2 * ct + 1 : ct + nmain);
  const bool act0 = edge ? lane == 0 : ct < nmain && j0 < w;
  const bool act1 = edge ? lane == 0 : ct < nmain && j1 < w;
  const bool idle = __all_sync(0xffffffffu, !act0);
  // Where node j - 1, j, j + 1 of this thread's nodes (0 for lanes without one) lie
  // in a ring row: a wrapped node lies behind the row's padding.
  const int pad = (HT - G.nx % HT) % HT;
  const int padl = x0 == 0 ? pad : 0, padr = x0 + w == G.nx ? pad : 0;
  const auto pos = [&](int j) { return HL + j - (j < 0 ? padl : 0) + (j >= w ? padr : 0); };
  const int n0 = act0 ? j0 : 0, n1 = act1 ? j1 : 0;
  const T* st0[3] = {ring + pos(n0 + 1), ring + pos(n0), ring + pos(n0 - 1)};  // index 1 + e_x
  const T* st1[3] = {ring + pos(n1 + 1), ring + pos(n1), ring + pos(n1 - 1)};
  T* m0 = mid + 4 + n0;
  T* m1 = mid + 4 + n1;
  int s = 0;
  uint32_t u = 0;
  int r2 = 0, r3 = 0, r4 = 0;  // current row slot of the planes with e_y = -1, 0, +1
  bool dead = false;
  F2 rest1 = {0.f, 0.f}, up1 = {0.f, 0.f}, up2 = {0.f, 0.f};  // rest: previous row; e = (0, 1): two rows
  long long own = (long long)(ya - 1) * G.pitch + x0;         // row r - 1 at k = 1: ya - 1 + k - 1
  for (int k = 0; k < nrows; ++k) {
    const unsigned int so = (unsigned)s * (L::Q * SLOT);
    if (!dead && !mbar_wait_warp(smem_addr(full + s), u & 1u, abort_flag, a.err, a.timeout_ns)) dead = true;
    F2 g[L::Q];
    F2 dn = {0.f, 0.f}, rest0 = {0.f, 0.f}, up0 = {0.f, 0.f};
    if (!dead) {
      if (!idle) {
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
          g[i] = F2{S::dec(st0[1 + L::cx(i)][so + i * SLOT]), S::dec(st1[1 + L::cx(i)][so + i * SLOT])};
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_addr(empty + s));
      if (!idle) {
        const unsigned bad = collide_v<L, COLL, FORCE, F2>(g, a.c);
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
          if (L::cx(i) == 0) continue;
          const int row = pair_slot0<L>(i) + (L::cy(i) == 0 ? r3 : (L::cy(i) < 0 ? r2 : r4));
          pair_put<S, ADJ>(m0 + row * Sh::kSlot, m1 + row * Sh::kSlot, act0, act1, edge, g[i]);
        }
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
          if (L::cx(i) != 0) continue;
          const F2 v = F2{S::dec(S::enc(g[i].x)), S::dec(S::enc(g[i].y))};
          if (L::cy(i) == 0) rest0 = v;
          else if (L::cy(i) > 0) up0 = v;
          else dn = v;
        }
        record_bad(a.flag, a.step, (act0 && (bad & 1u)) || (act1 && (bad & 2u)));
      }
    }
    if (++s == ST) {
      s = 0;
      ++u;
    }
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(32 * Sh::kConsumerWarps) : "memory");
    if (k >= 2 && !dead && !idle && !edge) {
      // second step of row ya + k - 2: planes with e_y = -1 come from the row
      // just written, 0 from the one before, +1 from the one before that
      const int p3 = r3 == 0 ? 2 : r3 - 1, p4 = (r4 + 2) & 3;
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        if (L::cx(i) == 0) {
          g[i] = L::cy(i) == 0 ? rest1 : (L::cy(i) > 0 ? up2 : dn);
        } else {
          const int row = pair_slot0<L>(i) + (L::cy(i) == 0 ? p3 : (L::cy(i) < 0 ? r2 : p4));
          g[i] = F2{S::dec(m0[row * Sh::kSlot - L::cx(i)]), S::dec(m1[row * Sh::kSlot - L::cx(i)])};
        }
      }
      const unsigned bad = collide_v<L, COLL, FORCE, F2>(g, a.c);
      T* op = dst + own;
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        pair_put<S, ADJ>(op + n0, op + n1, act0, act1, false, g[i]);
        op += G.plane;
      }
      record_bad(a.flag, a.step + 1, (act0 && (bad & 1u)) || (act1 && (bad & 2u)));
    }
    if (k >= 1) own += G.pitch;
    rest1 = rest0;
    up2 = up1;
    up1 = up0;
    r2 ^= 1;
    r3 = r3 == 2 ? 0 : r3 + 1;
    r4 = (r4 + 1) & 3;
  }
}

}  // namespace lbm
