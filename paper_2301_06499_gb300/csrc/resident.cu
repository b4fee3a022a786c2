// The whole round loop of a propagation in one cooperative launch (rows of up
// to 8 words, gathered whole; one graph or a packed batch; PROPAGATE-P, or
// PROPAGATE-S passes as words).
//
// What bounded it: a round of a small or sparse graph moves little, so its
// time was launches (two or three kernels and an iteration of the captured
// loop), ramp-up, and chains of dependent loads: about 20 us for 1,000 nodes
// and 40 us for a round of the 1024^2 grid (s = 128) whose traffic is worth
// 5-6 us of L2. Here a round is one pass over its work and one grid barrier.
//
// A round in one pass. X[v] holds everything v has been sent so far, also
// what this round has added; a round only ever sends the deltas of the round
// before (D of t-1), so it still sees none of its own updates (the
// synchronous diffusion of Alg. 1). Whoever adds bits to X[v] learns which
// of them are new: a row swept whole has one owner, everything else adds with
// a 64-bit atomicOr and compares with the old word. So each new pair (seed,
// node) has exactly one finder, which counts it (the collision count of
// round t), records it in D of round t and, first on that row, appends the
// row to F_t. Nothing is left for a second kernel: the signatures are synced,
// a block's counts leave it while the next round starts, and three delta
// buffers take turns (t-1 read, t written, t-2 cleared through F_{t-2}).
//
// m_active (the in-degrees of the rows round t revisits: a zero bit left at
// its start and a changed in-neighbour): a row that reads full was either
// full before the round, or was filled in this round by a finder that saw it
// not full and claimed it. So testing the running X and claiming once per
// round counts exactly the active rows.
//
// Sparse rounds push: a lane per frontier row (rows of more than kBigRow
// out-arcs in pieces of kBigPiece, a warp each) reads its out-neighbours'
// signatures first and sends an atomic only for bits they lack; on a grid
// half of the sends carry nothing new. Dense rounds sweep the sliced-ELL copy
// as k_pull does, with its early stop.
//
// Measured per call, round by round (with dense rounds that stop early) and
// here (a range: by the seeds drawn): ER 10^3 (s = 64) 215 -> 94 us, ER 10^4
// (s = 64) 288 -> 135 us, 1024^2 grid (s = 128, ~2,050 rounds) 83 -> 37.5 ms,
// R-MAT 22 (s = 256) 2.23 -> 1.5 to 1.7 ms, R-MAT 26 (s = 512) 54.9 -> 43 to
// 50 ms, 30 packed graphs 33.6 -> 16.4 ms. What bounds it now: a round of
// little work is five dependent accesses, two block-wide steps and the barrier,
// 6 to 7 us; heavy pushes the L2's atomics (25 to 28 per ns on spread addresses:
// the grid sends 0.98 G of them in 34.5 ms), which is why marks are loaded before
// they are set; heavy sweeps the gathers that a thread's registers hold in
// flight.
//
// The blocks are co-resident by the cooperative launch. Every wait at the barrier
// is bounded; on expiry the call returns PG_ETIMEOUT. A launch holds its SMs: it
// ends early, to go on in another, when other propagations want a part of them
// and every 20 ms (should_yield, share.cpp).
#include "kernels.cuh"

namespace pg {

namespace {

constexpr int kBigRow = kResidentRow;
constexpr int kBigPiece = kResidentPiece;
constexpr int kMaxThreads = kResidentThreads;
constexpr int kStage = 256;      // staged frontier rows per warp

// Loads of data that other blocks write in this launch (never the read-only
// path): coherent after the barrier's fence; within a round a stale
// signature only costs an atomic that finds nothing.
__device__ __forceinline__ void ld_256(uint64_t *a, const uint64_t *p) {
  asm volatile("ld.global.L1::no_allocate.v4.u64 {%0, %1, %2, %3}, [%4];"
               : "=l"(a[0]), "=l"(a[1]), "=l"(a[2]), "=l"(a[3])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void ld_128(uint64_t *a, const uint64_t *p) {
  asm volatile("ld.global.L1::no_allocate.v2.u64 {%0, %1}, [%2];"
               : "=l"(a[0]), "=l"(a[1])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void ld_64(uint64_t *a, const uint64_t *p) {
  asm volatile("ld.global.L1::no_allocate.u64 %0, [%1];" : "=l"(a[0]) : "l"(p) : "memory");
}
template <int CW>
__device__ __forceinline__ void ld_row(uint64_t (&a)[CW], const uint64_t *p) {
  if constexpr (CW == 1) {
    ld_64(a, p);
  } else if constexpr (CW == 2) {
    ld_128(a, p);
  } else {
#pragma unroll
    for (int k = 0; k < CW; k += 4) ld_256(a + k, p + k);
  }
}

__device__ __forceinline__ uint32_t ld_u32(const uint32_t *p) {
  return *((volatile const uint32_t *)p);
}
// Row marks of a round, two bits a row: claimed (counted in m_active) and
// changed (in F_t). One atomic sets and tells both.
constexpr uint32_t kClaimed = 1u, kChanged = 2u;
// (mark_word: the row's whole word, so that several can be under way.)
__device__ __forceinline__ uint32_t mark_word(uint32_t *M, int64_t v, uint32_t bits) {
  return atomicOr(M + (v >> 4), bits << ((v & 15) * 2));
}
__device__ __forceinline__ uint32_t mark(uint32_t *M, int64_t v, uint32_t bits) {
  return mark_word(M, v, bits) >> ((v & 15) * 2);
}
__device__ __forceinline__ bool changed(const uint32_t *M, int64_t v) {
  return ((M[v >> 4] >> ((v & 15) * 2)) & kChanged) != 0u;
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(uint32_t *p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" : : "l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void red_or(uint64_t *p, uint64_t v) {
  asm volatile("red.global.or.b64 [%0], %1;" : : "l"(p), "l"(v) : "memory");
}

// Per-block state: the staged rows' totals of each warp, the round's counters.
struct Shared {
  unsigned long long od, ne;  // out-arcs and pieces of the block's staged rows
  unsigned long long base_f, base_e;
  unsigned long long mact, work;
  uint32_t rows, staged;
  uint64_t alive[kAliveWords];
  uint16_t col[kResidentSorted];   // count column of each bit (p.sort_seeds)
  uint16_t place[kResidentSorted]; // bit of each seed
  unsigned long long fp, ne_all;
  unsigned long long sums[3];
  int rows_out;  // count rows to hand over at the fixpoint, else -1
  uint32_t bar;  // barriers this block has arrived at
  int last;      // this block arrived last
  unsigned long long yield;
  long long t0;    // launch time, in cycles
  long long look;  // when its part of the SMs is looked at next, since then
  int failed;    // the barrier gave up
};

// Per-thread state of one round.
struct Lane {
  int lane, wid;         // within the warp, warp within the block
  int64_t warp, nwarps;  // across the grid, neighbours on different SMs
  int64_t tid, nth;
  int t, cur;            // round, its delta buffer
  const uint64_t *Dp;    // deltas of round t-1
  uint64_t *Dc;          // deltas of round t
  const uint32_t *Mp;    // marks of round t-1
  uint32_t *Mc;          // marks of round t
  uint32_t *Kc;          // passes as words: claim bytes of round t
  int32_t *F;            // F_t
  unsigned long long *E; // pieces of F_t's long rows
  uint32_t cs;           // counters of this round: shared-memory address,
  uint32_t *cg;          // or (cs = 0) the counts row
  int32_t *stage;
  int scnt;
  bool pieces;           // append E_t (a round that may be followed by a push)
  unsigned long long od, ne;  // out-arcs and pieces of the rows staged by this lane
  int gcur;                   // a packed batch: graph and out-arcs not yet added to its sum
  unsigned long long gacc;
  unsigned long long mact, work;
  uint32_t rows;
  // over the whole launch
  uint32_t scan, gath, items;
};

__device__ __forceinline__ uint64_t *delta_buf(const Params &p, int k) {
  return k == 0 ? p.D0 : k == 1 ? p.D1 : p.D2;
}
__device__ __forceinline__ uint32_t *mark_buf(const Params &p, int k) {
  return k == 0 ? p.C0 : k == 1 ? p.C1 : p.C2;
}
__device__ __forceinline__ int32_t *frontier_buf(const Params &p, int k) {
  return k == 0 ? p.F0 : k == 1 ? p.F1 : p.F2;
}

// Whether the launch should end after this round, to be launched again where it
// stopped (run_resident): when other propagations came and its part of the SMs
// is smaller, or they left and it is larger by half, but not at once: a call
// soon over is waited for (ending a launch and starting another takes about
// 50 us), and a larger part is worth that only for a long one. And when it has
// held its SMs for a slice, so that other work on the device gets in between.
// Times in cycles of the SM that asks, about 2 to the nanosecond: reading the
// device's timer takes longer. The host's memory is looked at every 50 us, not in
// every round, which would be a wait for the link in every round. A call that
// has the device to itself pays 0.4% for all this on a 85^2 grid of short rounds
// (s = 31, 1,117 against 1,113 us), where it paid 1.1% with a look in every round
// and the answer read behind the round's other conditions.
constexpr long long kShrinkCycles = 200 * 1000;
constexpr long long kGrowCycles = 4 * 1000 * 1000;
constexpr long long kLookCycles = 100 * 1000;

__device__ __forceinline__ bool should_yield(const Params &p, Shared &sh) {
  const long long ran = clock64() - sh.t0;
  if (ran < sh.look) return false;
  sh.look = min(ran + kLookCycles, p.slice_cycles + 1);
  const int want = *(volatile int32_t *)&p.out->want, have = (int)gridDim.x;
  return ran > p.slice_cycles || (want > 0 && want < have) ||
         (2 * want >= 3 * have && ran > kGrowCycles);
}

// Waits until *word, counting up, reaches target (modulo 2^32). A block that
// gives up leaves the launch. One that arrives after that finds the word
// reached and goes on to its next barrier, where it gives up too; after the
// launch's last barrier it runs to the end. So no block's own end says that the
// launch was whole: only all of them, counted at the exit, do.
__device__ __forceinline__ bool wait_for(const Params &p, const uint32_t *word, uint32_t target) {
  ResidentCtl *rc = p.rctl;
  unsigned long long t0 = 0;
  for (int spin = 0; (int32_t)(ld_acquire(word) - target) < 0; ++spin) {
    if ((spin & 255) == 255) {
      const unsigned long long t = now_ns();
      if (!t0) t0 = t;
      if (ld_acquire(&rc->abort) || t - t0 > p.barrier_ns) {
        st_release(&rc->abort, 1u);
        return false;
      }
    }
  }
  return true;
}

// Grid barrier number sh.bar of the launch. Blocks count up one word and wait
// for it to reach the next multiple of the grid: no answer to wait for before
// the word can be polled, no release by a last block (about 1.2 us less a
// round than an arrival counter with a generation word). With a finalizer (a
// packed batch) the block that arrives last runs it and then releases the
// others. Returns false once any block gave up.
template <bool SEG, class Fin>
__device__ __forceinline__ bool grid_barrier(const Params &p, Shared &sh, Fin fin) {
  ResidentCtl *rc = p.rctl;
  __syncthreads();
  if constexpr (SEG) {
    if (threadIdx.x == 0) {
      ++sh.bar;
      __threadfence();
      sh.last = atomicAdd(&rc->arrive, 1u) + 1u == sh.bar * gridDim.x;
    }
    __syncthreads();
    if (sh.last) {
      __threadfence();
      fin();
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      sh.failed = 0;
      if (sh.last) {
        __threadfence();
        st_release(&rc->gen, sh.bar);
      } else {
        sh.failed = !wait_for(p, &rc->gen, sh.bar);
      }
      __threadfence();
    }
  } else if (threadIdx.x == 0) {
    ++sh.bar;
    __threadfence();
    atomicAdd(&rc->arrive, 1u);
    sh.failed = !wait_for(p, &rc->arrive, sh.bar * gridDim.x);
    __threadfence();
  }
  __syncthreads();
  return !sh.failed;
}

// A row staged by this lane: its out-arcs (od), for the choice of the next
// round, and its pieces; in a packed batch, for its graph g's own choice.
template <bool SEG>
__device__ __forceinline__ void stage_degree(const Params &p, Lane &L, uint32_t od, int g) {
  L.od += od;
  if (od > kBigRow) L.ne += (od + kBigPiece - 1) / kBigPiece;
  if (SEG && od) {
    if (g != L.gcur) {
      if (L.gacc) atomicAdd(p.gfsum + (size_t)L.cur * (size_t)p.nseg + L.gcur, L.gacc);
      L.gcur = g;
      L.gacc = 0;
    }
    L.gacc += od;
  }
}

// Out-arcs and pieces of the warp's staged rows (and, in a packed batch,
// their graphs' frontier sums).
template <bool SEG>
__device__ __forceinline__ void stage_totals(const Params &p, Lane &L, unsigned long long &od_t,
                                             unsigned long long &ne_t) {
  __syncwarp();
  if constexpr (SEG) {  // one atomic per warp when its lanes ended on one graph
    unsigned long long *gf = p.gfsum + (size_t)L.cur * (size_t)p.nseg;
    const unsigned has = __ballot_sync(kFullMask, L.gacc != 0);
    if (has) {
      const int g0 = __shfl_sync(kFullMask, L.gcur, __ffs(has) - 1);
      if (__all_sync(kFullMask, L.gacc == 0 || L.gcur == g0)) {
        unsigned long long tot;
        warp_excl_scan64(L.gacc, L.lane, &tot);
        if (L.lane == 0) atomicAdd(gf + g0, tot);
      } else if (L.gacc) {
        atomicAdd(gf + L.gcur, L.gacc);
      }
    }
    L.gacc = 0;
  }
  od_t = L.od;
  ne_t = L.pieces ? L.ne : 0ULL;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    od_t += __shfl_xor_sync(kFullMask, od_t, off);
    ne_t += __shfl_xor_sync(kFullMask, ne_t, off);
  }
  L.od = L.ne = 0;
}

// Writes the warp's staged rows at F[bf] and their pieces at E[be].
__device__ __forceinline__ void stage_write(const Params &p, const Lane &L, unsigned long long bf,
                                            unsigned long long be, unsigned long long ne_t) {
  for (int i = L.lane; i < L.scnt; i += 32) L.F[bf + i] = L.stage[i];
  if (!ne_t) return;
  for (int j0 = 0; j0 < L.scnt; j0 += 32) {
    const int i = j0 + L.lane;
    int32_t v = 0;
    unsigned long long ne = 0;
    if (i < L.scnt) {
      v = L.stage[i];
      const unsigned long long od =
          (unsigned long long)(__ldg(p.out_ptr + v + 1) - __ldg(p.out_ptr + v));
      if (od > kBigRow) ne = (od + kBigPiece - 1) / kBigPiece;
    }
    unsigned long long tot;
    const unsigned long long ex = warp_excl_scan64(ne, L.lane, &tot);
    if (tot) write_pieces(L.E, be + ex, v, ne, L.lane);
    be += tot;
  }
}

// A full stage in the middle of a round: the warp reserves its own places.
template <bool SEG>
__device__ __forceinline__ void stage_spill(const Params &p, Lane &L) {
  unsigned long long od_t, ne_t, bf = 0, be = 0;
  stage_totals<SEG>(p, L, od_t, ne_t);
  if (L.lane == 0) {
    bf = atomicAdd(&p.rctl->fp[L.cur], ((unsigned long long)L.scnt << kFsumBits) + od_t);
    if (ne_t) be = atomicAdd(&p.rctl->next[L.cur].ne, ne_t);
  }
  bf = __shfl_sync(kFullMask, bf, 0) >> kFsumBits;
  be = __shfl_sync(kFullMask, be, 0);
  stage_write(p, L, bf, be, ne_t);
  __syncwarp();
  L.scnt = 0;
}

__device__ __forceinline__ void stage_row(Lane &L, int32_t v, bool app) {
  const unsigned mask = __ballot_sync(kFullMask, app);
  if (app) L.stage[L.scnt + __popc(mask & ((1u << L.lane) - 1u))] = v;
  L.scnt += __popc(mask);
}

// The end of a round's work: the block's staged rows with one reservation for
// all its warps (a warp each would queue at the counters: same-address
// atomics take about 0.65 ns each), its counts and work sums.
template <bool PW, bool SEG>
__device__ __forceinline__ void round_flush(const Params &p, Lane &L, Shared &sh, uint32_t *scnt_s) {
  unsigned long long od_t = 0, ne_t = 0;
  if (L.scnt) stage_totals<SEG>(p, L, od_t, ne_t);
  if (__any_sync(kFullMask, L.rows != 0u)) {
    unsigned long long m = L.mact, w = L.work;
    uint32_t r = __reduce_add_sync(kFullMask, L.rows);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m += __shfl_xor_sync(kFullMask, m, off);
    if (PW || SEG) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) w += __shfl_xor_sync(kFullMask, w, off);
    } else {
      w = m * (unsigned long long)p.s;
    }
    if (L.lane == 0) {
      atomicAdd(&sh.mact, m);
      atomicAdd(&sh.work, w);
      atomicAdd(&sh.rows, r);
    }
  }
  uint32_t at = 0;
  unsigned long long ae = 0;
  if (L.lane == 0 && L.scnt) {  // the warp's place among the block's rows
    at = atomicAdd(&sh.staged, (uint32_t)L.scnt);
    atomicAdd(&sh.od, od_t);
    if (ne_t) ae = atomicAdd(&sh.ne, ne_t);
  }
  at = __shfl_sync(kFullMask, at, 0);
  ae = __shfl_sync(kFullMask, ae, 0);
  __syncthreads();
  RoundStats *rs = p.rs + (L.t - p.row_base);
  if (threadIdx.x == 0) {  // one reservation for the block
    unsigned long long bf = 0, be = 0;
    if (sh.staged) bf = atomicAdd(&p.rctl->fp[L.cur], ((unsigned long long)sh.staged << kFsumBits) + sh.od);
    if (sh.ne) be = atomicAdd(&p.rctl->next[L.cur].ne, sh.ne);
    if (sh.rows) {
      atomicAdd(&rs->m_active, sh.mact);
      atomicAdd(&rs->work, sh.work);
      atomicAdd(&rs->rows, (unsigned long long)sh.rows);
    }
    sh.base_f = bf >> kFsumBits;
    sh.base_e = be;
    sh.mact = sh.work = sh.od = sh.ne = 0;
    sh.rows = sh.staged = 0;
  }
  if (!SEG && p.early_stop) {  // the seeds that gained a pair
    for (int w = L.wid; w * 64 < p.ncols; w += blockDim.x >> 5) {
      const int i = w * 64 + L.lane;
      const unsigned lo = __ballot_sync(kFullMask, i < p.ncols && scnt_s[i] != 0u);
      const unsigned hi = __ballot_sync(kFullMask, i + 32 < p.ncols && scnt_s[i + 32] != 0u);
      if (L.lane == 0 && (lo | hi)) atomicOr(&p.rctl->alive[L.cur][w], ((unsigned long long)hi << 32) | lo);
    }
  }
  __syncthreads();
  if (L.scnt) stage_write(p, L, sh.base_f + at, sh.base_e + ae, ne_t);
  L.scnt = 0;
  L.mact = L.work = 0;
  L.rows = 0;
}

__device__ __forceinline__ void count_add(const Lane &L, int col, uint32_t x) {
  if (L.cs)
    asm volatile("red.shared.add.u32 [%0], %1;" : : "r"(L.cs + 4u * (uint32_t)col), "r"(x) : "memory");
  else
    atomicAdd(L.cg + col, x);
}

// Counts the bits of each lane's nw (word k of a row whose count columns
// start at c0): one bit per finder, a handful per row in a sparse round.
__device__ __forceinline__ void count_bits(const Lane &L, int c0, int k, uint64_t nw) {
  while (nw) {
    const int b = __ffsll((long long)nw) - 1;
    nw &= nw - 1;
    count_add(L, c0 + k * 64 + b, 1u);
  }
}

// Claims row v for the passes (bits) of mask that no one claimed in this
// round; returns those newly claimed. One byte per row.
__device__ __forceinline__ uint32_t claim_passes(uint32_t *Kb, int64_t v, uint32_t mask) {
  uint32_t *w = Kb + (v >> 2);
  const int sh = (int)(v & 3) * 8;
  uint32_t have = (ld_u32(w) >> sh) & 0xFFu;
  mask &= ~have;
  if (!mask) return 0u;
  have = (atomicOr(w, mask << sh) >> sh) & 0xFFu;
  return mask & ~have;
}

// ------------------------------------------------------------ sparse rounds
// A lane takes four out-arcs of a frontier row together: their loads, then
// their signature atomics, then their marks are under way at once, so that a
// row of four arcs costs five dependent accesses, not five per arc. Of a row's
// words only the pairs with new bits are sent, one pair after another: a
// sparse round's delta holds a bit or two, and rows of 8 words then cost what
// rows of 2 do. (Four lanes a row, two words each, took 9.6 ms for 105 M hub
// arcs of R-MAT 26 at s = 512 and 2.5 ms for its 10 M short rows.)
template <int CW, bool PW, bool SEG>
__device__ __forceinline__ void push_round(const Params &p, Lane &L, const int32_t *Fp,
                                           const unsigned long long *Ep, int64_t nF, int64_t nE) {
  constexpr int UNR = 4;                // out-arcs a lane handles together
  constexpr int WL = CW <= 2 ? CW : 2;  // words sent together
  constexpr int PAIRS = CW / WL;
  // a small frontier spreads each row's arcs over more lanes, so that its
  // rows of up to kBigRow arcs take one step
  int gl = 0;  // log2 of the lanes per row
  while (gl < 3 && (nF << (gl + 1)) <= L.nth) ++gl;
  const int rows = 32 >> gl;  // rows per warp
  const int64_t groups = (nF + rows - 1) / rows;
  const unsigned long long *gfp =
      SEG ? p.gfsum + (size_t)((L.t + 2) % 3) * (size_t)p.nseg : nullptr;
  // a degree is wanted once per claimed row. Up to 2^22 rows (16 MB of degrees,
  // which stay in L2 beside the signatures a round touches) it is fetched with the
  // signature, above after the claim: on R-MAT 26 (268 MB of them) one access in
  // eight on the hub rows. Where between the two it turns was not measured.
  const bool deg_now = p.n <= (1 << 22);
  // row and arcs of an item: fetched for the next item ahead of this one's work
  auto item = [&](int64_t it, int32_t &u, int64_t &ob, int64_t &oe) {
    u = -1;
    ob = oe = 0;
    if (it < groups) {
      const int64_t i = it * rows + (L.lane >> gl);
      if (i < nF) {
        u = Fp[i];
        ob = __ldg(p.out_ptr + u);
        oe = __ldg(p.out_ptr + u + 1);
        if (oe - ob > kBigRow) oe = ob;  // in pieces, below
        ob += L.lane & ((1 << gl) - 1);
      }
    } else if (it < groups + nE) {
      const unsigned long long e = Ep[it - groups];
      u = (int32_t)(e >> 32);
      const int64_t b0 = __ldg(p.out_ptr + u) + (int64_t)(e & 0xFFFFFFFFULL) * kBigPiece;
      oe = min(__ldg(p.out_ptr + u + 1), b0 + kBigPiece);
      ob = b0 + L.lane;
    }
  };
  int32_t u_next;
  int64_t ob_next, oe_next;
  item(L.warp, u_next, ob_next, oe_next);
  for (int64_t it = L.warp; it < groups + nE; it += L.nwarps) {
    const int32_t u = u_next;
    int64_t ob = ob_next, oe = oe_next;
    const bool piece = it >= groups;  // 32 lanes on one long row: the same delta
    const int stride = piece ? 32 : 1 << gl;
    item(it + L.nwarps, u_next, ob_next, oe_next);
    int gs = p.s, c0 = 0, g = 0;
    unsigned long long *gm = nullptr;
    if (SEG && u >= 0) {
      g = __ldg(p.node_graph + u);
      // a packed batch: graphs swept whole in this round take no push
      if (gfp[g] > __ldg(p.gthr + g)) oe = ob;
      gs = __ldg(p.graph_s + g);
      c0 = __ldg(p.graph_col0 + g);
      if (p.gmact) gm = p.gmact + (size_t)(L.t - p.row_base) * (size_t)p.nseg + g;
    }
    uint64_t d[CW];
#pragma unroll
    for (int k = 0; k < CW; ++k) d[k] = 0ULL;
    if (ob < oe && gather_ok(p, u, CW - 1)) {
      ld_row<CW>(d, L.Dp + (size_t)u * CW);
      ++L.items;
      ++L.gath;
    }
    uint32_t pairs = 0;  // the pairs of words with new bits
#pragma unroll
    for (int j = 0; j < PAIRS; ++j) {
      uint64_t any = 0;
#pragma unroll
      for (int k = 0; k < WL; ++k) any |= d[j * WL + k];
      if (any) pairs |= 1u << j;
    }
    while (__any_sync(kFullMask, ob < oe)) {
      int32_t v[UNR];
      uint32_t deg[UNR], mk[UNR];
      if (stride == 1 && p.col_quads && (ob & ~3LL) + 8 <= p.m) {
        // a row's next four arcs: the two 16-byte quads that hold them
        int4 lo = make_int4(-1, -1, -1, -1), hi = lo;
        if (ob < oe) {
          const int4 *c4 = reinterpret_cast<const int4 *>(p.out_col) + (ob >> 2);
          lo = __ldg(c4);
          if (((ob & 3) + (oe - ob)) > 4) hi = __ldg(c4 + 1);
        }
        if (ob & 1) lo.x = lo.y, lo.y = lo.z, lo.z = lo.w, lo.w = hi.x, hi.x = hi.y, hi.y = hi.z;
        if (ob & 2) lo.x = lo.z, lo.y = lo.w, lo.z = hi.x, lo.w = hi.y;
        v[0] = lo.x, v[1] = lo.y, v[2] = lo.z, v[3] = lo.w;
#pragma unroll
        for (int q = 0; q < UNR; ++q)
          if (ob + q >= oe) v[q] = -1;
      } else {
#pragma unroll
        for (int q = 0; q < UNR; ++q) {
          const int64_t j = ob + (int64_t)q * stride;
          v[q] = j < oe ? __ldg(p.out_col + j) : -1;
        }
      }
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
        if (v[q] >= 0 && !gather_ok(p, v[q], CW - 1)) v[q] = -1;
        deg[q] = 0;
        mk[q] = ~0u;
        if (v[q] >= 0) {
          ++L.scan;
          mk[q] = ld_u32(L.Mc + (v[q] >> 4));  // an atomic only for a mark not seen set
          if (deg_now) deg[q] = p.deg_in[v[q]];
        }
      }
      uint32_t gain = 0, room = 0;  // by arc; PW: room by arc and word
      uint32_t left = pairs;
      do {
        const int j = left ? __ffs(left) - 1 : 0;
        const bool on = left != 0u;
        left &= left - 1;
        const int w0 = j * WL;
        uint64_t dj[WL], x[UNR][WL], old[UNR][WL];
#pragma unroll
        for (int k = 0; k < WL; ++k) {
          dj[k] = d[k];
#pragma unroll
          for (int i = 1; i < PAIRS; ++i)
            if (j == i) dj[k] = d[i * WL + k];
        }
#pragma unroll
        for (int q = 0; q < UNR; ++q) {
#pragma unroll
          for (int k = 0; k < WL; ++k) x[q][k] = ~0ULL;
          if (on && v[q] >= 0) ld_row<WL>(x[q], p.X + (size_t)v[q] * CW + w0);
        }
#pragma unroll
        for (int q = 0; q < UNR; ++q)
#pragma unroll
          for (int k = 0; k < WL; ++k) {
            // a zero bit left (PW: per pass, and only passes sent to)
            if ((x[q][k] | ~valid_mask(w0 + k, gs)) != ~0ULL) {
              if constexpr (PW) {
                if (dj[k]) room |= 1u << (8 * q + w0 + k);
              } else {
                room |= 1u << q;
              }
            }
            // the bits the row lacks: all atomics under way at once
            x[q][k] = dj[k] & ~x[q][k];
            old[q][k] = 0ULL;
            if (x[q][k])
              old[q][k] = (uint64_t)atomicOr(
                  reinterpret_cast<unsigned long long *>(p.X + (size_t)v[q] * CW + w0 + k),
                  (unsigned long long)x[q][k]);
          }
        // new bits: each has this lane as its only finder
#pragma unroll
        for (int q = 0; q < UNR; ++q)
#pragma unroll
          for (int k = 0; k < WL; ++k) {
            x[q][k] &= ~old[q][k];
            if (x[q][k]) {
              red_or(L.Dc + (size_t)v[q] * CW + w0 + k, x[q][k]);
              gain |= 1u << q;
            }
          }
        if (piece) {  // one delta for the warp: its bits counted over the lanes
#pragma unroll
          for (int k = 0; k < WL; ++k) {
            uint64_t any = 0;
#pragma unroll
            for (int q = 0; q < UNR; ++q) any |= x[q][k];
            if (!__any_sync(kFullMask, any != 0ULL)) continue;
            uint64_t m = __shfl_sync(kFullMask, dj[k], 0);  // the piece's first lane has an arc
            while (m) {
              const int bit = __ffsll((long long)m) - 1;
              m &= m - 1;
              uint32_t n = 0;
#pragma unroll
              for (int q = 0; q < UNR; ++q) n += (uint32_t)(x[q][k] >> bit) & 1u;
              n = __reduce_add_sync(kFullMask, n);
              if (L.lane == 0 && n) count_add(L, c0 + (w0 + k) * 64 + bit, n);
            }
          }
        } else {
#pragma unroll
          for (int q = 0; q < UNR; ++q)
#pragma unroll
            for (int k = 0; k < WL; ++k) count_bits(L, c0, w0 + k, x[q][k]);
        }
      } while (__any_sync(kFullMask, left != 0u));
      if constexpr (!PW && PAIRS > 1) {
        // full in every word sent: the others decide whether the row is active
#pragma unroll
        for (int q = 0; q < UNR; ++q)
          if (v[q] >= 0 && !((room >> q) & 1u)) {
            uint64_t y[CW];
            ld_row<CW>(y, p.X + (size_t)v[q] * CW);
            bool full = true;
#pragma unroll
            for (int k = 0; k < CW; ++k) full &= (y[k] | ~valid_mask(k, gs)) == ~0ULL;
            if (!full) room |= 1u << q;
          }
      }
      // the claim and the place in F_t, for rows with room
      uint32_t od[UNR];
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
        od[q] = 0;
        const bool gq = (gain >> q) & 1u;
        const uint32_t want = (gq ? kChanged : 0u) | (!PW && ((room >> q) & 1u) ? kClaimed : 0u);
        if (!want) mk[q] = ~0u;
        if (want & ~(mk[q] >> ((v[q] & 15) * 2))) {
          mk[q] = mark_word(L.Mc, v[q], want);
          if (deg_now && gq && p.deg_out != p.deg_in) od[q] = p.deg_out[v[q]];
        }
      }
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
        mk[q] >>= (v[q] & 15) * 2;
        if (!deg_now) {
          const bool app = ((gain >> q) & 1u) && !(mk[q] & kChanged);
          if (v[q] >= 0 && (PW ? ((room >> (8 * q)) & 0xFFu) != 0u : !(mk[q] & kClaimed)))
            deg[q] = p.deg_in[v[q]];
          if (app) od[q] = p.deg_out[v[q]];
        } else if (p.deg_out == p.deg_in) {
          od[q] = deg[q];
        }
      }
      if (L.scnt > kStage - 32 * UNR) stage_spill<SEG>(p, L);
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
        if constexpr (PW) {
          uint32_t m = (room >> (8 * q)) & 0xFFu;
          if (m) m = claim_passes(L.Kc, v[q], m);
          if (m) {
            L.mact += (unsigned long long)deg[q] * __popc(m);
            L.rows += __popc(m);
            for (; m; m &= m - 1)
              L.work += (unsigned long long)deg[q] * __popcll(valid_mask(__ffs(m) - 1, p.s));
          }
        } else if (!(mk[q] & kClaimed)) {
          L.mact += deg[q];
          if (SEG) L.work += (unsigned long long)deg[q] * (unsigned long long)gs;
          ++L.rows;
          if (SEG && gm) atomicAdd(gm, (unsigned long long)deg[q]);
        }
        const bool app = ((gain >> q) & 1u) && !(mk[q] & kChanged);
        if (app) stage_degree<SEG>(p, L, od[q], g);
        stage_row(L, v[q], app);
      }
      ob += (int64_t)UNR * stride;
    }
  }
}

// ------------------------------------------------------------- dense rounds
// The sweep of pull_dense (kernels.cuh) with its early stop, finishing each
// row on the spot: new bits go to X and D of this round and are counted by a
// 32 x 32 bit transpose per word and half.
//
// PAIR (rows of 8 words, graphs of kEarlyStopArcs arcs and more): a lane holds
// four words of a row (one 32-byte sector), a pair of lanes the row, and a
// warp takes a chunk in two halves. The pair's gathers of a neighbour are one
// L1 access instead of two, eight arcs a lane fit the registers, and each lane
// stops at the arc where its own half can gain nothing more: R-MAT 20 (s =
// 400) 996 -> 826 us a call. Smaller graphs wait for the two halves in turn
// (900^2 grid, s = 500: 101 -> 120 ms), so a lane takes the whole row there.
template <int CW, bool PW, bool SEG, bool PAIR>
__device__ __forceinline__ void sweep_round(const Params &p, Lane &L, bool tc,
                                            const uint64_t *alive) {
  constexpr int SUB = PAIR ? 2 : 1;       // lanes per row
  constexpr int U = SEG || CW / SUB > 4 ? 4 : 8;  // arcs a lane gathers together
  constexpr int WL = CW / SUB;            // words per lane
  constexpr int RPW = 32 / SUB;           // rows per warp
  const int sub = L.lane % SUB, w0 = sub * WL;
  const int nd = SEG ? *(volatile int32_t *)&p.ctrl->ndense : 0;
  const int64_t nunits = SUB * (SEG ? *(volatile int64_t *)(p.dpref + nd) : p.sell_chunks);
  // a chunk's graph and place: all chunks in order, or (a packed batch) those
  // of the graphs in a full sweep
  auto chunk_at = [&](int64_t ci, int &g) -> int64_t {
    if constexpr (!SEG) {
      g = 0;
      return ci;
    } else {
      int lo = 0, hi = nd - 1;  // the last k with dpref[k] <= ci
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (*(volatile int64_t *)(p.dpref + mid) <= ci) lo = mid; else hi = mid - 1;
      }
      g = *(volatile int32_t *)(p.dlist + lo);
      return __ldg(p.seg_chunk0 + g) + (ci - *(volatile int64_t *)(p.dpref + lo));
    }
  };
  // the next unit's descriptor is fetched when a unit starts, its first
  // columns and signatures when the unit ends (a row cut into pieces may gain
  // bits from another warp in between: its atomics find that out)
  int g_next = 0, clen_next = 0;
  int64_t off_next = 0;
  ulonglong2 it_next = make_ulonglong2(0ULL, 0ULL);
  int32_t u_next[U];
  uint64_t own_next[WL];
  auto descriptor = [&](int64_t ui) {
    it_next = make_ulonglong2(0ULL, 0ULL);
    clen_next = 0;
    if (ui < nunits) {
      const int64_t c = chunk_at(ui / SUB, g_next);
      const int r = (int)(ui % SUB) * RPW + L.lane / SUB;  // row of the chunk
      it_next = __ldg(p.sell_items + c * 32 + r);
      clen_next = __ldg(p.sell_len + c);
      off_next = __ldg(p.sell_off + c) + r;
    }
  };
  auto first_columns = [&]() {
    const int len = (int)(it_next.y & 0x7FFFFFFFULL);
    const int32_t *cc = p.sell_col + off_next;
#pragma unroll
    for (int q = 0; q < U; ++q) u_next[q] = q < len ? __ldg(cc + 32LL * q) : -1;
#pragma unroll
    for (int k = 0; k < WL; ++k) own_next[k] = ~0ULL;
    if (len > 0) ld_row<WL>(own_next, p.X + (size_t)(it_next.y >> 32) * CW + w0);
  };
  descriptor(L.warp);
  first_columns();
  for (int64_t ui = L.warp; ui < nunits; ui += L.nwarps) {
    int gs = p.s, c0 = 0;
    const int g = g_next;
    unsigned long long *gm = nullptr;
    if constexpr (SEG) {
      gs = __ldg(p.graph_s + g);
      c0 = __ldg(p.graph_col0 + g);
      if (p.gmact) gm = p.gmact + (size_t)(L.t - p.row_base) * (size_t)p.nseg + g;
    }
    const ulonglong2 it = it_next;
    const int clen = clen_next;
    const int32_t *cc = p.sell_col + off_next;
    const int32_t v = (int32_t)(it.y >> 32);
    const bool whole = (it.y & 0x80000000ULL) != 0ULL;
    const int len = (int)(it.y & 0x7FFFFFFFULL);
    uint64_t own[WL], acc[WL];
#pragma unroll
    for (int k = 0; k < WL; ++k) {
      own[k] = own_next[k];
      acc[k] = 0ULL;
    }
    int32_t u[U];
#pragma unroll
    for (int q = 0; q < U; ++q) u[q] = u_next[q];
    descriptor(ui + L.nwarps);
    auto pair_any = [&](bool x) {
      return SUB == 1 ? x : (__shfl_xor_sync(kFullMask, (int)x, 1) != 0) || x;
    };
    auto can_gain = [&]() {
      uint64_t r = 0;
#pragma unroll
      for (int k = 0; k < WL; ++k) {
        const uint64_t lim = alive ? alive[w0 + k] : valid_mask(w0 + k, gs);
        r |= lim & ~(own[k] | acc[k]);
        if (PW && !acc[k] && lim && (own[k] | ~valid_mask(w0 + k, p.s)) != ~0ULL) r |= 1ULL;
      }
      return r != 0ULL;
    };
    bool act = false;  // a zero bit left
#pragma unroll
    for (int k = 0; k < WL; ++k) act |= (own[k] | ~valid_mask(w0 + k, gs)) != ~0ULL;
    act = pair_any(act);
    bool open = act && can_gain();
    bool found = false;  // an in-neighbour changed
    bool need = PW ? open : act;
    for (int k0 = 0; k0 < clen; k0 += U) {
      if (!__any_sync(kFullMask, need)) break;
      int32_t un[U];
      const bool more = k0 + U < clen;
      if (more) {
#pragma unroll
        for (int q = 0; q < U; ++q)
          un[q] = (need && k0 + U + q < len) ? __ldg(cc + 32LL * (k0 + U + q)) : -1;
      }
      // (a pair gathers together until it has seen a change)
      const bool other_open = SUB > 1 && __shfl_xor_sync(kFullMask, (int)open, 1) != 0;
      const bool pair_open = open || other_open;  // every lane takes part in the exchange
      const bool together = !PW && !found;
      const bool gather = open || (together && need && pair_open);
      // an arc is read, and a row gathered, once if either lane does so
      if (sub == 0 && (pair_open || (together && act)))
        L.scan += (uint32_t)max(0, min(U, len - k0));
      const bool counts = sub == 0 || !(other_open || together);
      if (gather) {
        if (tc) {
#pragma unroll
          for (int q = 0; q < U; ++q)
            if (u[q] >= 0 && !changed(L.Mp, u[q])) u[q] = -1;
        }
#pragma unroll
        for (int q = 0; q < U; ++q)
          if (u[q] >= 0 && gather_ok(p, u[q], CW - 1)) {
            uint64_t d[WL];
            ld_row<WL>(d, L.Dp + (size_t)u[q] * CW + w0);
#pragma unroll
            for (int k = 0; k < WL; ++k) acc[k] |= d[k];
            if (counts) ++L.gath;
          }
#pragma unroll
        for (int k = 0; k < WL; ++k) found |= acc[k] != 0ULL;
        open = can_gain();
      } else if (need) {  // only whether the row is active
#pragma unroll
        for (int q = 0; q < U; ++q)
          if (u[q] >= 0 && gather_ok(p, u[q], 0)) found |= changed(L.Mp, u[q]);
      }
      found = pair_any(found);
      need = open || (need && !PW && !found);
      if (more) {
#pragma unroll
        for (int q = 0; q < U; ++q) u[q] = need ? un[q] : -1;
      }
    }
    first_columns();
    if (act && sub == 0) ++L.items;
    act = act && found;
    // m_active
    uint32_t gdeg = 0, mask = 0;
    if constexpr (PW) {
      if (act) {
#pragma unroll
        for (int k = 0; k < WL; ++k)
          if (acc[k] && (own[k] | ~valid_mask(w0 + k, p.s)) != ~0ULL) mask |= 1u << (w0 + k);
      }
      if (SUB > 1) mask |= __shfl_xor_sync(kFullMask, mask, 1);
    }
    if (act && sub == 0) {
      const unsigned long long deg = whole ? (uint32_t)len : p.deg_in[v];
      if constexpr (PW) {
        if (mask && !whole) mask = claim_passes(L.Kc, v, mask);
        L.mact += deg * __popc(mask);
        L.rows += __popc(mask);
        for (; mask; mask &= mask - 1)
          L.work += deg * __popcll(valid_mask(__ffs(mask) - 1, p.s));
      } else if (whole || !(mark(L.Mc, v, kClaimed) & kClaimed)) {
        L.mact += deg;
        if (SEG) L.work += deg * (unsigned long long)gs;
        ++L.rows;
        gdeg = (uint32_t)deg;
      }
    }
    if (SEG && gm) {  // the rows of a chunk are one graph's
      const unsigned any = __ballot_sync(kFullMask, gdeg != 0u);
      if (any) {
        unsigned long long sum = gdeg;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(kFullMask, sum, off);
        if (L.lane == 0) atomicAdd(gm, sum);
      }
    }
    // new bits: to X and D of this round
    bool gain = false;
#pragma unroll
    for (int k = 0; k < WL; ++k) {
      acc[k] &= act ? ~own[k] : 0ULL;
      gain |= acc[k] != 0ULL;
    }
    if (gain) {
      uint64_t *xr = p.X + (size_t)v * CW + w0, *dr = L.Dc + (size_t)v * CW + w0;
      if (whole) {
#pragma unroll
        for (int k = 0; k < WL; ++k) own[k] |= acc[k];
        store_words<WL>(xr, own);
        store_words<WL>(dr, acc);
      } else {
        gain = false;
#pragma unroll
        for (int k = 0; k < WL; ++k)
          if (acc[k]) {
            acc[k] &= ~(uint64_t)atomicOr(reinterpret_cast<unsigned long long *>(xr + k),
                                          (unsigned long long)acc[k]);
            if (acc[k]) {
              red_or(dr + k, acc[k]);
              gain = true;
            }
          }
      }
    }
    gain = pair_any(gain);
    bool app = false;
    if (gain && sub == 0) {
      if (whole) {
        mark(L.Mc, v, kChanged);
        app = true;
      } else {
        app = !(mark(L.Mc, v, kChanged) & kChanged);
      }
    }
    if (__any_sync(kFullMask, gain)) {
#pragma unroll
      for (int k = 0; k < WL; ++k)
        if (__any_sync(kFullMask, acc[k] != 0ULL)) {
          const uint32_t t0 = transpose32((uint32_t)acc[k], L.lane);
          const uint32_t t1 = transpose32((uint32_t)(acc[k] >> 32), L.lane);
#pragma unroll
          for (int h = 0; h < SUB; ++h) {  // the rows' word k is on every SUB-th lane
            const uint32_t m = SUB == 1 ? ~0u : h ? 0xAAAAAAAAu : 0x55555555u;
            const uint32_t n0 = __popc(t0 & m), n1 = __popc(t1 & m);
            const int col = c0 + (h * WL + k) * 64 + L.lane;
            if (n0) count_add(L, col, n0);
            if (n1) count_add(L, col + 32, n1);
          }
        }
      if (L.scnt > kStage - 32) stage_spill<SEG>(p, L);
      if (app) stage_degree<SEG>(p, L, p.deg_out[v], g);
      stage_row(L, v, app);
    }
  }
}

// Rows of 8 words: which seed owns which bit. A sweep gathers a row's two
// 32-byte parts on two lanes and leaves a part out once the row can gain
// nothing in it, so the seeds that reach the hubs late (those with few out-arcs) share
// one part: they keep that part open in every row for a round, and the other
// one closes after a few arcs. Seeds in order of out-degree, the first half of
// those with any in words 0-3, the others in words 4-7, seeds without
// out-arcs in the places left. Simulated on R-MAT 21 (s = 512), the largest
// round gathers 63 M parts instead of 103 M.
__device__ void place_seeds(const Params &p, Shared &sh, uint32_t *deg, const int32_t *seeds,
                            int sp) {
  for (int i = threadIdx.x; i < sp; i += blockDim.x) {
    int64_t x = seeds[i];
    if (p.perm) x = __ldg(p.perm + x);
    deg[i] = (uint32_t)(__ldg(p.out_ptr + x + 1) - __ldg(p.out_ptr + x));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < sp; i += blockDim.x) {
    const uint32_t d = deg[i];
    int r = 0, alive = 0;  // rank by degree, seeds with out-arcs
    for (int j = 0; j < sp; ++j) {
      const uint32_t e = deg[j];
      r += e > d || (e == d && j < i);
      alive += e != 0u;
    }
    const int nb = min(sp - 256, alive / 2), na = alive - nb;  // in words 4-7, in words 0-3
    const int k = r - alive;
    const int at = r < na        ? r
                   : r < alive   ? 256 + r - na
                   : k < 256 - na ? na + k
                                  : 256 + nb + k - (256 - na);
    sh.place[i] = (uint16_t)at;
    sh.col[at] = (uint16_t)i;
  }
  __syncthreads();
}

// A packed batch, by the block that arrived last: the graphs whose frontier
// asks for a full sweep of the next round, in graph order, with the prefix of
// their chunk counts.
__device__ void list_dense(const Params &p, int cur) {
  if (!p.dlist) return;
  const unsigned long long *gf = p.gfsum + (size_t)cur * (size_t)p.nseg;
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  long long at = 0, chunks = 0;
  for (int g0 = 0; g0 < p.nseg; g0 += 32) {
    const int g = g0 + lane;
    const bool d = g < p.nseg && *(volatile unsigned long long *)(gf + g) > __ldg(p.gthr + g);
    const unsigned mask = __ballot_sync(kFullMask, d);
    unsigned long long tot;
    const unsigned long long ex = warp_excl_scan64(
        d ? (unsigned long long)(p.seg_chunk0[g + 1] - p.seg_chunk0[g]) : 0ULL, lane, &tot);
    if (d) {
      const long long k = at + __popc(mask & ((1u << lane) - 1u));
      p.dlist[k] = g;
      p.dpref[k] = chunks + (long long)ex;
    }
    at += __popc(mask);
    chunks += (long long)tot;
  }
  if (lane == 0) {
    p.dpref[at] = chunks;
    p.ctrl->ndense = (int32_t)at;
  }
}

// The launch's results, to pinned host memory.
__device__ __forceinline__ void hand_over(ResidentOut *out, const RoundStats *stats,
                                          const uint32_t *counts, int ncols, const Ctrl *ctrl,
                                          const int *rows_out, unsigned long long *sums,
                                          uint32_t scan, uint32_t gath, uint32_t items) {
  const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long s3[3] = {scan, gath, items};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s3[k] += __shfl_xor_sync(kFullMask, s3[k], off);
    if ((threadIdx.x & 31) == 0) atomicAdd(sums + k, s3[k]);
  }
  __syncthreads();
  if (threadIdx.x < 3) out->sums[blockIdx.x][threadIdx.x] = sums[threadIdx.x];
  // at the fixpoint every row is complete: the last counts left their blocks a
  // round ago
  const int rows = *rows_out;  // thread 0's, after the barrier
  const size_t rs_bytes = sizeof(RoundStats) * (size_t)(rows + 1);
  const bool fits = rows >= 0 &&
                    rs_bytes + sizeof(uint32_t) * (size_t)rows * (size_t)ncols <= kResidentOut;
  if (fits) {
    if (blockIdx.x == 0) {
      const unsigned long long *rs = reinterpret_cast<const unsigned long long *>(stats);
      unsigned long long *to = reinterpret_cast<unsigned long long *>(out->data);
      for (int i = threadIdx.x; i < (int)(rs_bytes / 8); i += blockDim.x)
        to[i] = *(volatile const unsigned long long *)(rs + i);
    }
    uint32_t *to = reinterpret_cast<uint32_t *>(out->data + rs_bytes);
    // (32-bit indices: 64-bit ones made the rounds spill)
    for (uint32_t i = tid; i < (uint32_t)(rows * ncols); i += gridDim.x * blockDim.x)
      to[i] = ld_u32(counts + i);
  }
  if (tid == 0) {
    out->ctrl = *ctrl;
    out->rows = fits ? rows : -1;
  }
}

template <int CW, bool PW, bool SEG, bool PAIR>
__global__ void __launch_bounds__(kMaxThreads, 1)
    k_rounds(const __grid_constant__ Params p, const int32_t *seeds, const int32_t *seed_bit,
             int sp, int resume, int epoch) {
  extern __shared__ uint32_t dyn[];
  __shared__ Shared sh;
  const bool smem_counts = p.ncols <= kResidentCounts;  // two rows of counters, by round parity
  Ctrl *ctrl = p.ctrl;
  ResidentCtl *rc = p.rctl;
  Lane L;
  L.lane = threadIdx.x & 31;
  L.wid = threadIdx.x >> 5;
  L.warp = (int64_t)L.wid * gridDim.x + blockIdx.x;
  L.nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  L.tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  L.nth = (int64_t)gridDim.x * blockDim.x;
  L.stage = reinterpret_cast<int32_t *>(dyn + (smem_counts ? 2 * p.ncols : 0)) + L.wid * kStage;
  L.scnt = 0;
  L.od = L.ne = L.gacc = 0;
  L.gcur = -1;
  L.mact = L.work = 0;
  L.rows = L.scan = L.gath = L.items = 0;
  if (smem_counts)
    for (int i = threadIdx.x; i < 2 * p.ncols; i += blockDim.x) dyn[i] = 0u;
  // the thread that looks for a changed part: in the warp that comes last to a
  // round's work, so that a short round does not wait for the host's memory
  const bool poll = blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1;
  if (poll) {
    sh.t0 = clock64();
    sh.look = min(kShrinkCycles, p.slice_cycles) + 1;
  }
  if (threadIdx.x == 0) {
    sh.mact = sh.work = sh.od = sh.ne = 0;
    sh.rows = sh.staged = 0;
    sh.bar = 0;
    sh.sums[0] = sh.sums[1] = sh.sums[2] = 0;
  }
  if (L.tid == 0) ctrl->bad_index = 0;
  // (the stages are free until the first round)
  if (PAIR && p.sort_seeds) place_seeds(p, sh, dyn + 2 * p.ncols, seeds, sp);
  auto none = [] {};
  const int64_t mwords = (p.n + 15) / 16, kwords = (p.n + 3) / 4;  // marks, claim bytes
  int t;
  int64_t nF_old = 0;  // |F_{t-2}|
  int prev_dense = 0;  // round t was a sweep (its long rows are not in E)
  int dense_rounds = 0;
  if (!resume) {
    // everything zero, then the seeds as the change of round 0
    const ulonglong2 z = make_ulonglong2(0ULL, 0ULL);
    const int64_t words = p.n * CW, pairs = words >> 1;
    ulonglong2 *x2 = reinterpret_cast<ulonglong2 *>(p.X);
    ulonglong2 *d0 = reinterpret_cast<ulonglong2 *>(p.D0);
    ulonglong2 *d1 = reinterpret_cast<ulonglong2 *>(p.D1);
    ulonglong2 *d2 = reinterpret_cast<ulonglong2 *>(p.D2);
    for (int64_t i = L.tid; i < pairs; i += L.nth) x2[i] = z;
    if ((words & 1) && L.tid == 0) p.X[words - 1] = 0ULL;
    // (three quarters of this traffic: 1.9 of R-MAT 26's 43 ms)
    if (p.zero_d) {
      for (int64_t i = L.tid; i < pairs; i += L.nth) {
        d0[i] = z;
        d1[i] = z;
        d2[i] = z;
      }
      if ((words & 1) && L.tid == 0) p.D0[words - 1] = p.D1[words - 1] = p.D2[words - 1] = 0ULL;
    }
    for (int64_t i = L.tid; i < mwords; i += L.nth) p.C0[i] = p.C1[i] = p.C2[i] = 0u;
    if constexpr (PW)
      for (int64_t i = L.tid; i < kwords; i += L.nth) p.Kw0[i] = p.Kw1[i] = 0u;
    // degrees as one 32-bit word a row (a row's columns are distinct, so < n):
    // one access per claim or append instead of two row bounds
    for (int64_t i = L.tid; i < p.n; i += L.nth)
      p.deg_in[i] = (uint32_t)(__ldg(p.row_ptr + i + 1) - __ldg(p.row_ptr + i));
    if (p.deg_out != p.deg_in)
      for (int64_t i = L.tid; i < p.n; i += L.nth)
        p.deg_out[i] = (uint32_t)(__ldg(p.out_ptr + i + 1) - __ldg(p.out_ptr + i));
    for (int64_t i = L.tid; i < (int64_t)p.ncols * 2 && i < (int64_t)p.ncols * p.row_cap; i += L.nth)
      p.counts[i] = 0u;
    if constexpr (SEG)
      for (int64_t i = L.tid; i < 3LL * p.nseg; i += L.nth) p.gfsum[i] = 0ULL;
    if (SEG && p.gmact)
      for (int64_t i = L.tid; i < 2LL * p.nseg; i += L.nth) p.gmact[i] = 0ULL;
    if (L.tid == 0) ctrl->ndense = 0;
    if (L.tid < 2) p.rs[L.tid] = RoundStats{};
    if (L.tid < 3) {
      rc->fp[L.tid] = 0ULL;
      rc->next[L.tid] = {0ULL, 0ULL};
    }
    if (!SEG && p.early_stop && L.tid < 3 * kAliveWords) {  // every seed starts alive
      const int w = (int)L.tid % kAliveWords;
      rc->alive[L.tid / kAliveWords][w] = L.tid < kAliveWords ? valid_mask(w, p.s) : 0ULL;
    }
    if (!grid_barrier<SEG>(p, sh, none)) return;
    for (int64_t base = L.warp * 32; base < sp; base += L.nwarps * 32) {
      const int64_t i = base + L.lane;
      unsigned long long od = 0;
      int32_t x = 0;
      bool first = false;
      if (i < sp) {
        x = seeds[i];
        if (p.perm) {  // the caller's id of a relabelled graph (of its copy k)
          const int64_t k = (int64_t)x / p.perm_n;
          x = (int32_t)(k * p.perm_n + __ldg(p.perm + ((int64_t)x - k * p.perm_n)));
        }
        const int bit = seed_bit ? seed_bit[i] : PAIR && p.sort_seeds ? sh.place[i] : (int)i;
        int col = (int)i;
        if (SEG) col = __ldg(p.graph_col0 + __ldg(p.node_graph + x)) + bit;
        red_or(p.X + (size_t)x * CW + (bit >> 6), 1ULL << (bit & 63));
        red_or(p.D0 + (size_t)x * CW + (bit >> 6), 1ULL << (bit & 63));
        atomicAdd(p.counts + col, 1u);
        first = !(mark(p.C0, x, kChanged) & kChanged);
        if (first) od = (unsigned long long)(__ldg(p.out_ptr + x + 1) - __ldg(p.out_ptr + x));
        if (SEG && od) atomicAdd(p.gfsum + __ldg(p.node_graph + x), od);
      }
      const unsigned mask = __ballot_sync(kFullMask, first);
      if (!mask) continue;
      const unsigned long long ne = od > kBigRow ? (od + kBigPiece - 1) / kBigPiece : 0ULL;
      unsigned long long ot, et;
      warp_excl_scan64(od, L.lane, &ot);
      const unsigned long long ex = warp_excl_scan64(ne, L.lane, &et);
      unsigned long long bf = 0, be = 0;
      if (L.lane == 0) {
        bf = atomicAdd(&rc->fp[0], ((unsigned long long)__popc(mask) << kFsumBits) + ot);
        if (et) be = atomicAdd(&rc->next[0].ne, et);
      }
      bf = __shfl_sync(kFullMask, bf, 0) >> kFsumBits;
      be = __shfl_sync(kFullMask, be, 0);
      if (first) p.F0[bf + __popc(mask & ((1u << L.lane) - 1u))] = x;
      if (et) write_pieces(p.E, be + ex, x, ne, L.lane);
    }
    if (!grid_barrier<SEG>(p, sh, [&] { list_dense(p, 0); })) return;
    t = 0;  // round 0 is complete
  } else {
    t = ctrl->t - 1;
    nF_old = (int64_t)ctrl->nF_prev;
    prev_dense = ctrl->mode;
    dense_rounds = ctrl->dense_rounds;
    // a new counts window: its first row and statistics slot
    for (int64_t i = L.tid; i < (int64_t)p.ncols * 2 && i < (int64_t)p.ncols * p.row_cap; i += L.nth)
      p.counts[i] = 0u;
    if (SEG && p.gmact)
      for (int64_t i = L.tid; i < 2LL * p.nseg; i += L.nth) p.gmact[i] = 0ULL;
    if (L.tid < 2) p.rs[L.tid] = RoundStats{};
    if (!grid_barrier<SEG>(p, sh, none)) return;
  }
  bool first_pass = resume != 0;  // round t's statistics are in the last window
  for (;;) {
    // round t is complete: what it left, the same in every block
    // (one reader a block: every warp of the grid at one word would queue)
    if (threadIdx.x == 0) {
      sh.fp = *(volatile unsigned long long *)&rc->fp[t % 3];
      asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];"
                   : "=l"(sh.ne_all), "=l"(sh.yield)
                   : "l"(&rc->next[t % 3])
                   : "memory");
    }
    __syncthreads();
    const unsigned long long fp = sh.fp;
    int64_t nE = (int64_t)sh.ne_all;
    const bool yield = sh.yield != 0ULL;
    const int64_t nF = (int64_t)(fp >> kFsumBits);
    const int64_t fsum = (int64_t)(fp & kFsumMask);
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    // round t's counts leave the block here, while the next round starts: a
    // block adds up to ncols words to the same few lines as every other, and
    // at the end of the round the barrier would wait for that queue
    if (smem_counts && !first_pass) {
      uint32_t *cs = dyn + (t & 1) * p.ncols;
      uint32_t *crow = p.counts + (size_t)(t - p.row_base) * (size_t)p.ncols;
      for (int i = threadIdx.x; i < p.ncols; i += blockDim.x) {
        const uint32_t c = cs[i];
        if (c) {
          atomicAdd(&crow[PAIR && p.sort_seeds ? sh.col[i] : i], c);
          cs[i] = 0u;
        }
      }
    }
    if (lead && !first_pass) {
      RoundStats *r = p.rs + (t - p.row_base);
      r->changed = (unsigned long long)nF;
      r->fsum = (unsigned long long)fsum;
    }
    bool stop = true;
    int status = PG_OK, last_round = t;
    if (nF == 0) {
      last_round = t - 1;
    } else if (t >= p.max_rounds + 1) {
      status = PG_ERANGE;
    } else if (!first_pass && ((t + 1 - p.row_base >= p.row_cap) | yield)) {
      status = kStatusWindow;
    } else {
      stop = false;
    }
    if (stop) {
      if (nF == 0) {  // the last deltas; the buffers are zero again
        const int32_t *Fl = frontier_buf(p, (t + 2) % 3);
        uint64_t *Dl = delta_buf(p, (t + 2) % 3);
        for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (uint32_t)nF_old;
             i += gridDim.x * blockDim.x)
          for (int k = 0; k < CW; ++k) Dl[(size_t)Fl[i] * CW + k] = 0ULL;
      }
      if (threadIdx.x == 0) sh.rows_out = !SEG && nF == 0 ? t - p.row_base : -1;
      if (lead) {
        ctrl->t = t + 1;
        ctrl->mode = prev_dense;
        ctrl->nF_prev = (unsigned long long)nF_old;
        ctrl->last_round = last_round;
        ctrl->dense_rounds = dense_rounds;
        ctrl->status = status;
        ctrl->done = 1;
      }
      break;
    }
    first_pass = false;
    const bool dense = !SEG && (p.direction == PG_DIR_DENSE ||
                                    (p.direction == PG_DIR_AUTO && fsum > p.dense_above));
    const bool tc = p.test_adapt ? 2 * fsum < p.m : p.test_changed != 0;  // kTestDensity
    const int prev = t % 3;
    ++t;
    L.t = t;
    L.cur = t % 3;
    const int old = (t + 1) % 3;  // of round t-2, next of round t+1
    L.Dp = delta_buf(p, prev);
    L.Dc = delta_buf(p, L.cur);
    L.Mp = mark_buf(p, prev);
    L.Mc = mark_buf(p, L.cur);
    L.Kc = (t & 1) ? p.Kw1 : p.Kw0;
    L.F = frontier_buf(p, L.cur);
    L.E = (t & 1) ? p.E1 : p.E;
    L.pieces = SEG || !dense;
    uint32_t *scnt_s = smem_counts ? dyn + (t & 1) * p.ncols : nullptr;
    L.cs = scnt_s ? (uint32_t)__cvta_generic_to_shared(scnt_s) : 0u;
    L.cg = p.counts + (size_t)(t - p.row_base) * (size_t)p.ncols;
    const int32_t *Fp = frontier_buf(p, prev);
    const unsigned long long *Ep = (t & 1) ? p.E : p.E1;
    if (!SEG && prev_dense && !dense) {
      // after a sweep: the long rows of its frontier, in pieces
      unsigned long long *E = (t & 1) ? p.E : p.E1;
      for (int64_t base = L.warp * 32; base < nF; base += L.nwarps * 32) {
        const int64_t i = base + L.lane;
        int32_t v = 0;
        unsigned long long ne = 0;
        if (i < nF) {
          v = Fp[i];
          const unsigned long long od =
              (unsigned long long)(__ldg(p.out_ptr + v + 1) - __ldg(p.out_ptr + v));
          if (od > kBigRow) ne = (od + kBigPiece - 1) / kBigPiece;
        }
        if (__any_sync(kFullMask, ne != 0ULL)) warp_append_pieces(E, &rc->next[prev].ne, v, ne, L.lane);
      }
      if (!grid_barrier<SEG>(p, sh, none)) return;
      if (threadIdx.x == 0) sh.ne_all = *(volatile unsigned long long *)&rc->next[prev].ne;
      __syncthreads();
      nE = (int64_t)sh.ne_all;
    }
    // round t-2's buffers become round t+1's; from the last thread down, as
    // the work below goes from the first warp up
    {
      const ulonglong2 z = make_ulonglong2(0ULL, 0ULL);
      const int32_t *Fo = frontier_buf(p, old);
      uint64_t *Do = delta_buf(p, old);
      for (int64_t i = L.nth - 1 - L.tid; i < nF_old; i += L.nth) {
        uint64_t *dr = Do + (size_t)Fo[i] * CW;
        if constexpr (CW == 1) {
          dr[0] = 0ULL;
        } else {
#pragma unroll
          for (int k = 0; k < CW; k += 2) *reinterpret_cast<ulonglong2 *>(dr + k) = z;
        }
      }
      uint32_t *Mo = mark_buf(p, old);
      for (int64_t i = L.tid; i < mwords; i += L.nth) Mo[i] = 0u;
      if constexpr (PW) {
        uint32_t *Kn = (t & 1) ? p.Kw0 : p.Kw1;
        for (int64_t i = L.tid; i < kwords; i += L.nth) Kn[i] = 0u;
      }
      const int nrow = t + 1 - p.row_base;  // row t+1 of the counts window
      if (nrow < p.row_cap)
        for (int64_t i = L.tid; i < p.ncols; i += L.nth) p.counts[(size_t)nrow * p.ncols + i] = 0u;
      if (SEG && p.gmact)
        for (int64_t i = L.tid; i < p.nseg; i += L.nth) p.gmact[(size_t)nrow * p.nseg + i] = 0ULL;
      if constexpr (SEG)
        for (int64_t i = L.tid; i < p.nseg; i += L.nth) p.gfsum[(size_t)old * p.nseg + i] = 0ULL;
      if (lead) {
        p.rs[nrow] = RoundStats{};
        rc->fp[old] = 0ULL;
        rc->next[old] = {0ULL, 0ULL};
        if (!SEG && p.early_stop)
          for (int w = 0; w < CW; ++w) rc->alive[old][w] = 0ULL;
      }
    }
    if (poll && should_yield(p, sh)) *(volatile unsigned long long *)&rc->next[L.cur].yield = 1ULL;
    if (dense && p.early_stop) {  // bits that can still travel: round t-1's seeds
      if (threadIdx.x < CW) sh.alive[threadIdx.x] = *(volatile unsigned long long *)&rc->alive[prev][threadIdx.x];
      __syncthreads();
    }
    if (SEG ? p.dlist && *(volatile int32_t *)&ctrl->ndense > 0 : dense)
      sweep_round<CW, PW, SEG, PAIR>(p, L, tc, dense && p.early_stop ? sh.alive : nullptr);
    if (!dense) push_round<CW, PW, SEG>(p, L, Fp, Ep, nF, nE);
    round_flush<PW, SEG>(p, L, sh, scnt_s);
    if (!grid_barrier<SEG>(p, sh, [&] { list_dense(p, L.cur); })) return;
    nF_old = nF;
    prev_dense = dense;
    dense_rounds += dense;
  }
  // once every block got here the launch is whole: the last one out says so, and
  // leaves the barrier's words as the next launch needs them
  if (threadIdx.x == 0 && atomicAdd(&rc->exited, 1u) == gridDim.x - 1) {
    rc->arrive = 0u;
    rc->gen = 0u;
    rc->exited = 0u;
    p.out->complete = epoch;
  }
  hand_over(p.out, p.rs, p.counts, p.ncols, ctrl, &sh.rows_out, sh.sums, L.scan, L.gath, L.items);
}

}  // namespace

template <int CW, bool PAIR = false>
static ResidentFn pick_resident(bool pw, bool seg) {
  if constexpr (!PAIR)
    if (seg) return &k_rounds<CW, false, true, false>;
  return pw ? &k_rounds<CW, true, false, PAIR> : &k_rounds<CW, false, false, PAIR>;
}

ResidentFn resident_fn(int CW, bool pw, bool seg, bool pair) {
  switch (CW) {
    case 1: return pick_resident<1>(pw, seg);
    case 2: return pick_resident<2>(pw, seg);
    case 4: return pick_resident<4>(pw, seg);
    case 8: return pair ? pick_resident<8, true>(pw, false) : pick_resident<8>(pw, seg);
  }
  return nullptr;
}

size_t resident_smem(int ncols, int threads) {
  return sizeof(uint32_t) * (size_t)(ncols <= kResidentCounts ? 2 * ncols : 0) +
         sizeof(int32_t) * (size_t)(threads / 32) * kStage;
}

}  // namespace pg
