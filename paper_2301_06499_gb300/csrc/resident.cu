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
// the counts are complete at the barrier, and three delta buffers take turns
// (t-1 read, t written, t-2 cleared through F_{t-2}).
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
// resident: ER 10^3 (s = 64) 214 -> 136 us, ER 10^4 (s = 64) 282 -> 209 us,
// 1024^2 grid (s = 128, ~2,050 rounds) 82.7 -> 55.8 ms, R-MAT 22 (s = 256)
// 2.23 -> 1.91 ms, R-MAT 26 (s = 512) 54.9 -> 46.7 ms, 30 packed graphs
// 33.6 -> 18.6 ms.
//
// Every wait at the barrier is bounded; on expiry the call returns
// PG_ETIMEOUT. The blocks are co-resident by the cooperative launch.
#include "kernels.cuh"

namespace pg {

namespace {

constexpr int kBigRow = kResidentRow;
constexpr int kBigPiece = kResidentPiece;
constexpr int kStage = 256;      // staged frontier rows per warp
constexpr unsigned long long kBarrierNs = 20ULL * 1000 * 1000 * 1000;

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
__device__ __forceinline__ bool bit_live(const uint32_t *bm, int64_t v) {
  return (ld_u32(bm + (v >> 5)) >> (v & 31)) & 1u;
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
  unsigned long long od[32], ne[32];
  int cnt[32];
  unsigned long long base_f, base_e;
  unsigned long long mact, work;
  uint32_t rows;
  uint64_t alive[kAliveWords];
  int last;    // this block arrived last
  int failed;  // the barrier gave up
  unsigned long long fp, ne_all;
};

// Per-thread state of one round.
struct Lane {
  int lane, wid;         // within the warp, warp within the block
  int64_t warp, nwarps;  // across the grid, neighbours on different SMs
  int64_t tid, nth;
  int t, cur;            // round, its delta buffer
  const uint64_t *Dp;    // deltas of round t-1
  uint64_t *Dc;          // deltas of round t
  const uint32_t *Cp;
  uint32_t *Cc, *Kc;
  int32_t *F;            // F_t
  unsigned long long *E; // pieces of F_t's long rows
  uint32_t *cnt;         // counters of this round: shared memory, or the counts row
  int32_t *stage;
  int scnt;
  bool pieces;           // append E_t (a round that may be followed by a push)
  unsigned long long mact, work;
  uint32_t rows;
  // over the whole launch
  uint32_t scan, gath, items;
};

__device__ __forceinline__ uint64_t *delta_buf(const Params &p, int k) {
  return k == 0 ? p.D0 : k == 1 ? p.D1 : p.D2;
}
__device__ __forceinline__ uint32_t *changed_buf(const Params &p, int k) {
  return k == 0 ? p.C0 : k == 1 ? p.C1 : p.C2;
}
__device__ __forceinline__ int32_t *frontier_buf(const Params &p, int k) {
  return k == 0 ? p.F0 : k == 1 ? p.F1 : p.F2;
}

// Grid barrier. With a finalizer (a packed batch) the block that arrives last
// runs it before the others go on. Returns false once any block gave up.
template <class Fin>
__device__ __forceinline__ bool grid_barrier(const Params &p, Shared &sh, Fin fin) {
  ResidentCtl *rc = p.rctl;
  __syncthreads();
  uint32_t gen = 0;
  if (threadIdx.x == 0) {
    gen = ld_acquire(&rc->gen);
    __threadfence();
    sh.last = atomicAdd(&rc->arrive, 1u) == gridDim.x - 1;
    sh.failed = 0;
  }
  if (p.gfsum) {  // the last block lists the graphs to sweep
    __syncthreads();
    if (sh.last) {
      __threadfence();
      fin();
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) {
    if (sh.last) {
      rc->arrive = 0u;
      __threadfence();
      st_release(&rc->gen, gen + 1u);
    } else {
      unsigned long long t0 = 0;
      for (int spin = 0; ld_acquire(&rc->gen) == gen; ++spin) {
        if ((spin & 255) == 255) {
          const unsigned long long t = now_ns();
          if (!t0) t0 = t;
          if (ld_acquire(&rc->abort) || t - t0 > kBarrierNs) {
            st_release(&rc->abort, 1u);  // the host reads it: the call never reports done
            sh.failed = 1;
            break;
          }
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
  return !sh.failed;
}

// Out-degree and piece totals of the warp's staged rows (and, in a packed
// batch, their graphs' frontier sums).
__device__ __forceinline__ void stage_totals(const Params &p, const Lane &L, unsigned long long &od_t,
                                             unsigned long long &ne_t) {
  __syncwarp();
  unsigned long long od_l = 0, ne_l = 0, gacc = 0;
  unsigned long long *gf = p.gfsum ? p.gfsum + (size_t)L.cur * (size_t)p.nseg : nullptr;
  int gcur = -1;
  for (int i = L.lane; i < L.scnt; i += 32) {
    const int32_t v = L.stage[i];
    const unsigned long long od =
        (unsigned long long)(__ldg(p.out_ptr + v + 1) - __ldg(p.out_ptr + v));
    od_l += od;
    if (od > kBigRow) ne_l += (od + kBigPiece - 1) / kBigPiece;
    if (gf && od) {
      const int gq = __ldg(p.node_graph + v);
      if (gq != gcur) {
        if (gacc) atomicAdd(gf + gcur, gacc);
        gcur = gq;
        gacc = 0;
      }
      gacc += od;
    }
  }
  if (gf) {  // one atomic per warp when its lanes ended on one graph
    const unsigned has = __ballot_sync(kFullMask, gacc != 0);
    if (has) {
      const int g0 = __shfl_sync(kFullMask, gcur, __ffs(has) - 1);
      if (__all_sync(kFullMask, gacc == 0 || gcur == g0)) {
        unsigned long long tot;
        warp_excl_scan64(gacc, L.lane, &tot);
        if (L.lane == 0) atomicAdd(gf + g0, tot);
      } else if (gacc) {
        atomicAdd(gf + gcur, gacc);
      }
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    od_l += __shfl_xor_sync(kFullMask, od_l, off);
    ne_l += __shfl_xor_sync(kFullMask, ne_l, off);
  }
  od_t = od_l;
  ne_t = L.pieces ? ne_l : 0ULL;
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
__device__ __forceinline__ void stage_spill(const Params &p, Lane &L) {
  unsigned long long od_t, ne_t, bf = 0, be = 0;
  stage_totals(p, L, od_t, ne_t);
  if (L.lane == 0) {
    bf = atomicAdd(&p.rctl->fp[L.cur], ((unsigned long long)L.scnt << kFsumBits) + od_t);
    if (ne_t) be = atomicAdd(&p.rctl->ne[L.cur], ne_t);
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
__device__ __forceinline__ void round_flush(const Params &p, Lane &L, Shared &sh, uint32_t *scnt_s) {
  unsigned long long od_t, ne_t;
  stage_totals(p, L, od_t, ne_t);
  unsigned long long m = L.mact, w = L.work, r = L.rows;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    m += __shfl_xor_sync(kFullMask, m, off);
    w += __shfl_xor_sync(kFullMask, w, off);
    r += __shfl_xor_sync(kFullMask, r, off);
  }
  if (L.lane == 0) {
    sh.cnt[L.wid] = L.scnt;
    sh.od[L.wid] = od_t;
    sh.ne[L.wid] = ne_t;
    if (r) {
      atomicAdd(&sh.mact, m);
      atomicAdd(&sh.work, w);
      atomicAdd(&sh.rows, (uint32_t)r);
    }
  }
  __syncthreads();
  const int nw = blockDim.x >> 5;
  RoundStats *rs = p.rs + (L.t - p.row_base);
  if (L.wid == 0) {  // one reservation for the block
    const unsigned long long c = L.lane < nw ? (unsigned long long)sh.cnt[L.lane] : 0ULL;
    const unsigned long long o = L.lane < nw ? sh.od[L.lane] : 0ULL;
    const unsigned long long e = L.lane < nw ? sh.ne[L.lane] : 0ULL;
    unsigned long long ct, ot, et;
    const unsigned long long cx = warp_excl_scan64(c, L.lane, &ct);
    warp_excl_scan64(o, L.lane, &ot);
    const unsigned long long ex = warp_excl_scan64(e, L.lane, &et);
    unsigned long long bf = 0, be = 0;
    if (L.lane == 0) {
      if (et) be = atomicAdd(&p.rctl->ne[L.cur], et);
      if (ct) bf = atomicAdd(&p.rctl->fp[L.cur], (ct << kFsumBits) + ot) >> kFsumBits;
    }
    bf = __shfl_sync(kFullMask, bf, 0);
    be = __shfl_sync(kFullMask, be, 0);
    if (L.lane < nw) {
      sh.od[L.lane] = bf + cx;
      sh.ne[L.lane] = be + ex;
    }
  } else if (L.wid == 1 || nw == 1) {
    if (L.lane == 0 && sh.rows) {
      atomicAdd(&rs->m_active, sh.mact);
      atomicAdd(&rs->work, sh.work);
      atomicAdd(&rs->rows, (unsigned long long)sh.rows);
    }
  }
  if (scnt_s) {
    uint32_t *crow = p.counts + (size_t)(L.t - p.row_base) * (size_t)p.ncols;
    for (int i = threadIdx.x; i < p.ncols; i += blockDim.x) {
      const uint32_t c = scnt_s[i];
      if (c) {
        atomicAdd(&crow[i], c);
        scnt_s[i] = 0u;
      }
    }
  }
  __syncthreads();
  if (L.scnt) stage_write(p, L, sh.od[L.wid], sh.ne[L.wid], ne_t);
  L.scnt = 0;
  L.mact = L.work = 0;
  L.rows = 0;
  if (threadIdx.x == 0) {
    sh.mact = sh.work = 0;
    sh.rows = 0;
  }
}

// Counts the bits of each lane's nw (word k of a row whose count columns
// start at c0): one bit per finder, a handful per row in a sparse round.
__device__ __forceinline__ void count_bits(uint32_t *cnt, int c0, int k, uint64_t nw) {
  while (nw) {
    const int b = __ffsll((long long)nw) - 1;
    nw &= nw - 1;
    atomicAdd(cnt + c0 + k * 64 + b, 1u);
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
template <int CW, bool PW>
__device__ __forceinline__ void push_round(const Params &p, Lane &L, const int32_t *Fp,
                                           const unsigned long long *Ep, int64_t nF, int64_t nE) {
  // arcs a lane handles together; the signatures of 8-word rows fill the
  // registers two at a time
  constexpr int UNR = CW <= 2 ? 4 : (CW == 4 ? 2 : 1);
  const size_t Wp = CW;
  const int64_t groups = (nF + 31) >> 5;
  const unsigned long long *gfp =
      p.gfsum ? p.gfsum + (size_t)((L.t + 2) % 3) * (size_t)p.nseg : nullptr;
  for (int64_t it = L.warp; it < groups + nE; it += L.nwarps) {
    int32_t u = -1;
    int64_t ob = 0, oe = 0;
    int stride = 1;
    if (it < groups) {
      const int64_t i = it * 32 + L.lane;
      if (i < nF) {
        u = Fp[i];
        ob = __ldg(p.out_ptr + u);
        oe = __ldg(p.out_ptr + u + 1);
        if (oe - ob > kBigRow) oe = ob;  // in pieces, below
      }
    } else {
      const unsigned long long e = Ep[it - groups];
      u = (int32_t)(e >> 32);
      const int64_t b0 = __ldg(p.out_ptr + u) + (int64_t)(e & 0xFFFFFFFFULL) * kBigPiece;
      oe = min(__ldg(p.out_ptr + u + 1), b0 + kBigPiece);
      ob = b0 + L.lane;
      stride = 32;
    }
    int gs = p.s, c0 = 0;
    unsigned long long *gm = nullptr;
    if (p.node_graph && u >= 0) {
      const int g = __ldg(p.node_graph + u);
      // a packed batch: graphs swept whole in this round take no push
      if (gfp && gfp[g] > __ldg(p.gthr + g)) oe = ob;
      gs = __ldg(p.graph_s + g);
      c0 = __ldg(p.graph_col0 + g);
      if (p.gmact) gm = p.gmact + (size_t)(L.t - p.row_base) * (size_t)p.nseg + g;
    }
    uint64_t d[CW];
#pragma unroll
    for (int k = 0; k < CW; ++k) d[k] = 0ULL;
    if (ob < oe) {
      if (gather_ok(p, u, CW - 1)) ld_row<CW>(d, L.Dp + (size_t)u * Wp);
      ++L.items;
      ++L.gath;
    }
    while (__any_sync(kFullMask, ob < oe)) {
      int32_t v[UNR];
      uint64_t x[UNR][CW];
      uint32_t kw[UNR];
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
        const int64_t j = ob + (int64_t)q * stride;
        v[q] = j < oe ? __ldg(p.out_col + j) : -1;
        if (v[q] >= 0 && !gather_ok(p, v[q], CW - 1)) v[q] = -1;
      }
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
        kw[q] = 0;
#pragma unroll
        for (int k = 0; k < CW; ++k) x[q][k] = ~0ULL;
        if (v[q] >= 0) {
          ++L.scan;
          ld_row<CW>(x[q], p.X + (size_t)v[q] * Wp);
          if (!PW) kw[q] = ld_u32(L.Kc + (v[q] >> 5));
        }
      }
      // claims (m_active): rows with a zero bit left
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
        if (v[q] < 0) continue;
        if constexpr (PW) {
          uint32_t mask = 0;
#pragma unroll
          for (int k = 0; k < CW; ++k)
            if (d[k] && (x[q][k] | ~valid_mask(k, p.s)) != ~0ULL) mask |= 1u << k;
          if (mask) mask = claim_passes(L.Kc, v[q], mask);
          if (mask) {
            const unsigned long long deg =
                (unsigned long long)(__ldg(p.row_ptr + v[q] + 1) - __ldg(p.row_ptr + v[q]));
            L.mact += deg * __popc(mask);
            L.rows += __popc(mask);
            for (; mask; mask &= mask - 1)
              L.work += deg * __popcll(valid_mask(__ffs(mask) - 1, p.s));
          }
        } else {
          bool full = true;
#pragma unroll
          for (int k = 0; k < CW; ++k) full &= (x[q][k] | ~valid_mask(k, gs)) == ~0ULL;
          if (full) {
            v[q] = -1;
          } else if (!((kw[q] >> (v[q] & 31)) & 1u) && !set_bit(L.Kc, v[q])) {
            const unsigned long long deg =
                (unsigned long long)(__ldg(p.row_ptr + v[q] + 1) - __ldg(p.row_ptr + v[q]));
            L.mact += deg;
            L.work += deg * (unsigned long long)gs;
            ++L.rows;
            if (gm) atomicAdd(gm, deg);
          }
        }
      }
      // the bits each row lacks
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
#pragma unroll
        for (int k = 0; k < CW; ++k) {
          const uint64_t g = v[q] >= 0 ? d[k] & ~x[q][k] : 0ULL;
          x[q][k] = 0ULL;
          if (g)
            x[q][k] = g & ~(uint64_t)atomicOr(
                               reinterpret_cast<unsigned long long *>(p.X + (size_t)v[q] * Wp + k),
                               (unsigned long long)g);
        }
      }
#pragma unroll
      for (int q = 0; q < UNR; ++q) {
        bool app = false;
#pragma unroll
        for (int k = 0; k < CW; ++k)
          if (x[q][k]) {
            red_or(L.Dc + (size_t)v[q] * Wp + k, x[q][k]);
            app = true;
          }
        if (app) app = !bit_live(L.Cc, v[q]) && !set_bit(L.Cc, v[q]);
        if (L.scnt > kStage - 32) stage_spill(p, L);
        stage_row(L, v[q], app);
#pragma unroll
        for (int k = 0; k < CW; ++k) count_bits(L.cnt, c0, k, x[q][k]);
      }
      ob += (int64_t)UNR * stride;
    }
  }
}

// ------------------------------------------------------------- dense rounds
// The sweep of pull_dense (kernels.cuh) with its early stop, finishing each
// row on the spot: new bits go to X and D of this round and are counted by a
// 32 x 32 bit transpose per word and half.
template <int CW, bool PW>
__device__ __forceinline__ void sweep_round(const Params &p, Lane &L, bool tc,
                                            const uint64_t *alive) {
  constexpr int U = 4;
  constexpr bool kPipe = CW <= 4;  // at 8 words the registers are not there
  const size_t Wp = CW;
  const int nd = p.dlist ? *(volatile int32_t *)&p.ctrl->ndense : 0;
  const int64_t nchunks = p.dlist ? *(volatile int64_t *)(p.dpref + nd) : p.sell_chunks;
  for (int64_t ci = L.warp; ci < nchunks; ci += L.nwarps) {
    int64_t c = ci;
    int gs = p.s, c0 = 0;
    unsigned long long *gm = nullptr;
    if (p.dlist) {  // the chunks of the graphs in a full sweep
      int lo = 0, hi = nd - 1;  // the last k with dpref[k] <= ci
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (*(volatile int64_t *)(p.dpref + mid) <= ci) lo = mid; else hi = mid - 1;
      }
      const int g = *(volatile int32_t *)(p.dlist + lo);
      c = __ldg(p.seg_chunk0 + g) + (ci - *(volatile int64_t *)(p.dpref + lo));
      gs = __ldg(p.graph_s + g);
      c0 = __ldg(p.graph_col0 + g);
      if (p.gmact) gm = p.gmact + (size_t)(L.t - p.row_base) * (size_t)p.nseg + g;
    }
    const ulonglong2 it = p.sell_items[c * 32 + L.lane];
    const int clen = __ldg(p.sell_len + c);
    const int32_t *cc = p.sell_col + __ldg(p.sell_off + c) + L.lane;
    const int32_t v = (int32_t)(it.y >> 32);
    const bool whole = (it.y & 0x80000000ULL) != 0ULL;
    const int len = (int)(it.y & 0x7FFFFFFFULL);
    uint64_t own[CW], acc[CW];
#pragma unroll
    for (int k = 0; k < CW; ++k) {
      own[k] = ~0ULL;
      acc[k] = 0ULL;
    }
    if (len > 0) ld_row<CW>(own, p.X + (size_t)v * Wp);
    int32_t u[U];
#pragma unroll
    for (int q = 0; q < U; ++q) u[q] = q < len ? __ldg(cc + 32LL * q) : -1;
    auto can_gain = [&]() {
      uint64_t r = 0;
#pragma unroll
      for (int k = 0; k < CW; ++k) {
        const uint64_t lim = alive ? alive[k] : valid_mask(k, gs);
        r |= lim & ~(own[k] | acc[k]);
        if (PW && !acc[k] && lim && (own[k] | ~valid_mask(k, p.s)) != ~0ULL) r |= 1ULL;
      }
      return r != 0ULL;
    };
    bool act = false;  // a zero bit left
#pragma unroll
    for (int k = 0; k < CW; ++k) act |= (own[k] | ~valid_mask(k, gs)) != ~0ULL;
    bool open = act && can_gain();
    bool found = false;  // an in-neighbour changed
    bool need = PW ? open : act;
    for (int k0 = 0; k0 < clen; k0 += U) {
      if (!__any_sync(kFullMask, need)) break;
      if (!kPipe && k0 > 0) {
#pragma unroll
        for (int q = 0; q < U; ++q)
          u[q] = (need && k0 + q < len) ? __ldg(cc + 32LL * (k0 + q)) : -1;
      }
      int32_t un[U];
      const bool more = kPipe && k0 + U < clen;
      if (more) {
#pragma unroll
        for (int q = 0; q < U; ++q)
          un[q] = (need && k0 + U + q < len) ? __ldg(cc + 32LL * (k0 + U + q)) : -1;
      }
      if (need) L.scan += (uint32_t)max(0, min(U, len - k0));
      if (open) {
        if (tc) {
#pragma unroll
          for (int q = 0; q < U; ++q)
            if (u[q] >= 0 && !((L.Cp[u[q] >> 5] >> (u[q] & 31)) & 1u)) u[q] = -1;
        }
#pragma unroll
        for (int q = 0; q < U; ++q)
          if (u[q] >= 0 && gather_ok(p, u[q], CW - 1)) {
            uint64_t d[CW];
            ld_row<CW>(d, L.Dp + (size_t)u[q] * Wp);
#pragma unroll
            for (int k = 0; k < CW; ++k) acc[k] |= d[k];
            ++L.gath;
          }
#pragma unroll
        for (int k = 0; k < CW; ++k) found |= acc[k] != 0ULL;
        open = can_gain();
      } else if (need) {  // only whether the row is active
#pragma unroll
        for (int q = 0; q < U; ++q)
          if (u[q] >= 0 && gather_ok(p, u[q], 0))
            found |= ((L.Cp[u[q] >> 5] >> (u[q] & 31)) & 1u) != 0u;
      }
      need = open || (need && !PW && !found);
      if (more) {
#pragma unroll
        for (int q = 0; q < U; ++q) u[q] = need ? un[q] : -1;
      }
    }
    if (act) ++L.items;
    act = act && found;
    // m_active
    uint32_t gdeg = 0;
    if (act) {
      const unsigned long long deg =
          whole ? (unsigned long long)len
                : (unsigned long long)(__ldg(p.row_ptr + v + 1) - __ldg(p.row_ptr + v));
      if constexpr (PW) {
        uint32_t mask = 0;
#pragma unroll
        for (int k = 0; k < CW; ++k)
          if (acc[k] && (own[k] | ~valid_mask(k, p.s)) != ~0ULL) mask |= 1u << k;
        if (mask && !whole) mask = claim_passes(L.Kc, v, mask);
        L.mact += deg * __popc(mask);
        L.rows += __popc(mask);
        for (; mask; mask &= mask - 1)
          L.work += deg * __popcll(valid_mask(__ffs(mask) - 1, p.s));
      } else if (whole || !set_bit(L.Kc, v)) {
        L.mact += deg;
        L.work += deg * (unsigned long long)gs;
        ++L.rows;
        gdeg = (uint32_t)deg;
      }
    }
    if (gm) {  // the rows of a chunk are one graph's
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
    for (int k = 0; k < CW; ++k) {
      acc[k] &= act ? ~own[k] : 0ULL;
      gain |= acc[k] != 0ULL;
    }
    if (gain) {
      uint64_t *xr = p.X + (size_t)v * Wp, *dr = L.Dc + (size_t)v * Wp;
      if (whole) {
#pragma unroll
        for (int k = 0; k < CW; ++k) own[k] |= acc[k];
        store_words<CW>(xr, own);
        store_words<CW>(dr, acc);
      } else {
        gain = false;
#pragma unroll
        for (int k = 0; k < CW; ++k)
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
    bool app = false;
    if (gain) {
      if (whole) {
        atomicOr(L.Cc + (v >> 5), 1u << (v & 31));
        app = true;
      } else {
        app = !set_bit(L.Cc, v);
      }
    }
    if (__any_sync(kFullMask, gain)) {
#pragma unroll
      for (int k = 0; k < CW; ++k)
        if (__any_sync(kFullMask, acc[k] != 0ULL)) {
          const uint32_t n0 = __popc(transpose32((uint32_t)acc[k], L.lane));
          const uint32_t n1 = __popc(transpose32((uint32_t)(acc[k] >> 32), L.lane));
          if (n0) atomicAdd(L.cnt + c0 + k * 64 + L.lane, n0);
          if (n1) atomicAdd(L.cnt + c0 + k * 64 + 32 + L.lane, n1);
        }
      if (L.scnt > kStage - 32) stage_spill(p, L);
      stage_row(L, v, app);
    }
  }
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

template <int CW, bool PW>
__global__ void __launch_bounds__(1024, 1)
    k_rounds(const __grid_constant__ Params p, const int32_t *seeds, const int32_t *seed_bit,
             int sp, int resume, int epoch) {
  extern __shared__ uint32_t dyn[];
  __shared__ Shared sh;
  const bool smem_counts = p.ncols <= kResidentCounts;
  uint32_t *scnt_s = smem_counts ? dyn : nullptr;
  Ctrl *ctrl = p.ctrl;
  ResidentCtl *rc = p.rctl;
  Lane L;
  L.lane = threadIdx.x & 31;
  L.wid = threadIdx.x >> 5;
  L.warp = (int64_t)L.wid * gridDim.x + blockIdx.x;
  L.nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  L.tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  L.nth = (int64_t)gridDim.x * blockDim.x;
  L.stage = reinterpret_cast<int32_t *>(dyn + (smem_counts ? p.ncols : 0)) + L.wid * kStage;
  L.scnt = 0;
  L.mact = L.work = L.scan = L.gath = L.items = 0;
  L.rows = 0;
  if (scnt_s)
    for (int i = threadIdx.x; i < p.ncols; i += blockDim.x) scnt_s[i] = 0u;
  if (threadIdx.x == 0) {
    sh.mact = sh.work = 0;
    sh.rows = 0;
  }
  if (L.tid == 0) ctrl->bad_index = 0;
  auto none = [] {};
  const int64_t kwords = PW ? (p.n + 3) / 4 : p.nbm;  // claim words
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
    for (int64_t i = L.tid; i < pairs; i += L.nth) {
      x2[i] = z;
      d0[i] = z;
      d1[i] = z;
      d2[i] = z;
    }
    if ((words & 1) && L.tid == 0)
      p.X[words - 1] = p.D0[words - 1] = p.D1[words - 1] = p.D2[words - 1] = 0ULL;
    for (int64_t i = L.tid; i < p.nbm; i += L.nth) p.C0[i] = p.C1[i] = p.C2[i] = 0u;
    for (int64_t i = L.tid; i < kwords; i += L.nth) p.K0[i] = p.K1[i] = 0u;
    for (int64_t i = L.tid; i < (int64_t)p.ncols * 2 && i < (int64_t)p.ncols * p.row_cap; i += L.nth)
      p.counts[i] = 0u;
    if (p.gfsum)
      for (int64_t i = L.tid; i < 3LL * p.nseg; i += L.nth) p.gfsum[i] = 0ULL;
    if (p.gmact)
      for (int64_t i = L.tid; i < 2LL * p.nseg; i += L.nth) p.gmact[i] = 0ULL;
    if (L.tid == 0) ctrl->ndense = 0;
    if (L.tid < 2) p.rs[L.tid] = RoundStats{};
    if (L.tid < 3) rc->fp[L.tid] = rc->ne[L.tid] = 0ULL;
    if (!grid_barrier(p, sh, none)) return;
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
        const int bit = seed_bit ? seed_bit[i] : (int)i;
        int col = (int)i;
        if (p.node_graph) col = __ldg(p.graph_col0 + __ldg(p.node_graph + x)) + bit;
        red_or(p.X + (size_t)x * CW + (bit >> 6), 1ULL << (bit & 63));
        red_or(p.D0 + (size_t)x * CW + (bit >> 6), 1ULL << (bit & 63));
        atomicAdd(p.counts + col, 1u);
        first = !set_bit(p.C0, x);
        if (first) od = (unsigned long long)(__ldg(p.out_ptr + x + 1) - __ldg(p.out_ptr + x));
        if (p.gfsum && od) atomicAdd(p.gfsum + __ldg(p.node_graph + x), od);
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
        if (et) be = atomicAdd(&rc->ne[0], et);
      }
      bf = __shfl_sync(kFullMask, bf, 0) >> kFsumBits;
      be = __shfl_sync(kFullMask, be, 0);
      if (first) p.F0[bf + __popc(mask & ((1u << L.lane) - 1u))] = x;
      if (et) write_pieces(p.E, be + ex, x, ne, L.lane);
    }
    if (!grid_barrier(p, sh, [&] { list_dense(p, 0); })) return;
    t = 0;  // round 0 is complete
  } else {
    t = ctrl->t - 1;
    nF_old = (int64_t)ctrl->nF_prev;
    prev_dense = ctrl->mode;
    dense_rounds = ctrl->dense_rounds;
    // a new counts window: its first row and statistics slot
    for (int64_t i = L.tid; i < (int64_t)p.ncols * 2 && i < (int64_t)p.ncols * p.row_cap; i += L.nth)
      p.counts[i] = 0u;
    if (p.gmact)
      for (int64_t i = L.tid; i < 2LL * p.nseg; i += L.nth) p.gmact[i] = 0ULL;
    if (L.tid < 2) p.rs[L.tid] = RoundStats{};
    if (!grid_barrier(p, sh, none)) return;
  }
  bool first_pass = resume != 0;  // round t's statistics are in the last window
  for (;;) {
    // round t is complete: what it left, the same in every block
    if (threadIdx.x == 0) {
      sh.fp = *(volatile unsigned long long *)&rc->fp[t % 3];
      sh.ne_all = *(volatile unsigned long long *)&rc->ne[t % 3];
    }
    __syncthreads();
    const int64_t nF = (int64_t)(sh.fp >> kFsumBits);
    const int64_t fsum = (int64_t)(sh.fp & kFsumMask);
    int64_t nE = (int64_t)sh.ne_all;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
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
    } else if (!first_pass && t + 1 - p.row_base >= p.row_cap) {
      status = kStatusWindow;
    } else {
      stop = false;
    }
    if (stop) {
      if (lead) {
        ctrl->t = t + 1;
        ctrl->mode = prev_dense;
        ctrl->nF_prev = (unsigned long long)nF_old;
        ctrl->last_round = last_round;
        ctrl->dense_rounds = dense_rounds;
        ctrl->status = status;
        ctrl->done = 1;
        ctrl->iters = epoch;  // written by this launch
      }
      break;
    }
    first_pass = false;
    const bool dense = !p.gfsum && (p.direction == PG_DIR_DENSE ||
                                    (p.direction == PG_DIR_AUTO &&
                                     (double)fsum > (double)p.dense_threshold * (double)p.m));
    const bool tc = p.test_adapt ? (double)fsum < kTestDensity * (double)p.m : p.test_changed != 0;
    const int prev = t % 3;
    ++t;
    L.t = t;
    L.cur = t % 3;
    const int old = (t + 1) % 3;  // of round t-2, next of round t+1
    L.Dp = delta_buf(p, prev);
    L.Dc = delta_buf(p, L.cur);
    L.Cp = changed_buf(p, prev);
    L.Cc = changed_buf(p, L.cur);
    L.Kc = (t & 1) ? p.K1 : p.K0;
    L.F = frontier_buf(p, L.cur);
    L.E = (t & 1) ? p.E1 : p.E;
    L.pieces = p.gfsum || !dense;
    L.cnt = scnt_s ? scnt_s : p.counts + (size_t)(t - p.row_base) * (size_t)p.ncols;
    const int32_t *Fp = frontier_buf(p, prev);
    const unsigned long long *Ep = (t & 1) ? p.E : p.E1;
    if (prev_dense && !dense && !p.gfsum) {
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
        if (__any_sync(kFullMask, ne != 0ULL)) warp_append_pieces(E, &rc->ne[prev], v, ne, L.lane);
      }
      if (!grid_barrier(p, sh, none)) return;
      if (threadIdx.x == 0) sh.ne_all = *(volatile unsigned long long *)&rc->ne[prev];
      __syncthreads();
      nE = (int64_t)sh.ne_all;
    }
    if (dense && p.early_stop) {  // bits that can still travel: round t-1's seeds
      const int pr = t - 1 - p.row_base;  // < 0: the row left with the last window
      const uint32_t *row = p.counts + (size_t)(pr < 0 ? 0 : pr) * (size_t)p.ncols;
      for (int w = L.wid; w < CW; w += blockDim.x >> 5) {
        const int i = w * 64 + L.lane;
        const unsigned lo = __ballot_sync(kFullMask, i < p.s && (pr < 0 || ld_u32(row + i) != 0u));
        const unsigned hi =
            __ballot_sync(kFullMask, i + 32 < p.s && (pr < 0 || ld_u32(row + i + 32) != 0u));
        if (L.lane == 0) sh.alive[w] = ((uint64_t)hi << 32) | lo;
      }
      __syncthreads();
    }
    if (dense || (p.dlist && *(volatile int32_t *)&ctrl->ndense > 0))
      sweep_round<CW, PW>(p, L, tc, dense && p.early_stop ? sh.alive : nullptr);
    if (!dense) push_round<CW, PW>(p, L, Fp, Ep, nF, nE);
    // round t-2's buffers become round t+1's
    {
      const ulonglong2 z = make_ulonglong2(0ULL, 0ULL);
      const int32_t *Fo = frontier_buf(p, old);
      uint64_t *Do = delta_buf(p, old);
      for (int64_t i = L.tid; i < nF_old; i += L.nth) {
        uint64_t *dr = Do + (size_t)Fo[i] * CW;
        if constexpr (CW == 1) {
          dr[0] = 0ULL;
        } else {
#pragma unroll
          for (int k = 0; k < CW; k += 2) *reinterpret_cast<ulonglong2 *>(dr + k) = z;
        }
      }
      uint32_t *Co = changed_buf(p, old);
      for (int64_t i = L.tid; i < p.nbm; i += L.nth) Co[i] = 0u;
      uint32_t *Kn = (t & 1) ? p.K0 : p.K1;
      for (int64_t i = L.tid; i < kwords; i += L.nth) Kn[i] = 0u;
      const int nrow = t + 1 - p.row_base;  // row t+1 of the counts window
      if (nrow < p.row_cap)
        for (int64_t i = L.tid; i < p.ncols; i += L.nth) p.counts[(size_t)nrow * p.ncols + i] = 0u;
      if (p.gmact)
        for (int64_t i = L.tid; i < p.nseg; i += L.nth) p.gmact[(size_t)nrow * p.nseg + i] = 0ULL;
      if (p.gfsum)
        for (int64_t i = L.tid; i < p.nseg; i += L.nth) p.gfsum[(size_t)old * p.nseg + i] = 0ULL;
      if (lead) {
        p.rs[nrow] = RoundStats{};
        rc->fp[old] = 0ULL;
        rc->ne[old] = 0ULL;
      }
    }
    round_flush(p, L, sh, scnt_s);
    if (!grid_barrier(p, sh, [&] { list_dense(p, L.cur); })) return;
    nF_old = nF;
    prev_dense = dense;
    dense_rounds += dense;
  }
  // work counters of the launch, on the slot of its last round
  unsigned long long s3[3] = {L.scan, L.gath, L.items};
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s3[k] += __shfl_xor_sync(kFullMask, s3[k], off);
  if (L.lane == 0) {
    RoundStats *r = p.rs + (t - p.row_base);
    if (s3[0]) atomicAdd(&r->scanned, s3[0]);
    if (s3[1]) atomicAdd(&r->gathered, s3[1]);
    if (s3[2]) atomicAdd(&r->items, s3[2]);
  }
}

}  // namespace

ResidentFn resident_fn(int CW, bool pw) {
  switch (CW) {
    case 1: return pw ? &k_rounds<1, true> : &k_rounds<1, false>;
    case 2: return pw ? &k_rounds<2, true> : &k_rounds<2, false>;
    case 4: return pw ? &k_rounds<4, true> : &k_rounds<4, false>;
    case 8: return pw ? &k_rounds<8, true> : &k_rounds<8, false>;
  }
  return nullptr;
}

size_t resident_smem(int ncols, int threads) {
  return sizeof(uint32_t) * (size_t)(ncols <= kResidentCounts ? ncols : 0) +
         sizeof(int32_t) * (size_t)(threads / 32) * kStage;
}

}  // namespace pg
