// Pull kernel for wide signatures (many seeds per node): a warp per row
// piece, its 32 lanes spread over the row's words.
//
// Same round as k_pull (Alg. 1 inner loop on the deltas of round t-1): for
// each in-neighbour u of the piece, Sig_next(v) |= D_{t-1}(u). With W words
// per node, lane l holds words l, l + 32, l + 64, ... of the row, so the
// warp reads each gathered neighbour row as one contiguous 8·W-byte segment
// (256 bytes per 32 words) instead of W/8 separate 64-byte pieces; column
// indices are loaded 32 at a time (one per lane), tested in parallel, and the
// surviving neighbours broadcast by shuffle. Dense rounds walk the row-major
// piece list of every unsaturated row, sparse rounds the pieces the post
// kernel claimed. Activity, statistics and the finish of split rows follow
// k_pull.
//
// What bounds it is the bytes gathered: 704 a neighbour at s = 5,568, more
// than L2 holds of them. Two things keep most of them in place:
//  - a 32-bit mask per row and round says which parts of its delta (4 words
//    each, up to 128 words; more beyond) hold a bit. Early rounds' deltas are
//    nearly empty (1.4 bits in 88 words in the second round of ER 10^6), and
//    a part without a bit is not read;
//  - a lane whose word of the row is full, by the row's signature or by what
//    it has gathered, reads no more of it, and a row whose words are all full
//    ends there (Alg. 2's early break). In the last rounds few words are open.
// One graph's rows go to X and D at once (dm0): the post kernel then only
// counts. ER 10^6, degree 16, s = 5,568, per launch in rounds 2 to 7: 2.38 4.03
// 4.00 4.06 4.01 1.20 ms before, 1.05 2.03 2.78 2.79 2.26 0.43 ms now (round 5
// at 4.9 TB/s, 0.72 of the measured copy bandwidth; rounds 2 and 3 wait on
// chains of dependent loads, a row a warp).
#include "kernels.cuh"

namespace pg {

// NW words per lane held in registers (rows of up to 32·NW words); NW = 0
// sweeps a longer row in passes of 128 words (4 per lane, so that 16 loads
// of four neighbours are in flight), re-reading the piece's columns (from
// L1) in each pass.
// Three resident blocks per SM (80 registers; four of 64 for rows of 32 words):
// at 88 words four blocks spill, 16.0 against 14.9 ms a call on ER 10^6. Three
// blocks spill too where a lane holds four words (NW = 4, and NW = 0 for rows
// above 128): about 200 bytes of stores and 120 to 210 of loads.
//
// PW: PROPAGATE-S passes as the words of one signature; m_active is counted
// per pass here, in dense and sparse rounds alike (see count_pass_words).
template <int NW, bool PW>
__global__ void __launch_bounds__(kBlock, NW == 1 ? 4 : 3) k_pull_wide(Params p) {
  constexpr int R = NW > 0 ? NW : 4;  // words per lane per pass
  Ctrl *ctrl = p.ctrl;
  if (*(volatile int32_t *)&ctrl->done) return;
  const int t = ctrl->t;
  const int mode = ctrl->mode;
  const uint64_t *Dprev = (t & 1) ? p.D0 : p.D1;
  uint64_t *Dcur = (t & 1) ? p.D1 : p.D0;
  const uint32_t *Cprev = (t & 1) ? p.C0 : p.C1;
  const uint32_t *Mprev = (t & 1) ? p.dm0 : p.dm1;  // parts of the deltas (else null)
  uint32_t *Mcur = (t & 1) ? p.dm1 : p.dm0;
  int32_t *F = (t & 1) ? p.F1 : p.F0;
  uint32_t *Ccur = (t & 1) ? p.C1 : p.C0;
  uint32_t *Kcur = (t & 1) ? p.K1 : p.K0;
  uint32_t *Knext = (t & 1) ? p.K0 : p.K1;
  uint32_t *Kwcur = (t & 1) ? p.Kw1 : p.Kw0;

  const int64_t gtid = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  const int64_t nthreads = (int64_t)gridDim.x * kBlock;
  for (int64_t i = gtid; i < p.nbm; i += nthreads) Knext[i] = 0u;
  if constexpr (PW) {  // the per-pass claim bits of round t+1
    uint32_t *Kwnext = (t & 1) ? p.Kw0 : p.Kw1;
    for (int64_t i = gtid; i < p.nbm * p.Wp; i += nthreads) Kwnext[i] = 0u;
  }

  const int lane = threadIdx.x & 31;
  const int64_t warp = gtid >> 5;
  const int64_t nwarps = nthreads >> 5;
  const int Wp = p.Wp;
  const int passes = NW > 0 ? 1 : (Wp + 32 * R - 1) / (32 * R);
  const bool tc = test_changed_now(p, ctrl);
  unsigned long long my_mact = 0, my_work = 0;
  uint32_t my_scan = 0, my_gath = 0, my_items = 0, my_rows = 0;
  __shared__ int32_t s_stage[kBlock / 32][kStageRows];  // staged frontier rows per warp
  int32_t *stage = s_stage[threadIdx.x >> 5];
  int scnt = 0;
  // dense: every row's pieces; sparse: the claimed pieces; mixed (a packed
  // batch): the pieces of graphs that chose a full sweep, then the claimed ones
  const int64_t ndense = mode != kModeSparse ? p.nPall : 0;
  const int64_t nitems = ndense + (mode != kModeDense ? (int64_t)ctrl->nA : 0);

  // the next item is fetched ahead of this one's work
  auto item_at = [&](int64_t i) {
    return i < ndense ? p.Pall[i] : i < nitems ? p.A[i - ndense] : make_ulonglong2(0ULL, 0ULL);
  };
  ulonglong2 it_next = item_at(warp);
  for (int64_t item = warp; item < nitems; item += nwarps) {
    const bool dense = item < ndense;
    const ulonglong2 it = it_next;
    it_next = item_at(item + nwarps);
    const int64_t b = (int64_t)it.x;
    const int32_t v = (int32_t)(it.y >> 32);
    const bool whole = (it.y & 0x80000000ULL) != 0ULL;
    const int len = (int)(it.y & 0x7FFFFFFFULL);
    if (len == 0) continue;
    if (dense && test_bit_live(p.Sat, v)) continue;  // warp-uniform
    if (dense && p.gfsum) {  // a packed batch: only graphs in a full sweep
      const int gs = __ldg(p.node_graph + v);
      if (p.gfsum[(size_t)((t - 1) & 1) * (size_t)p.nseg + gs] <= __ldg(p.gthr + gs)) continue;
    }
    const int sv = seeds_of(p, v);
    uint64_t *xr = p.X + (size_t)v * Wp;
    // columns of the piece from a0 on: the lane's one, -1 when its row did not
    // change (if that is known before the gather), and its delta's parts
    auto columns = [&](int a0, uint32_t &parts) {
      int32_t u = a0 + lane < len ? __ldg(p.col + b + a0 + lane) : -1;
      parts = ~0u;
      if (u >= 0 && !gather_ok(p, u, 0)) u = -1;
      if (u >= 0 && Mprev) {
        parts = __ldg(Mprev + u);
        if (!parts) u = -1;
      } else if (u >= 0 && tc && !test_bit(Cprev, u)) {
        u = -1;
      }
      return u;
    };
    uint32_t parts0;
    const int32_t u0 = columns(0, parts0);    // under way with the row's own words
    bool found = false, row_changed = false;  // an in-neighbour changed (warp-uniform)
    uint32_t pw_words = 0, pw_seeds = 0;      // PW: this lane's active passes
    uint32_t out_parts = 0;                   // parts of this row's own delta
    bool full = true;                         // no zero bit left in the row
    for (int pass = 0; pass < passes; ++pass) {
      const int w0 = pass * 32 * R + lane;  // lane's first word of this pass
      uint64_t own[R], acc[R];
      uint32_t open = 0;  // words that can still gain a bit
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int w = w0 + 32 * r;
        acc[r] = 0ULL;
        own[r] = ~0ULL;
        if (w < Wp) {
          own[r] = xr[w];  // (rows cut into pieces: bits of this round may be there already)
          if (valid_mask(w, sv) & ~own[r]) open |= 1u << r;
        }
      }
      bool any = __any_sync(kFullMask, open != 0u);
      for (int a0 = 0; any && a0 < len; a0 += 32) {
        uint32_t parts = parts0;
        const int32_t u = a0 ? columns(a0, parts) : u0;
        unsigned m = __ballot_sync(kFullMask, u >= 0);
        if (Mprev || tc) found |= m != 0u;
        if (pass == 0 && lane == 0) my_gath += (uint32_t)__popc(m);
        while (m && any) {  // four neighbours at a time: their loads are independent
          int32_t uu[4];
          uint32_t pp[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int src = m ? __ffs(m) - 1 : 0;
            uu[q] = __shfl_sync(kFullMask, u, src);
            pp[q] = __shfl_sync(kFullMask, parts, src);
            if (!m) uu[q] = -1;
            m &= m ? m - 1 : 0u;
          }
          uint64_t d[4][R];
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const int w = w0 + 32 * r;
              d[q][r] = 0ULL;
              if (uu[q] >= 0 && ((open >> r) & 1u) && ((pp[q] >> (w >> p.dm_shift)) & 1u))
                d[q][r] = __ldg(reinterpret_cast<const unsigned long long *>(
                                    Dprev + (size_t)uu[q] * Wp) + w);
            }
#pragma unroll
          for (int r = 0; r < R; ++r) {
            acc[r] |= (d[0][r] | d[1][r]) | (d[2][r] | d[3][r]);
            if (((open >> r) & 1u) && !(valid_mask(w0 + 32 * r, sv) & ~(own[r] | acc[r])))
              open &= ~(1u << r);
          }
          any = __any_sync(kFullMask, open != 0u);
        }
      }
      full = full && !any;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int w = w0 + 32 * r;
        if (w >= Wp || !acc[r]) continue;
        if (!(Mprev || tc)) found = true;
        if (PW && (own[r] | ~valid_mask(w, p.s)) != ~0ULL &&
            (whole || !set_bit(Kwcur + (size_t)w * (size_t)p.nbm, v))) {
          ++pw_words;  // pass w is active in this row: it lacked one of its bits
          pw_seeds += (uint32_t)__popcll(valid_mask(w, p.s));
        }
        const uint64_t gain = acc[r] & ~own[r];
        if (!gain) continue;
        // p.dm0: new bits go to X and D at once, and the post kernel only
        // counts them; else to Y, which the post kernel compares with X
        bool mine = whole;
        if (p.dm0 && whole) {
          xr[w] = own[r] | acc[r];
          Dcur[(size_t)v * Wp + w] = gain;
        } else if (p.dm0) {
          const unsigned long long fresh =
              gain & ~atomicOr(reinterpret_cast<unsigned long long *>(xr + w),
                               (unsigned long long)gain);
          mine = fresh != 0ULL;
          if (mine)
            atomicOr(reinterpret_cast<unsigned long long *>(Dcur + (size_t)v * Wp + w), fresh);
        } else if (whole) {
          p.Y[(size_t)v * Wp + w] = own[r] | acc[r];
        } else {
          const unsigned long long old =
              atomicOr(reinterpret_cast<unsigned long long *>(p.Y + (size_t)v * Wp + w),
                       (unsigned long long)gain);
          mine = (old | gain) != old;
        }
        if (mine) {
          row_changed = true;
          out_parts |= 1u << (w >> p.dm_shift);
        }
      }
    }
    found = __any_sync(kFullMask, found);
    if (!PW && dense && !found) {
      // nothing in the open words: whether the row is active at all
      for (int a0 = 0; a0 < len && !found; a0 += 32) {
        const int32_t u = a0 + lane < len ? __ldg(p.col + b + a0 + lane) : -1;
        found = __any_sync(kFullMask, u >= 0 && gather_ok(p, u, 0) && test_bit(Cprev, u));
      }
    }
    row_changed = __any_sync(kFullMask, row_changed);
    if (Mcur && row_changed) {  // for the gathers of round t+1
      if (!whole) {  // other pieces add bits too: the last to do so sees them all
        __threadfence();
        full = true;
        for (int w = lane; w < Wp; w += 32)
          full &= (*(volatile const uint64_t *)(xr + w) | ~valid_mask(w, sv)) == ~0ULL;
        full = __all_sync(kFullMask, full);
      }
      if (full && lane == 0) set_bit(p.Sat, v);
      out_parts = __reduce_or_sync(kFullMask, out_parts);
      if (lane == 0) {
        if (whole)
          Mcur[v] = out_parts;
        else
          atomicOr(Mcur + v, out_parts);
      }
    }
    if constexpr (PW) {  // the row's active passes, summed over the lanes
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        pw_words += __shfl_xor_sync(kFullMask, pw_words, off);
        pw_seeds += __shfl_xor_sync(kFullMask, pw_seeds, off);
      }
      if (lane == 0 && pw_words) {
        const unsigned long long deg =
            whole ? (unsigned long long)len
                  : (unsigned long long)(__ldg(p.row_ptr + v + 1) - __ldg(p.row_ptr + v));
        my_mact += deg * pw_words;
        my_work += deg * pw_seeds;
        my_rows += pw_words;
      }
    }
    bool app = false;
    if (lane == 0) {
      ++my_items;
      my_scan += (uint32_t)len;
      if (!PW && dense && found) {  // active in round t (sparse rounds count at the claim)
        unsigned long long deg = 0;
        if (whole) {
          deg = (unsigned long long)len;
          ++my_rows;
        } else if (!set_bit(Kcur, v)) {
          deg = (unsigned long long)(__ldg(p.row_ptr + v + 1) - __ldg(p.row_ptr + v));
          ++my_rows;
        }
        my_mact += deg;
        my_work += deg * (unsigned long long)sv;
        if (p.gmact && deg)  // a packed batch: the row's own graph
          atomicAdd(p.gmact + (size_t)(t - ctrl->row_base) * (size_t)p.nseg + __ldg(p.node_graph + v),
                    deg);
      }
      if (row_changed) {
        if (whole) {
          atomicOr(Ccur + (v >> 5), 1u << (v & 31));
          app = true;
        } else {
          app = !set_bit(Ccur, v);
        }
      }
    }
    // staged: an append per row took two atomics on the round's counters,
    // which queue at 0.65 ns each (1.3 ms for a round of 10^6 rows)
    scnt = stage_append(p, ctrl, F, stage, scnt, v, app, lane);
  }
  if (scnt) stage_flush(p, ctrl, F, stage, scnt, lane);
  RoundStats *r = p.rs + (t - ctrl->row_base);
  const unsigned long long vals[6] = {my_mact, my_work, my_scan, my_gath, my_items, my_rows};
  unsigned long long *const dsts[6] = {&r->m_active, &r->work,  &r->scanned,
                                       &r->gathered, &r->items, &r->rows};
  block_add<6>(vals, dsts);
}

template <bool PW>
static PullFn pick(int Wp) {
  if (Wp <= 32) return &k_pull_wide<1, PW>;
  if (Wp <= 64) return &k_pull_wide<2, PW>;
  if (Wp <= 96) return &k_pull_wide<3, PW>;
  if (Wp <= 128) return &k_pull_wide<4, PW>;
  return &k_pull_wide<0, PW>;
}

PullFn pull_fn_wide(int Wp, bool pw) { return pw ? pick<true>(Wp) : pick<false>(Wp); }

}  // namespace pg
