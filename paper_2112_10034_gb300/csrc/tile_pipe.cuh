// Tile pipeline of the single-pass chained kernels (grid scan, compaction).
//
// Work on a tile has two parts with a wait between them: fold (read the tile
// in shared memory, publish its aggregate) and finish (needs the tile's
// prefix, the aggregates of all earlier tiles).  A CTA that runs the parts in
// a row has no copy in flight while it waits, and its next tile's aggregate,
// which later tiles wait for, comes late.  Here one resident CTA per SM keeps
// NB tiles in shared memory, each at its own point of
//   ticket, load -> fold, publish -> prefix -> finish -> store
// NW worker warps fold a tile as soon as it has landed and finish one as soon
// as its prefix is there; a loader warp takes tickets and starts loads, a
// prefix warp follows the published aggregates, a store warp copies results
// out.  They meet on mbarriers only: there is no CTA-wide barrier.  Tickets
// are taken as buffers become free, so SMs that reach memory faster take more.
//
// Prefixes.  A look-back per tile has some 900 warps re-reading the few words
// at the frontier of published tiles; their traffic on those lines delayed
// every answer (traced on 2^28 int32: 2.2 us from the last earlier tile's
// publishing to the end of the look-back).  Here each CTA follows the
// frontier once for all its tiles: its prefix warp walks the aggregates in
// tile order, one poll for up to 256 of them, keeps the running prefix, and
// hands it out as the walk reaches each of the CTA's tiles.  It sets out for a
// tile only once that tile is published: most earlier ones are by then, and
// walking as soon as the tile's number is known, at the frontier all the time,
// measured 344 us against 331 on 2^28 int32.  Publishing is one
// store (compaction: one atomicMax, which leaves a withheld word alone), without
// group words or inclusive prefixes.  A poll folds as many aggregates as are
// there, so the order in which fp32 sums are combined, and with it their last
// bits, may differ from run to run.
//
// Every wait ends: tickets are only given to running CTAs, and no tile's
// publishing waits for a prefix (its buffer is free when it gets its ticket,
// and workers never block on one event while another is due), so the lowest
// unpublished tile is always on its way.  Each wait is bounded all the same;
// one that runs out records kDevTimeout and makes the whole CTA stop.
#pragma once

#include "cox_common.cuh"

namespace cox {

// Whether the phase of the given parity has completed, without waiting.
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok)
               : "r"(smem_addr(bar)), "r"(parity)
               : "memory");
  return ok != 0;
}

template <int NB>
struct PipeShared {
  uint64_t full[NB];    // the tile has landed (1 arrival + bytes)
  uint64_t folded[NB];  // its aggregate is published (1)
  uint64_t pref[NB];    // its prefix is in shared memory (1)
  uint64_t done[NB];    // every worker has finished it (NW)
  uint64_t free[NB];    // its results have left the buffer (1)
  int64_t tile[NB];     // -1: no more tiles
  unsigned cnt[NB];     // workers that have folded it
  volatile int abort;
};

// Parity wait by a converged warp; false on abort or time-out.
template <int NB>
__device__ __forceinline__ bool pipe_wait(PipeShared<NB>& ps, uint64_t* bar, uint32_t parity, uint32_t limit) {
  for (uint32_t i = 0; i <= limit; ++i) {
    if (__all_sync(kFull, mbar_try_wait(bar, parity))) return true;
    if (__any_sync(kFull, ps.abort)) return false;
  }
  return false;
}

// A position in a ring of nb buffers and the parity of its round.
struct PipePos {
  int slot = 0;
  uint32_t round = 0;
  __device__ void next(int nb) {
    if (++slot == nb) {
      slot = 0;
      ++round;
    }
  }
  __device__ uint32_t parity() const { return round & 1u; }
};

// Runs the pipeline on a CTA of NG * NW + 3 warps with FL loads in flight.  The
// workers are NG groups of NW warps, group g taking every NG-th of the CTA's
// tiles from its g-th on: NG divides NB, so that a slot's tiles belong to one
// group, which has finished the slot's last tile before it asks for the next (a
// parity can only be told from the one before).  `op` provides, with `slot` the
// tile's buffer:
//   load(slot, tile)     one thread: starts the copies that complete full[slot]
//   fold(slot, tile)     each worker warp: its part of the tile's aggregate
//   publish(slot, tile)  the last worker warp to fold it
//   prefix(slot, tile, limit, abort)  the prefix warp: leaves the tile's prefix in
//                        shared memory; false: gave up
//   finish(slot, tile)   each worker warp: its part of the results
//   store(slot, tile)    one thread: copies out of the buffer; returns when
//                        they have read it
template <int NB, int NW, int NG, int FL, class Op>
__device__ __forceinline__ void tile_pipe(PipeShared<NB>& ps, Op& op, int64_t ntiles, unsigned* ticket,
                                          uint32_t limit, unsigned* status) {
  static_assert(NB % NG == 0 && FL <= NB);
  const int warp = threadIdx.x >> 5, lane = lane_id();
  if (threadIdx.x == 0) {
    for (int b = 0; b < NB; ++b) {
      mbar_init(ps.full + b, 1);
      mbar_init(ps.folded + b, 1);
      mbar_init(ps.pref + b, 1);
      mbar_init(ps.done + b, NW);
      mbar_init(ps.free + b, 1);
      ps.cnt[b] = 0;
    }
    ps.abort = 0;
    mbar_init_fence();
  }
  __syncthreads();
  auto give_up = [&] {
    if (lane == 0) {
      ps.abort = 1;
      atomicOr(status, (unsigned)kDevTimeout);
    }
  };
  if (warp == NG * NW) {  // ------------------------------------------- loader
    PipePos at, ahead;  // the next tile; the one FL before it
    bool ok = true;
    int64_t k = 0;
    int marked = 0;  // slots that have been told of the end
    unsigned t = 0;
    for (;; ++k) {
      if (k >= NB) ok = pipe_wait(ps, ps.free + at.slot, at.parity() ^ 1u, limit);
      if (ok && k >= FL) {
        ok = pipe_wait(ps, ps.full + ahead.slot, ahead.parity(), limit);
        ahead.next(NB);
      }
      if (!ok) break;
      // the first FL tiles are asked for together: one round trip
      if (k == 0 || k >= FL) {
        if (lane == 0) t = atomicAdd(ticket, k == 0 ? (unsigned)FL : 1u);
      } else {
        ++t;
      }
      const int64_t tile = (int64_t)__shfl_sync(kFull, t, 0);
      const bool more = tile < ntiles;
      if (lane == 0) {
        ps.tile[at.slot] = more ? tile : -1;
        if (more) op.load(at.slot, tile);
        else mbar_arrive(ps.full + at.slot);
      }
      __syncwarp();
      if (!more) {
        marked = 1;
        break;
      }
      at.next(NB);
    }
    for (int i = 1; ok && i < NG; ++i) {  // the other groups hear of the end on the slots after
      at.next(NB);
      if (k + i >= NB) ok = pipe_wait(ps, ps.free + at.slot, at.parity() ^ 1u, limit);
      if (ok && lane == 0) {
        ps.tile[at.slot] = -1;
        mbar_arrive(ps.full + at.slot);
      }
      marked += ok;
    }
    if (!ok) give_up();
    if (lane == 0)  // whatever becomes of the CTA, its copies in flight land before it ends
      for (int64_t i = k + marked > NB ? k + marked - NB : 0; i < k; ++i)
        mbar_drain(ps.full + (int)(i % NB), (uint32_t)((i / NB) & 1));
    __syncwarp();
    return;
  }
  if (warp == NG * NW + 2) {  // --------------------------------------- prefix
    for (PipePos at;; at.next(NB)) {
      if (!pipe_wait(ps, ps.full + at.slot, at.parity(), limit)) break;
      const int64_t tile = ps.tile[at.slot];
      if (tile < 0) return;
      if (!pipe_wait(ps, ps.folded + at.slot, at.parity(), limit)) break;
      const bool ok = op.prefix(at.slot, tile, limit, &ps.abort);
      __syncwarp();
      if (!ok) break;
      if (lane == 0) mbar_arrive(ps.pref + at.slot);
    }
    give_up();
    return;
  }
  if (warp == NG * NW + 1) {  // ---------------------------------------- store
    for (PipePos at;; at.next(NB)) {
      if (!pipe_wait(ps, ps.full + at.slot, at.parity(), limit)) break;
      const int64_t tile = ps.tile[at.slot];
      if (tile < 0) return;
      if (!pipe_wait(ps, ps.done + at.slot, at.parity(), limit)) break;
      if (lane == 0) {
        op.store(at.slot, tile);
        mbar_arrive(ps.free + at.slot);
      }
      __syncwarp();
    }
    give_up();
    return;
  }
  // ---------------------------------------------------------- workers
  const int group = warp / NW;
  PipePos f, p;  // the next tile to fold, to finish
  for (int i = 0; i < group; ++i) {
    f.next(NB);
    p.next(NB);
  }
  int held = 0;  // slots from p to f
  bool ended = false;
  uint32_t spin = 0;
  for (;;) {
    if (!ended && held < NB && __all_sync(kFull, mbar_test(ps.full + f.slot, f.parity()))) {
      const int64_t tile = ps.tile[f.slot];
      spin = 0;
      if (tile < 0) {
        ended = true;
        continue;
      }
      op.fold(f.slot, tile);
      __syncwarp();
      unsigned before = 0;
      if (lane == 0) {
        __threadfence_block();
        before = atomicAdd(ps.cnt + f.slot, 1u);
        __threadfence_block();
      }
      if (__shfl_sync(kFull, before, 0) == NW - 1) {
        op.publish(f.slot, tile);
        __syncwarp();
        if (lane == 0) {
          ps.cnt[f.slot] = 0;
          mbar_arrive(ps.folded + f.slot);
        }
      }
      held += NG;
      for (int i = 0; i < NG; ++i) f.next(NB);
      continue;
    }
    if (held) {
      if (__all_sync(kFull, mbar_test(ps.pref + p.slot, p.parity()))) {
        spin = 0;
        op.finish(p.slot, ps.tile[p.slot]);
        __syncwarp();
        if (lane == 0) mbar_arrive(ps.done + p.slot);
        held -= NG;
        for (int i = 0; i < NG; ++i) p.next(NB);
        continue;
      }
    } else if (ended) {
      return;
    }
    // Either event may come next, so neither is waited for (a try_wait
    // suspended on one sleeps through the other: a landed tile waited 1.9 us
    // for its fold).
    __nanosleep(20);
    if (__any_sync(kFull, ps.abort)) return;
    // A look at both takes 0.18 us, a poll of the other warps' waits up to 1 us:
    // counted alike, the workers would end a CTA whose prefix warp has most of
    // its polls left.
    if ((++spin >> 4) > limit) {
      give_up();
      return;
    }
  }
}

}  // namespace cox
