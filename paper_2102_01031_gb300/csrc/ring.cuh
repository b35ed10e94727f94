// ring.cuh -- the plane ring of a DK pass, as device functions: the shared
// memory behind the stages, the bulk copies that fill a stage with one z-plane
// tile of every array, the release count whose last warp refills the stage,
// the per-run flush of the sums into a partial-sum slot, and what joins two
// passes of one launch.
//
// A CTA's segments form one sequence of planes (each segment adds a halo
// plane at both ends); plane g of pass p lives in stage (p * ptot + g) mod S.
// A stage holds, for every array, the plane's BY rows of the segment's y-tile
// plus one halo row on each side, each row complete in x (with MOWN the momenta,
// read at the tile's own sites only, without the halo rows).
//
// Between two passes of a launch the whole lattice's sums decide the next scale
// factor.  Every CTA keeps the scalars of the lattices it works on in shared
// memory (LatRun) and runs their Friedmann update itself, from the slots all CTAs
// wrote: one counter and one wait join the passes.  (The update used to be run by
// the CTA that wrote a lattice's last slot, and a second counter told the others:
// two more trips through L2 and the new scalars read back, with FP64 coefficients
// formed by every warp.)  Two sets of slots alternate, since a CTA may write its
// next sums while another still reads these; every CTA adds the same slots in the
// same order, so all hold the same scalars.  The last pass of a launch leaves them
// in global memory: there the CTA that completes a lattice's arrival count runs
// the update and stores it.
#pragma once

#include "common.cuh"
#include "tail.cuh"

namespace clg {

// A CTA's run on one lattice: the lattice's evolving scalars as of the current
// pass, its constants, and the pass's coefficients in the storage precision.
template <typename T, int NCF>
struct alignas(16) LatRun {
  ScalarState W;
  LatPar L;
  T cf[NCF];
};
static_assert(sizeof(LatRun<float, 4>) == (sizeof(ScalarState) + sizeof(LatPar) + 16 + 15) / 16 * 16 &&
                  sizeof(LatRun<double, 9>) == (sizeof(ScalarState) + sizeof(LatPar) + 72 + 15) / 16 * 16,
              "run_record_bytes in capi.cu");

struct Ring {
  unsigned char* stages;  // S stages of stage_bytes
  uint64_t* full;         // one mbarrier per stage: all copies of the stage landed
  unsigned* released;     // warps done with each stage
  uint64_t* drifted;      // mbarrier, one arrival per warp (FP64 scalar pass)
  int* off;               // first plane of each segment, and the total
  double* red;            // [33][NQ] reduction scratch
  volatile int* flag;     // [0] timed out, [1] runs of the CTA, [2] lattice of the last run, [3] #pending tails
  int* pend;              // runs whose lattices' Friedmann update this CTA stores
  SegInfo* info;          // per segment
  unsigned char* runs;    // LatRun records
  int S;
  unsigned stage_bytes;
};

__device__ __forceinline__ Ring ring_view(unsigned char* smem, const PassArgs& P) {
  Ring R;
  R.S = P.stages;
  R.stage_bytes = P.stage_bytes_max;
  R.stages = smem;
  unsigned char* tail = smem + (size_t)R.S * R.stage_bytes;
  R.full = reinterpret_cast<uint64_t*>(tail + SM_FULL);
  R.released = reinterpret_cast<unsigned*>(tail + SM_RELEASED);
  R.drifted = reinterpret_cast<uint64_t*>(tail + SM_DRIFTED);
  R.off = reinterpret_cast<int*>(tail + SM_OFF);
  R.red = reinterpret_cast<double*>(tail + SM_RED);
  R.flag = reinterpret_cast<volatile int*>(tail + SM_FLAG);
  R.pend = reinterpret_cast<int*>(tail + SM_FLAG + 16);
  R.info = reinterpret_cast<SegInfo*>(tail + SM_INFO);
  R.runs = tail + SM_INFO + (size_t)P.nseg_max * sizeof(SegInfo);
  return R;
}

// Thread 0: barriers, counts, flags, plane offsets and the records of the CTA's
// `ns` segments starting at segs[sb].
template <int NA>
__device__ void ring_setup(const Ring& R, const PassArgs& P, int sb, int ns) {
  for (int s = 0; s < R.S; ++s) {
    mbar_init(&R.full[s], 1);
    R.released[s] = 0u;
  }
  mbar_init(R.drifted, CONSUMER_WARPS);
  fence_mbar_init();
  R.flag[0] = 0;
  R.flag[2] = ns > 0 ? P.segs[sb].lat : 0;
  R.flag[3] = 0;
  R.off[0] = 0;
  int run = -1;
  for (int i = 0; i < ns; ++i) {
    const Seg sg = P.segs[sb + i];
    const LatConst& L = P.lat[sg.lat];
    R.off[i + 1] = R.off[i] + sg.nz + 2;
    SegInfo& in = R.info[i];
    if (i == 0 || R.info[i - 1].lat != sg.lat) ++run;
    in.z0 = sg.z0;
    in.nz = sg.nz;
    in.dir = sg.dir;
    in.ylo = sg.ytile * L.BY;
    in.N = L.N;
    in.rows = L.BY + 2;
    in.slot = sg.slot;
    in.flush = sg.flush;
    in.run = run;
    in.lat = sg.lat;
    in.slot_begin = L.slot_begin;
    in.slot_end = L.slot_end;
    in.V = L.V;
    for (int p = 0; p < 2; ++p)
      for (int a = 0; a < NA; ++a) in.src[p][a] = L.buf[p][a];
  }
  R.flag[1] = run + 1;
}

// A segment of run r of the CTA (its segments are grouped by lattice).
__device__ __forceinline__ const SegInfo& ring_run(const Ring& R, int ns, int r) {
  int i = 0;
  while (i + 1 < ns && R.info[i].run != r) ++i;
  return R.info[i];
}

// Sums of the first NUSED quantities of the lattices of the CTA's runs which(0) ..
// which(nb - 1) into rows of red, the warps sharing the (lattice, quantity) pairs,
// each over the lattice's slots in a fixed order (warp_slot_sum), so that the result
// depends neither on timing nor on the CTA.
template <int NUSED, class Which>
__device__ __forceinline__ void ring_slot_sums(const Ring& R, const PassArgs& P, int pass, int ns, int nb, int warp,
                                               int lane, Which which) {
  constexpr int NQU = NUSED > 0 ? NUSED : 1;
  const double* slots = P.partials + (size_t)(pass & 1) * NQ * P.nslot;
  for (int it = CONSUMER_WARPS - 1 - warp; it < nb * NUSED; it += CONSUMER_WARPS) {
    const int l = it / NQU, q = it - l * NQU;
    const SegInfo& in = ring_run(R, ns, which(l));
    const double s = warp_slot_sum(slots + (size_t)q * P.nslot, in.slot_begin, in.slot_end, lane);
    if (lane == 0) R.red[l * NQ + q] = s;
  }
}

template <typename T>
__device__ __forceinline__ const T* ring_stage(const Ring& R, int s) {
  return reinterpret_cast<const T*>(R.stages + (size_t)s * R.stage_bytes);
}

// Bulk copies of plane g (of the forward sequence) into stage s, issued by a
// whole warp (warp-uniform call): lane a + NA k copies run k of array a (a
// tile's rows form up to three runs where they wrap around the periodic y
// boundary).  MOWN: the odd arrays (momenta of a field/momentum layout) are
// copied without their halo rows -- the tile's own rows only, one run -- and
// each (field, momentum) pair occupies rows + (rows - 2) rows of the stage,
// the field's first.
// The reuse of stage memory is ordered by the release count.  The passes read it through the
// generic proxy, and a copy needs no proxy fence after reads; the FP64 scalar pass also writes
// drifted values into it, and fences them itself before it releases the stage
// (fence_proxy_async_smem in pass_scalar.cu).
template <typename T, int NA, bool MOWN = false>
__device__ void ring_issue_warp(const Ring& R, int g, int s, int parity, int lane) {
  static_assert(3 * NA <= 32, "one lane per copy");
  int i = 0;
  while (g >= R.off[i + 1]) ++i;
  const SegInfo& in = R.info[i];
  const int N = in.N, rows = in.rows, arr_elems = rows * N;
  const int j = g - R.off[i];
  int zp = in.dir > 0 ? in.z0 - 1 + j : in.z0 + in.nz - j;
  zp = zp < 0 ? zp + N : (zp >= N ? zp - N : zp);
  // rows ylo-1 .. ylo+rows-2 of the plane, periodic in y: r1 rows from y1, then
  // r2 rows from row 0, then (a tile as tall as the lattice wraps twice) r3 from row 0
  const int y0 = in.ylo - 1;
  const int y1 = y0 < 0 ? y0 + N : y0;
  const int r1 = min(rows, N - y1), r2 = min(rows - r1, N), r3 = rows - r1 - r2;
  const size_t stage_elems = MOWN ? (size_t)(NA / 2) * (2 * rows - 2) * N : (size_t)NA * arr_elems;
  if (lane == 0) mbar_arrive_expect_tx(&R.full[s], (uint32_t)(stage_elems * sizeof(T)));
  __syncwarp();
  if (lane < 3 * NA) {
    const int run = lane / NA, a = lane - run * NA;
    const bool own_only = MOWN && (a & 1);
    int nr = run == 0 ? r1 : (run == 1 ? r2 : r3);
    if (own_only) nr = run == 0 ? rows - 2 : 0;  // rows ylo .. ylo + BY - 1 never wrap
    if (nr > 0) {
      const int d = own_only ? 0 : (run == 0 ? 0 : (run == 1 ? r1 : r1 + r2));
      const int ys = own_only ? in.ylo : (run == 0 ? y1 : 0);
      const size_t aoff = MOWN ? (size_t)(a >> 1) * (2 * rows - 2) * N + (a & 1) * (size_t)rows * N
                               : (size_t)a * arr_elems;
      T* st = reinterpret_cast<T*>(R.stages + (size_t)s * R.stage_bytes) + aoff;
      const T* src = reinterpret_cast<const T*>(in.src[parity][a]) + (long long)zp * N * N;
      bulk_g2s(st + (size_t)d * N, src + (long long)ys * N, (uint32_t)(nr * N * sizeof(T)), &R.full[s]);
    }
  }
}

// A warp is done with plane g (in stage s); the last of the CTA's warps
// refills s with plane g + S of the same pass (which belongs in the same stage).
// rev: the pass marches the CTA's sequence backwards (plane g is plane
// ptot - 1 - g of the forward sequence).
template <typename T, int NA, bool MOWN = false>
__device__ __forceinline__ void ring_release(const Ring& R, int g, int s, int parity, int ptot, int lane,
                                             bool rev = false) {
  __syncwarp();
  int refill = 0;
  if (lane == 0) {
    __threadfence_block();
    const unsigned prev = atomicAdd(&R.released[s], 1u);
    if (prev == CONSUMER_WARPS - 1u) {
      R.released[s] = 0u;
      refill = g + R.S < ptot && !R.flag[0];
    }
  }
  if (__shfl_sync(0xffffffffu, refill, 0))
    ring_issue_warp<T, NA, MOWN>(R, rev ? ptot - 1 - (g + R.S) : g + R.S, s, parity, lane);
  __syncwarp();
}

__device__ __forceinline__ void ring_wait(const Ring& R, int s, uint32_t par,
                                          unsigned long long limit_ns) {
  if (R.flag[0]) return;
  if (!mbar_wait_bounded(&R.full[s], par, limit_ns)) R.flag[0] = 1;
}

__device__ __forceinline__ void ring_advance(int S, int& s, uint32_t& p) {
  if (++s == S) {
    s = 0;
    p ^= 1u;
  }
}

__device__ __forceinline__ bool last_pass(const PassArgs& P, int pass) { return pass + 1 >= P.npass; }

// This pass's set of partial-sum slots.
__device__ __forceinline__ double* pass_slots(const PassArgs& P, int pass) {
  return P.partials + (size_t)(pass & 1) * NQ * P.nslot;
}

// End of a CTA's run on a lattice (all threads): warp partials of the NUSED
// slots (accumulators acc[0..NACC), slot NQ-1 = non-finite count) into rb, a fixed
// shuffle tree over the warps per quantity into this pass's slots; in the last pass
// also one arrival per quantity on the lattice's count, and the arrival that
// completes it queues the lattice's update.  busy: warps that had any site (the
// others' sums are zero and are not formed).  rb: one of two alternating halves of
// red (a warp can reach the next flush while others still read this one, but not
// the one after, which waits for all).  Returns false if a wait of this CTA had
// timed out.
template <int NACC, int NUSED, typename T>
__device__ __forceinline__ bool ring_flush(const Ring& R, const PassArgs& P, const SegInfo& sg, int pass,
                                           Acc<T> (&acc)[NACC], float& nonfinite, double* red_half, int busy, int warp,
                                           int lane) {
  constexpr int NARRIVE = NUSED > 0 ? NUSED : 1;
  static_assert(sizeof(WarpPart<T>) == sizeof(double), "a warp's part takes one entry of red");
  WarpPart<T>* const rb = reinterpret_cast<WarpPart<T>*>(red_half);
  if (NUSED > 0 && warp < busy) {
#pragma unroll
    for (int k = 0; k < NUSED; ++k) {
      WarpPart<T> v = {};
      if (k < NACC) {
        v = warp_part(acc[k]);
      } else if (k == NQ - 1) {
        float c = nonfinite;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        v = WarpPart<T>{c};
      }
      if (lane == 0) rb[warp * NQ + k] = v;
    }
  }
#pragma unroll
  for (int k = 0; k < NACC; ++k) acc[k].zero();
  nonfinite = 0.f;
  __syncthreads();
  if (R.flag[0]) return false;
  const bool last = last_pass(P, pass);
  if (warp < NARRIVE) {
    double v = 0.0;
    if (NUSED > 0) {
      v = lane < busy ? part_value(rb[lane * NQ + warp]) : 0.0;
#pragma unroll
      for (int o = CONSUMER_WARPS / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    if (lane == 0) {
      if (NUSED > 0) pass_slots(P, pass)[(size_t)warp * P.nslot + sg.slot] = v;
      if (last) {
        __threadfence();
        const unsigned nslot = (unsigned)(sg.slot_end - sg.slot_begin);
        const unsigned prev = atomicAdd(&P.counters[sg.lat], 1u);
        if (prev == NARRIVE * nslot - 1u) R.pend[atomicAdd(const_cast<int*>(&R.flag[3]), 1)] = sg.run;
      }
    }
  }
  if (threadIdx.x == 0) R.flag[2] = sg.lat;
  return true;
}

// Joins pass - 1 and pass of a launch, or starts it (pass 0); all threads.  Waits
// (bounded) until every CTA's writes of the previous pass are done, issues the
// first planes of this pass, one warp per plane, and meanwhile brings the record of
// every lattice of the CTA up to date, lane r mod 32 of the last warp for run r:
//   U::load(P, lattice, record)             pass 0: constants and scalars from global memory;
//   U::ready(P, done, next, record, prep)   before the wait: the weights of the pass whose sums are taken
//                                           and of the next, and what does not depend on the sums;
//   U::update(record, prep, sums, log of the last pass, ...)   with the previous pass's NUSED sums
//                                           (without sums it does not have to wait either);
//   U::coefficients(record, prep, log of this pass)            this pass's coefficients;
//   U::fast_drift, U::fast_powers           both of the latter for alpha = 1, on two warps at once.
// These are out of line and keep their state in shared memory: inlined, they cost the
// marching loop 6 % (registers), and in local memory the update misses L1, which the
// wait drops.  On return every thread may read the records.  False if a wait timed out.
__device__ __forceinline__ double* pass_log(const PassArgs& P, int pass, int lat) {
  return P.log && lat == 0 ? P.log + ADJ_LOG_W * (P.log_base + pass) : nullptr;
}
static __device__ __noinline__ void pass_weights_of(const PassStep* steps, PassStep one, int done, int next,
                                                    TailPrep* q) {
  const PassStep st = steps && done >= 0 ? steps[done] : one;
  const PassStep nx = steps && next >= 0 ? steps[next] : one;
  q->wout = st.wout;
  q->win = st.win;
  q->dnext = st.dnext;
  q->ckn = nx.ck;
  q->dnn = nx.dnext;
}
template <class Rec>
static __device__ __noinline__ void load_run(const LatConst* L, const LatScalars* sc, Rec* r) {
  r->L = *L;
  load_state_cg(r->W, sc);
}
template <typename T, int NA, bool MOWN, int NUSED, class U>
__device__ __forceinline__ bool ring_pass_begin(const Ring& R, const PassArgs& P, int pass, int ns, int ptot,
                                                int parity, bool rev, int warp, int lane) {
  typename U::Rec* const rec = reinterpret_cast<typename U::Rec*>(R.runs);
  TailPrep* const prep = reinterpret_cast<TailPrep*>(R.runs + P.nrun_max * sizeof(typename U::Rec)) + lane;
  const int nruns = R.flag[1];
  const bool mine = warp == CONSUMER_WARPS - 1;
  auto advance = [&](int r) {
    const bool logs = blockIdx.x == 0;
    if (pass > 0)
      U::update(&rec[r], prep, R.red + lane * NQ, logs ? pass_log(P, pass - 1, prep->lat) : nullptr, nullptr, 0);
    U::coefficients(&rec[r], prep, logs ? pass_log(P, pass, prep->lat) : nullptr);
  };
  auto ready = [&](int r) {
    prep->lat = ring_run(R, ns, r).lat;
    if (pass == 0) U::load(P, prep->lat, &rec[r]);
    U::ready(P, pass - 1, pass, &rec[r], prep);
    if (NUSED == 0) advance(r);
  };
  if (mine && lane < nruns) ready(lane);
  if (pass > 0) {
    if (threadIdx.x == 0 && !R.flag[0] && !wait_counter(P.gsync, gridDim.x * (unsigned)pass, P.wait_limit_ns))
      R.flag[0] = 1;
    __syncthreads();
    if (R.flag[0]) return false;
  }
  if (warp < R.S && warp < ptot) {
    if (pass > 0) fence_proxy_async_global();
    ring_issue_warp<T, NA, MOWN>(R, rev ? ptot - 1 - warp : warp, (pass * ptot + warp) % R.S, parity, lane);
  }
  for (int base = 0; base < nruns; base += 32) {
    const int nb = min(32, nruns - base);
    if (pass > 0 && NUSED > 0) {
      ring_slot_sums<NUSED>(R, P, pass - 1, ns, nb, warp, lane, [&](int l) { return base + l; });
      __syncthreads();
    }
    if (mine && lane < nb) {
      if (base > 0) ready(base + lane);
      if (pass > 0 && prep->fast) U::fast_drift(&rec[base + lane], prep, R.red + lane * NQ);
      else if (NUSED > 0) advance(base + lane);
    }
    if (NUSED > 0 && pass > 0) {
      if (base > 0) __syncthreads();  // prep holds these runs'
      if (warp == CONSUMER_WARPS - 2 && lane < nb && prep->fast) {
        const bool logs = blockIdx.x == 0;
        U::fast_powers(&rec[base + lane], prep, R.red + lane * NQ, logs ? pass_log(P, pass - 1, prep->lat) : nullptr,
                       logs ? pass_log(P, pass, prep->lat) : nullptr);
      }
    }
    __syncthreads();
  }
  return true;
}

// End of a pass (all threads): before another pass of the launch, the CTA's writes
// are done and counted; after the last one, the lattices whose arrival count this CTA
// completed are updated and U::store(P, lattice, record) leaves them in global memory.
template <int NUSED, class U>
__device__ __forceinline__ void ring_pass_end(const Ring& R, const PassArgs& P, int pass, int ns, int warp,
                                              int lane) {
  __syncthreads();
  if (!last_pass(P, pass)) {
    if (threadIdx.x == 0) {
      fence_proxy_async_global();
      red_release_inc(P.gsync);
    }
    return;
  }
  typename U::Rec* const rec = reinterpret_cast<typename U::Rec*>(R.runs);
  TailPrep* const prep = reinterpret_cast<TailPrep*>(R.runs + P.nrun_max * sizeof(typename U::Rec)) + lane;
  const int npend = R.flag[3];
  for (int base = 0; base < npend; base += 32) {
    const int nb = min(32, npend - base);
    __threadfence();
    // what the update needs besides the sums, by a warp that has none of the first sums to form
    // (one lane after the sums instead took a single pass 1 to 2 us longer)
    if (warp == 0 && lane < nb) {
      const int r = R.pend[base + lane];
      prep->lat = ring_run(R, ns, r).lat;
      U::ready(P, pass, -1, &rec[r], prep);
    }
    ring_slot_sums<NUSED>(R, P, pass, ns, nb, warp, lane, [&](int l) { return R.pend[base + l]; });
    __syncthreads();
    if (warp == CONSUMER_WARPS - 1 && lane < nb) {
      const int r = R.pend[base + lane], lat = prep->lat;
      if (prep->fast) {
        U::fast_drift(&rec[r], prep, R.red + lane * NQ);
        U::fast_powers(&rec[r], prep, R.red + lane * NQ, pass_log(P, pass, lat), nullptr);
      } else {
        U::update(&rec[r], prep, R.red + lane * NQ, pass_log(P, pass, lat), &P.sc[lat].obs, P.set_rho0);
      }
      U::store(P, lat, &rec[r]);
      P.counters[lat] = 0u;
    }
    __syncthreads();
  }
}

// After a timed-out wait (thread 0): wait, bounded, for copies still in
// flight so that none lands in shared memory after exit, and record it.
__device__ inline void ring_drain(const Ring& R, const PassArgs& P) {
  for (int s = 0; s < R.S; ++s)
    for (int par = 0; par < 2; ++par) mbar_wait_bounded(&R.full[s], (uint32_t)par, 1000000ull);
  P.sc[R.flag[2]].status = CL_ETIMEOUT;
}

}  // namespace clg
