// pass_su2_kd.cu -- the doublet-model pass in kick-then-drift form (without
// self-consistent expansion): the kick of the SU(2) x U(1) doublet model (Sec. 4.3 Hamiltonian
// form in temporal gauge, links, plaquettes and covariant derivatives of the
// U(1) and SU(N) toolkits of Sec. 4.2), and of the lphi4SU2U1 model's singlet
// and U(1)-charged scalar (Sec. 4.5), each site's drift right after its kick.
//
// The equations are those of pass_su2.cu; what differs is where the work is
// done.  Without self-consistent expansion a(eta) is constant or a fixed power
// law, so the drift coefficient of a pass is known before its sums and the
// pass's own drift can follow its kick at each site (kick, then drift by the
// pass's dnext).  The values each site
// goes through are the same as with the drift deferred to the next pass, but
// no neighbour needs to be drifted on read: a stage holds the source buffer's
// raw fields.
//
// Kernel layout.  A work item is a TX x TY tile of x-y sites (32 or 16 wide, 8
// rows; 16 rows for the FP32 lphi4SU2U1 step pass) over a chunk of z-planes
// (su2_work.h); the CTA's items form one sequence of planes (each item adds the
// plane below its chunk) that a three-stage ring of shared memory streams in:
// per plane, every field array's tile rows plus a halo row on each side, each
// row from 16 bytes before the tile to 16 bytes after it, in 16-byte pieces the
// threads copy themselves with cp.async (each thread the same piece of a fixed
// list of arrays, its place on the lattice, periodic in x and y, found once per
// item).  A plane's copies are counted on its stage's "full" mbarrier; every
// warp arrives on the stage's "empty" mbarrier when done with it, and the
// copies of the plane two ahead go into a stage once it is empty: no CTA
// barrier.  Each thread's own momenta of the next plane are copied into a slot
// beside the stages (prefetched into L1 where the slot does not fit).
//
// Each plaquette is formed once per site (xy, xz, yz at n) and serves the
// staples of its links at n directly (P and P^dag); along z it also serves the
// two links it reaches from below, rotated by a link,
//     m(L_iz(n)) = m(U_z^dag(n-z) P_iz(n-z)^dag U_z(n-z)),
// which the thread forms at plane z - 1 and carries to plane z in registers.
// The lower staples across x and y are formed directly at each site (handing
// them on between lanes would leave the tile's edge column to one lane of a
// warp, which costs the whole warp the work).  The same goes for the compact
// U(1) plaquette sines and the backward hops W_i^dag(n-i) psi(n-i): carried
// along z, direct across x and y.  In the FP32 step passes the seven U(1)
// plaquette sines are evaluated two at a time and the six plaquette products and
// four lower staples are formed two at a time, in the packed two-lane FP32 form,
// each lane rounded as the single evaluation (trig2.cuh, Q2 below).
#include "kd_drift.cuh"
#include "su2_kick.cuh"

namespace clg {

namespace {

// Asynchronous copies global -> shared by each thread (cp.async): 16 bytes (both
// addresses 16-byte aligned), or one element; completion either counted on an
// mbarrier (arrive once all of the thread's earlier copies landed) or awaited
// per thread by commit groups.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_el(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_el(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_committed() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Stage geometry: field array f of a stage holds HR = TY + 2 rows (the tile's
// and a halo row each side) of RW elements, from EPC = 16 B before the tile to
// 16 B after it; the tile's site (tx, ty) is element (ty + 1) RW + EPC + tx.
template <typename T, int TX, int TY, bool FULL>
struct KdGeom {
  static constexpr int EPC = 16 / (int)sizeof(T);
  static constexpr int RW = TX + 2 * EPC;
  static constexpr int HR = TY + 2;
  static constexpr int NFA = FULL ? 22 : 19;  // psi (4), A (3), U (12), [phi_s, vphi (2)]
  static constexpr int AE = HR * RW;
  static constexpr size_t STAGE = ((size_t)NFA * AE * sizeof(T) + 127) / 128 * 128;
  // a stage row in 16-byte pieces: NCOL per row, CPA per array
  static constexpr int NCOL = RW / EPC;
  static constexpr int CPA = HR * NCOL;
  // each thread's own momenta of the next plane in a slot after the stages (16
  // arrays, 19 for lphi4SU2U1); the lphi4SU2U1 pass with 8-row tiles, two CTAs
  // per SM, has no room for it and reads its momenta through L1
  static constexpr bool SLOT = !FULL || TY >= 16;
  static constexpr int NM = FULL ? 19 : 16;
  static constexpr size_t MSLOT = SLOT ? ((size_t)NM * TX * TY * sizeof(T) + 127) / 128 * 128 : 0;
  static constexpr size_t SMEM = 3 * STAGE + MSLOT;
};

// stage array f -> state array: psi 0..3, A 8..10, U 14..25, phi_s 35, vphi 37, 38
__device__ __forceinline__ int kd_state_array(int f) {
  return f < 4 ? f : (f < 7 ? f + 4 : (f < 19 ? f + 7 : (f == 19 ? SS : f + 17)));
}

enum : int { KF = 0, KA = 4, KU = 7, KS = 19, KV = 20 };  // stage arrays

}  // namespace

// RED: 0 = no sums, 2 = full measurement (the Friedmann sums of RED 1 are
// only needed with self-consistent expansion).  FULL: the lphi4SU2U1 model.  NC: 0 = the
// lattice size from the lattice constants; > 0 = built for N = NC (every array
// offset a compile-time constant).
template <typename T, int RED, int TX, int TY, bool FULL, int NC = 0>
__global__ void __launch_bounds__(TX * TY, (RED == 2 || sizeof(T) == 8) ? 1 : 2048 / (TX * TY * 4))
    kd_pass_su2(const PassArgs P) {
  using G = KdGeom<T, TX, TY, FULL>;
  constexpr int EPC = G::EPC, RW = G::RW, NFA = G::NFA, AE = G::AE;
  constexpr int nth = TX * TY, NW = nth / 32;
  constexpr bool SLOT = G::SLOT;
  constexpr int NACC = RED == 0 ? 1 : (FULL ? 29 : 23);
  static_assert(RED == 0 || RED == 2, "kick-then-drift passes take no Friedmann sums");
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ double red_s[SU2_NQ][9];
  __shared__ unsigned last_s;
  __shared__ __align__(8) uint64_t full_bar[3];   // per stage: every thread's copies of its plane landed
  __shared__ __align__(8) uint64_t empty_bar[3];  // per stage: every warp done with its plane
  __shared__ volatile int tflag;                   // a wait of this CTA ran out

  const LatConst& L = P.lat[0];
  const int N = NC ? NC : L.N;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int lane = tid & 31, warp = tid >> 5;
  const long long NN = (long long)N * N, V = NC ? (long long)NC * NC * NC : L.V;
  const int parity = P.parity;
  const T* const src = reinterpret_cast<const T*>(L.buf[parity][0]);
  T* const dst = reinterpret_cast<T*>(L.buf[parity ^ 1][0]);
  // array a of the source and destination buffers, indexed by site (V < 2^32)
  auto sa = [&](int a) { return src + (size_t)a * (size_t)V; };
  auto da = [&](int a) { return dst + (size_t)a * (size_t)V; };
  const int ntx = N / TX, ntiles = ntx * (N / TY), nzc = L.su2_nzc, nitems = ntiles * nzc;

  // this pass's drift, after its kick, and the kick's coefficients
  __shared__ Su2Pass<T> coef_s;
  if (warp == NW - 1) {
    double kd64, kdA64;
    ScalarState W;
    load_state_cg(W, P.sc);
    kd_drift_coefficients(L, W, P.dnext, kd64, kdA64);
    su2_coefficients<T>(L, P.sc, P.ck, kd64, kdA64, lane, &coef_s);
  }

  if (tid == 0) {
    for (int s = 0; s < 3; ++s) {
      mbar_init(&full_bar[s], nth);
      mbar_init(&empty_bar[s], NW);
    }
    fence_mbar_init();
    tflag = 0;
  }
  __syncthreads();
  const T kd = coef_s.cd, kdA = coef_s.cdA, hB = coef_s.hB;
  const Su2Coef<T> cf = coef_s.k;

  // The CTA's planes form one sequence of positions (item by item, each item's
  // planes z0 - 1 .. z0 + nz); position p lives in stage p mod 3.  produced: the
  // positions whose copies have gone out; ptot: the positions of the sequence.
  int produced = 0, ptot = 0;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int chunk = it / ntiles;
    ptot += (chunk + 1) * N / nzc - chunk * N / nzc + 2;
  }
  // Each thread copies the same 16-byte piece (column pc, row pr) of a fixed set
  // of arrays of every plane: with room for two sets, the CTA's two halves
  // (warp-uniform) take the first and the second half of the arrays, else the
  // first CPA threads take all of them.  pso: the piece's offset in a plane of the
  // lattice for the producer's current item (periodic in x and y).
  constexpr int NH = 2 * G::CPA <= nth ? 2 : 1, FPH = (NFA + NH - 1) / NH;
  const int ph = tid / (nth / NH), pt = tid - ph * (nth / NH);
  const bool pcopy = pt < G::CPA;
  const int pr = pt / G::NCOL, pc = pt - pr * G::NCOL;
  // the producer's item (CTA-uniform): its z-chunk length and the plane the next
  // position copies (pzp) with its index in the item (pj)
  int pit = blockIdx.x, pnz = 0, pzp = 0, pj = 0;
  unsigned pso = 0u;
  auto producer_item = [&]() {
    if (pit >= nitems) return;
    const int chunk = pit / ntiles, tile = pit - chunk * ntiles;
    const int z0 = chunk * N / nzc;
    pnz = (chunk + 1) * N / nzc - z0;
    const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
    pzp = z0 == 0 ? N - 1 : z0 - 1;
    pj = 0;
    int gx = x0 - EPC + pc * EPC, gy = y0 - 1 + pr;
    gx = gx < 0 ? gx + N : (gx >= N ? gx - N : gx);
    gy = gy < 0 ? gy + N : (gy >= N ? gy - N : gy);
    pso = (unsigned)(gy * N + gx);
  };
  producer_item();
  // The copies of a position go out in two bursts (part 0, then part 1 later in
  // the step, so that a thread's pieces do not queue up at once); after part 1
  // the thread's arrival on the stage's full barrier (once all its copies have
  // landed) and a commit group.
  auto produce = [&](int part) {
    if (pit >= nitems) return;
    const int s = produced % 3;
    if (pcopy) {
      T* const d = reinterpret_cast<T*>(smem + (size_t)s * G::STAGE) + pr * RW + pc * EPC;
      const T* const g = src + (size_t)((unsigned)pzp * (unsigned)NN + pso);
      constexpr int H0 = FPH / 2, H1 = FPH + (NFA - FPH) / 2;
      if (ph == 0 && part == 0) {
#pragma unroll
        for (int f = 0; f < H0; ++f) cp_async16(d + f * AE, g + (size_t)kd_state_array(f) * (size_t)V);
      } else if (ph == 0) {
#pragma unroll
        for (int f = H0; f < FPH; ++f) cp_async16(d + f * AE, g + (size_t)kd_state_array(f) * (size_t)V);
      } else if (part == 0) {
#pragma unroll
        for (int f = FPH; f < H1; ++f) cp_async16(d + f * AE, g + (size_t)kd_state_array(f) * (size_t)V);
      } else {
#pragma unroll
        for (int f = H1; f < NFA; ++f) cp_async16(d + f * AE, g + (size_t)kd_state_array(f) * (size_t)V);
      }
    }
    if (part == 0) return;
    cp_async_arrive(&full_bar[s]);
    cp_async_commit();
    ++produced;
    pzp = pzp + 1 == N ? 0 : pzp + 1;
    if (++pj == pnz + 2) {
      pit += gridDim.x;
      producer_item();
    }
  };
  auto wait_bar = [&](uint64_t* bar, int phase) {
    if (tflag) return;
    if (!mbar_wait_bounded(bar, (uint32_t)(phase & 1), P.wait_limit_ns)) tflag = 1;
  };
  // Step p works on positions p and p + 1: the copies of position p + 2 go out
  // (into the stage position p - 1 held, once every warp is done with it), their
  // first part at the step's beginning, the second (produce(1)) within the step.
  auto step_begin = [&](int p) {
    if (p >= 1) wait_bar(&empty_bar[(p - 1) % 3], (p - 1) / 3);
    if (!tflag) produce(0);
    if (p == 0) wait_bar(&full_bar[0], 0);
    if (p + 1 < ptot) wait_bar(&full_bar[(p + 1) % 3], (p + 1) / 3);
  };
  auto step_end = [&](int p) {
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty_bar[p % 3]);
  };
  for (int k = 0; k < 2; ++k) {
    produce(0);
    produce(1);
  }

  auto stage = [&](int q) { return reinterpret_cast<const T*>(smem + (size_t)(q % 3) * G::STAGE); };
  const int o = (ty + 1) * RW + EPC + tx;
  T* const mslot = reinterpret_cast<T*>(smem + 3 * G::STAGE);
  // a site's neighbourhood (su2_kick.cuh): planes in stages st[0] and st[1], its momenta
  // in the thread's slot or in global memory (prefetched into L1)
  struct Hood {
    const T *c, *p, *src;
    const T* slot;
    unsigned g;
    long long V;
    int o, tid;
    __device__ __forceinline__ T ld(int pl, int f, int dx, int dy) const {
      return (pl ? p : c)[f * AE + o + dy * RW + dx];
    }
    __device__ __forceinline__ Q4<T> ld4(int pl, int f, int dx, int dy) const {
      const T* q = (pl ? p : c) + f * AE + o + dy * RW + dx;
      Q4<T> r;
      r.w = q[0];
      r.x = q[AE];
      r.y = q[2 * AE];
      r.z = q[3 * AE];
      return r;
    }
    __device__ __forceinline__ Q4<T> f(int pl, int dx, int dy) const { return ld4(pl, KF, dx, dy); }
    __device__ __forceinline__ Q4<T> u(int pl, int i, int dx, int dy) const { return ld4(pl, KU + 4 * i, dx, dy); }
    __device__ __forceinline__ T a(int pl, int i, int dx, int dy) const { return ld(pl, KA + i, dx, dy); }
    __device__ __forceinline__ T x(int pl, int k, int dx, int dy) const { return ld(pl, KS + k, dx, dy); }
    // own momentum a (one of SP.., SPA.., SPB.., and for lphi4SU2U1 SPS, SPC..)
    __device__ __forceinline__ T mom(int a) const {
      if constexpr (!SLOT) {
        return __ldg(src + (size_t)a * (size_t)V + g);
      } else {
        const int m =
            a < SPA ? a - SP : (a < SU ? a - SPA + 4 : (a < SS ? a - SPB + 7 : (a == SPS ? 16 : a - SPC + 17)));
        return slot[m * nth + tid];
      }
    }
  };
  auto hood = [&](int pos, unsigned g) { return Hood{stage(pos), stage(pos + 1), src, mslot, g, V, o, tid}; };

  Acc<T> acc[NACC];
#pragma unroll
  for (int k = 0; k < NACC; ++k) acc[k].zero();
  float nonfinite = 0.f;

  Su2Carry<T> carry = {};

  int q = 0;  // position of the item's first plane in the CTA's sequence
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int chunk = it / ntiles, tile = it - chunk * ntiles;
    const int z0 = chunk * N / nzc, nz = (chunk + 1) * N / nzc - z0;
    const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
    const unsigned gown = (unsigned)((y0 + ty) * N + x0 + tx);
    // the momenta of own site g: into the thread's slot, or into L1 where the slot does not fit
    auto prefetch_momenta = [&](unsigned g) {
      if constexpr (SLOT) {
#pragma unroll
        for (int m = 0; m < G::NM; ++m)
          cp_async_el(mslot + m * nth + tid,
                      sa(m < 4 ? SP + m : (m < 7 ? SPA + m - 4 : (m < 16 ? SPB + m - 7 : (m == 16 ? SPS : SPC + m - 17)))) + g);
        cp_async_commit();
      } else {
#pragma unroll
        for (int m = 0; m < 4; ++m) prefetch_l1(sa(SP + m) + g);
#pragma unroll
        for (int m = 0; m < 3; ++m) prefetch_l1(sa(SPA + m) + g);
#pragma unroll
        for (int m = 0; m < 9; ++m) prefetch_l1(sa(SPB + m) + g);
        prefetch_l1(sa(SPS) + g);
        prefetch_l1(sa(SPC) + g);
        prefetch_l1(sa(SPC + 1) + g);
      }
    };

    // ---- the carries for plane z0 from plane z0 - 1 (position q) and z0 (q + 1) ----
    step_begin(q);
    prefetch_momenta((unsigned)z0 * (unsigned)NN + gown);
    su2_carry<T, FULL>(hood(q, 0u), cf, carry);
    if (!tflag) produce(1);
    step_end(q);

    for (int j = 1; j <= nz; ++j) {
      const int z = z0 + j - 1;
      const unsigned g = (unsigned)z * (unsigned)NN + gown;
      if (!SLOT && j < nz) prefetch_momenta(g + (unsigned)NN);
      step_begin(q + j);
      // this plane's momenta (the copies begun just now are not committed yet)
      if constexpr (SLOT) cp_async_wait_committed();
      // the drift of the link fields right after their kick: A_i += kdA pi_A,i, U_i <- exp(-i hB pi_B,i.s) U_i
      auto link = [&](int i, const Q4<T>& Ui, T Ai, T pnA, const T (&pnB)[3]) {
        if (!P.write) return;
        // drift of the link fields: A_i += kdA pi_A,i, U_i <- exp(-i hB pi_B,i.s) U_i
        const T p1 = hB * pnB[0], p2 = hB * pnB[1], p3 = hB * pnB[2];
        T c, sc;
        cos_sinc(p1 * p1 + p2 * p2 + p3 * p3, c, sc);
        Q4<T> e;
        e.w = c;
        e.x = sc * p1;
        e.y = sc * p2;
        e.z = sc * p3;
        Q4<T> u = qmul(e, Ui);
        renorm(u);
        da(SA + i)[g] = fmaT(kdA, pnA, Ai);
        da(SU + 4 * i)[g] = u.w;
        da(SU + 4 * i + 1)[g] = u.x;
        da(SU + 4 * i + 2)[g] = u.y;
        da(SU + 4 * i + 3)[g] = u.z;
        da(SPA + i)[g] = pnA;
#pragma unroll
        for (int a = 0; a < 3; ++a) da(SPB + 3 * i + a)[g] = pnB[a];
      };
      Su2Site<T> site;
      su2_kick<T, RED, FULL>(hood(q + j, g), cf, carry, site, [&]() { if (!tflag) produce(1); }, link);
      if (P.write) {
#pragma unroll
        for (int c2 = 0; c2 < 4; ++c2) {
          da(SF + c2)[g] = fmaT(kd, site.pn[c2], site.fc[c2]);
          da(SP + c2)[g] = site.pn[c2];
        }
        if constexpr (FULL) {
          da(SS)[g] = fmaT(kd, site.pns, site.xs0);
          da(SC)[g] = fmaT(kd, site.pnc0, site.xc0);
          da(SC + 1)[g] = fmaT(kd, site.pnc1, site.xc1);
          da(SPS)[g] = site.pns;
          da(SPC)[g] = site.pnc0;
          da(SPC + 1)[g] = site.pnc1;
        }
      }
      su2_sums<T, RED, FULL>(cf, site, acc, nonfinite);
      if (SLOT && j < nz) prefetch_momenta(g + (unsigned)NN);  // the slot is free again
      step_end(q + j);
    }
    step_begin(q + nz + 1);  // the item's last plane: nothing left to compute on it
    if (!tflag) produce(1);
    step_end(q + nz + 1);
    q += nz + 2;
  }

  __syncthreads();
  if (tflag) {  // a wait ran out: let this thread's copies in flight land, then report
    for (int p = produced > 3 ? produced - 3 : 0; p < produced; ++p)
      mbar_wait_bounded(&full_bar[p % 3], (uint32_t)((p / 3) & 1), 1000000ull);
    if (tid == 0) P.sc->status = CL_ETIMEOUT;
  }
  su2_pass_end<T, RED, FULL>(P, L, acc, nonfinite, red_s, last_s, tid, lane, warp, nth);
}

typedef void (*PassKernel)(const PassArgs);

// Kick-then-drift doublet passes (no self-consistent expansion): red 0 or 2, TX 16 or 32, tiles of
// 8 rows, and (FP32, 32 wide, red 0) of 16 rows with one 512-thread CTA per SM;
// n256: the FP32 32-wide step pass built for N = 256.
PassKernel su2_kd_pass_kernel(int fp32, int red, int TX, int TY, int full, int n256) {
  static const PassKernel tab[2][2][2][2] = {  // [full][TX == 32][fp32][red == 2]
      {{{kd_pass_su2<double, 0, 16, 8, false>, kd_pass_su2<double, 2, 16, 8, false>},
        {kd_pass_su2<float, 0, 16, 8, false>, kd_pass_su2<float, 2, 16, 8, false>}},
       {{kd_pass_su2<double, 0, 32, 8, false>, kd_pass_su2<double, 2, 32, 8, false>},
        {kd_pass_su2<float, 0, 32, 8, false>, kd_pass_su2<float, 2, 32, 8, false>}}},
      {{{kd_pass_su2<double, 0, 16, 8, true>, kd_pass_su2<double, 2, 16, 8, true>},
        {kd_pass_su2<float, 0, 16, 8, true>, kd_pass_su2<float, 2, 16, 8, true>}},
       {{kd_pass_su2<double, 0, 32, 8, true>, kd_pass_su2<double, 2, 32, 8, true>},
        {kd_pass_su2<float, 0, 32, 8, true>, kd_pass_su2<float, 2, 32, 8, true>}}}};
  if ((red != 0 && red != 2) || (TX != 16 && TX != 32)) return nullptr;
  if (n256 && (!fp32 || TX != 32 || red != 0)) return nullptr;
  if (TY == 16) {
    if (!fp32 || TX != 32 || red != 0) return nullptr;
    if (n256) return full ? kd_pass_su2<float, 0, 32, 16, true, 256> : kd_pass_su2<float, 0, 32, 16, false, 256>;
    return full ? kd_pass_su2<float, 0, 32, 16, true> : kd_pass_su2<float, 0, 32, 16, false>;
  }
  if (n256 && TY == 8) return full ? kd_pass_su2<float, 0, 32, 8, true, 256> : kd_pass_su2<float, 0, 32, 8, false, 256>;
  if (TY != 8) return nullptr;
  return tab[full ? 1 : 0][TX == 32 ? 1 : 0][fp32 ? 1 : 0][red == 2 ? 1 : 0];
}

// Dynamic shared memory of a kick-then-drift pass: three stages and the momentum slot.
size_t su2_kd_smem_bytes(int TX, int TY, int esz, int full) {
  if (TY == 16) return full ? KdGeom<float, 32, 16, true>::SMEM : KdGeom<float, 32, 16, false>::SMEM;
  if (TX == 32) {
    if (esz == 4) return full ? KdGeom<float, 32, 8, true>::SMEM : KdGeom<float, 32, 8, false>::SMEM;
    return full ? KdGeom<double, 32, 8, true>::SMEM : KdGeom<double, 32, 8, false>::SMEM;
  }
  if (esz == 4) return full ? KdGeom<float, 16, 8, true>::SMEM : KdGeom<float, 16, 8, false>::SMEM;
  return full ? KdGeom<double, 16, 8, true>::SMEM : KdGeom<double, 16, 8, false>::SMEM;
}

}  // namespace clg
