// pass_scalar.cu -- fused drift + kick pass for real scalar singlets
// (CosmoLattice manual, Sec. 3.5.2, Hamiltonian form):
//
//   drift (deferred from the previous pass):  phi += cd * pi,   cd = h abar^{alpha-3}
//   kick:   pi += c_k [ a^{1+alpha} Lap phi - a^{3+alpha} V_{,phi} ]
//   Lap phi = sum_i [phi(n+i) - 2 phi(n) + phi(n-i)] / dx^2       (eqs. neutrald, forwardbackwardd)
//   sums:   sum pi^2 before / after the kick, sum_i (grad^+_i phi)^2 (as -sum phi Lap phi
//           in the Friedmann passes), sum V (+ means in measurement passes)
//
// One pass per integrator stage: each field and momentum array is read once
// from HBM and written once.  A CTA owns runs of (y-tile, z-plane) tasks
// ("segments"): BY full x-rows marched along z.  Its segments form one
// continuous sequence of planes (each segment adds a halo plane at both
// ends); every plane tile (plus one halo row on each side in y) of every
// array streams into a ring of shared-memory stages by 1-D bulk async copies
// (TMA), completion counted on the stage's mbarrier.  The 16 warps never meet
// at a block barrier while marching: each waits for the stage it needs,
// applies the drift in registers as it reads (z-neighbours and the thread's own
// sites stay in registers, y-neighbours and the x-neighbours beyond its own sites
// come from the stage), kicks, stores, and releases the stage; the last warp to
// release a stage (shared memory count) issues the copies of the plane S places
// further in the sequence, so the ring runs on across segment boundaries.  FP32
// sums are formed per plane and added once per plane to compensated accumulators,
// FP64 sums site by site to plain ones, and flushed once per run into the run's
// slot; between two passes every CTA sums its lattices' slots in a fixed order
// and runs their Friedmann update itself (ring.cuh, tail.cuh).
//
// FP64 storage is bound by its FP64 operations (64 cycles a warp and operation; memory
// takes 97 of a 216^3 two-field pass's 380 us): 18 a field pair and site (35 before),
// with the Laplacian in integers (fix_lap.h), each site drifted once and shared through
// the stage, each sum one FMA, and the potential from factors the force needs anyway.
// The warps wait for each other's drifted plane a whole plane after writing theirs (a
// block barrier per plane left the unit idle a fifth of the time: 457 us a pass).
// 216^3, two fields, 5 VV4 steps and energies: 12340 us before, 10630 with a Laplacian
// whose FP64 form for values out of range was issued predicated, 7880 with that in a
// branch, 6590 with the deferred wait.
#include "common.cuh"
#include "ring.cuh"
#include "tail.cuh"
#include "fix_lap.h"

namespace clg {

// Program potentials (eq. PotNat): NF = 1: phi^4/4; NF = 2: phi^4/4 + (q/2) phi^2 chi^2.
template <int NF> struct ScalarPot;
template <> struct ScalarPot<1> {
  static constexpr int NPOT = 1;
  template <typename T>
  __device__ __forceinline__ static T total(const T (&f)[1], T hq) {
    const T f2 = f[0] * f[0];
    return T(0.25) * f2 * f2;
  }
  template <typename T>
  __device__ __forceinline__ static void eval(const T (&f)[1], T q, T (&d)[1], T (&t)[1]) {
    const T f2 = f[0] * f[0];
    d[0] = f2 * f[0];
    t[0] = T(0.25) * f2 * f2;
  }
  // FP64: the kicked momentum (k: momentum and Laplacian part), -A3 V_{,f} added, and the
  // potential's terms as products of two factors, w[t][0] w[t][1] x scale[t]
  __device__ __forceinline__ static void kick64(const double (&f)[1], double A3, double, double, const double (&k)[1],
                                                double (&pn)[1], double (&w)[1][2], double (&tot)[2]) {
    const double f2 = f[0] * f[0];
    pn[0] = fma(-A3, f2 * f[0], k[0]);
    w[0][0] = w[0][1] = tot[0] = tot[1] = f2;
  }
  __device__ __forceinline__ static double scale(int, double) { return 0.25; }
  static constexpr double kTotalScale = 0.25;
};
template <> struct ScalarPot<2> {
  static constexpr int NPOT = 2;
  // phi^4/4 + (q/2) phi^2 chi^2 = p2 (p2/4 + (q/2) c2), hq = q/2
  template <typename T>
  __device__ __forceinline__ static T total(const T (&f)[2], T hq) {
    const T p2 = f[0] * f[0], c2 = f[1] * f[1];
    return p2 * fmaT(T(0.25), p2, hq * c2);
  }
  template <typename T>
  __device__ __forceinline__ static void eval(const T (&f)[2], T q, T (&d)[2], T (&t)[2]) {
    const T p2 = f[0] * f[0], c2 = f[1] * f[1];
    d[0] = p2 * f[0] + q * f[0] * c2;
    d[1] = q * p2 * f[1];
    t[0] = T(0.25) * p2 * p2;
    t[1] = T(0.5) * q * p2 * c2;
  }
  // V = (1/2) p2 (s - p2/2) with s = p2 + q c2, the factor of phi in the force
  __device__ __forceinline__ static void kick64(const double (&f)[2], double A3, double q, double A3q,
                                                const double (&k)[2], double (&pn)[2], double (&w)[2][2],
                                                double (&tot)[2]) {
    const double p2 = f[0] * f[0], c2 = f[1] * f[1];
    const double s = fma(q, c2, p2);
    pn[0] = fma(-A3, f[0] * s, k[0]);
    pn[1] = fma(-(A3q * p2), f[1], k[1]);
    w[0][0] = w[0][1] = w[1][0] = p2;
    w[1][1] = c2;
    tot[0] = p2;
    tot[1] = fma(-0.5, p2, s);
  }
  __device__ __forceinline__ static double scale(int t, double q) { return t == 0 ? 0.25 : 0.5 * q; }
  static constexpr double kTotalScale = 0.5;
};

template <typename T, int VX>
__device__ __forceinline__ void ld_vec(T (&v)[VX], const T* p) {
  *reinterpret_cast<typename V16<T>::type*>(v) = *reinterpret_cast<const typename V16<T>::type*>(p);
}
template <typename T, int VX>
__device__ __forceinline__ void st_vec(T* p, const T (&v)[VX]) {
  *reinterpret_cast<typename V16<T>::type*>(p) = *reinterpret_cast<const typename V16<T>::type*>(v);
}

// z of plane j of a segment (j = 0 and nz + 1 are its halo planes), marched in direction dir
__device__ __forceinline__ int seg_plane_z(int z0, int nz, int N, int dir, int j) {
  const int z = dir > 0 ? z0 - 1 + j : z0 + nz - j;
  return z < 0 ? z + N : (z >= N ? z - N : z);
}

// The Friedmann update of a lattice between two passes and its coefficients in the
// next (ring_pass_begin, ring_pass_end).
template <typename T, int NF, int RED>
struct ScalarUpdate {
  static constexpr int NPOT = ScalarPot<NF>::NPOT;
  typedef LatRun<T, 4> Rec;  // cf: drift coefficient, c_k a^{1+alpha}/dx^2, c_k a^{3+alpha}, q

  __device__ __forceinline__ static void load(const PassArgs& P, int lat, Rec* r) {
    load_run(&P.lat[lat], &P.sc[lat], r);
    r->cf[3] = (T)r->L.q;
  }
  __device__ __forceinline__ static void ready(const PassArgs& P, int done, int next, Rec* r, TailPrep* q) {
    pass_weights_of(P.steps, PassStep{P.ck, P.wout, P.win, P.dnext}, done, next, q);
    if (done >= 0) prepare(r, q, P.log != nullptr);
  }
  // k: E_K per sum of pi^2, E_G per sum (grad^+ phi)^2
  __device__ __noinline__ static void prepare(const Rec* r, TailPrep* q, bool logged) {
    const LatPar& L = r->L;
    const bool self = RED > 0 && L.expansion == CL_EXP_SELF;
    q->fast = 0;
    if (RED == 1 && self && L.int_alpha && L.alpha_i == 1) {
      alpha1_ready(L, r->W, q);
      if (!logged) return;
    }
    const double a = r->W.a, ia2 = 1.0 / (a * a);
    q->k[0] = 0.5 * L.inv_V * (ia2 * ia2 * ia2);
    q->k[1] = 0.5 * L.inv_V * L.inv_dx2 * ia2;
    if (self) q->pref = kernel_a_pref(L, a);
  }
  // slot 1 holds sum phi Lap phi = -sum (grad^+ phi)^2
  __device__ __noinline__ static void fast_drift(Rec* r, const TailPrep* q, const double* sum) {
    alpha1_drift(r->W, q, alpha1_b(q->kick, sum[0], -sum[1], sum[2]));
    r->cf[0] = (T)r->W.cd;
    r->W.pi2 = sum[0];
  }
  __device__ __noinline__ static void fast_powers(Rec* r, const TailPrep* q, const double* sum, double* lgd,
                                                  double* lg) {
    alpha1_powers(r->W, q, alpha1_b(q->kick, sum[0], -sum[1], sum[2]));
    const double A1 = (q->ckn * r->L.inv_dx2) * r->W.apow1, A3 = q->ckn * r->W.apow3;
    r->cf[1] = (T)A1;
    r->cf[2] = (T)A3;
    if (lgd) {  // an adjoint sweep's log of the pass that is done, and of the one that starts
      const PassStep st = {0.0, q->wout, q->win, q->dnext};
      PassSums E = {0, 0, 0, 0, 0, 0, 0};
      E.EKpre = q->pi2 * q->k[0];
      E.EKpost = sum[0] * q->k[0];
      E.EG = -sum[1] * q->k[1];
      E.EV = sum[2] * r->L.inv_V;
      lgd[5] = kernel_a_da(st, r->L, q->a, E);
    }
    if (!lg) return;
    // the drift coefficient that fast_drift writes at the same time, formed alike
    const double abar = fma(0.5 * q->dnext, alpha1_b(q->kick, sum[0], -sum[1], sum[2]), q->a);
    lg[0] = q->dnext == 0.0 ? 0.0 : q->dnext / (abar * abar);
    lg[1] = q->ckn;
    lg[2] = A1;
    lg[3] = A3;
    lg[4] = r->W.a;
  }
  // the scalars after the pass with these sums; lg: its log; o: where a measurement goes
  __device__ __noinline__ static void update(Rec* r, const TailPrep* q, const double* sum, double* lg,
                                             cl_energies_t* o, int set_rho0) {
    const LatPar& L = r->L;
    const PassStep st = {0.0, q->wout, q->win, q->dnext};
    const double ck = q->k[0], cg = q->k[1];
    ScalarState W = r->W;
    const bool self = RED > 0 && L.expansion == CL_EXP_SELF;
    PassSums E = {0, 0, 0, 0, 0, 0, 0};
    if (RED > 0) {
      double spre = 0, spost = 0, gg = 0, vs = 0;
      if (RED == 1) {
        // slot 1 holds sum phi Lap phi = -sum (grad^+ phi)^2
        spre = W.pi2; spost = sum[0]; gg = -sum[1]; vs = sum[2];
      } else {
        for (int f = 0; f < NF; ++f) {
          spre += sum[6 * f]; spost += sum[6 * f + 1]; gg += sum[6 * f + 2];
        }
        for (int t = 0; t < NPOT; ++t) vs += sum[6 * NF + t];
      }
      E.EKpre = spre * ck;
      W.pi2 = spost;
      E.EKpost = spost * ck;
      E.EG = gg * cg;
      E.EV = vs * L.inv_V;
    }
    if (self) W.b = friedmann_kicks_scalar(friedmann_pre(L, q->pref, st.wout, st.win), E, W.b);
    if (lg) lg[5] = self ? kernel_a_da(st, L, W.a, E) : 0.0;
    if (RED == 2 && o) {
      for (int k = 0; k < 4; ++k) {
        o->EK[k] = o->EG[k] = o->EV[k] = 0.0;
        o->mean_phi[k] = o->mean_phi2[k] = o->mean_pi[k] = o->mean_pi2[k] = 0.0;
      }
      o->EKA = o->EGA = 0.0;
      for (int f = 0; f < NF; ++f) {
        o->EK[f] = sum[6 * f + 1] * ck;
        o->EG[f] = sum[6 * f + 2] * cg;
        o->mean_phi[f] = sum[6 * f + 3] * L.inv_V;
        o->mean_phi2[f] = sum[6 * f + 4] * L.inv_V;
        o->mean_pi[f] = sum[6 * f + 5] * L.inv_V;
        o->mean_pi2[f] = sum[6 * f + 1] * L.inv_V;
      }
      for (int t = 0; t < NPOT; ++t) o->EV[t] = sum[6 * NF + t] * L.inv_V;
      o->nonfinite = (int64_t)sum[NQ - 1];
      finish_obs(set_rho0, L, W, *o);
    }
    advance_drift(st.dnext, L, W);
    r->W = W;
  }
  // lg: the log of the pass that starts, for an adjoint sweep
  __device__ __noinline__ static void coefficients(Rec* r, const TailPrep* q, double* lg) {
    const double A1 = (q->ckn * r->L.inv_dx2) * r->W.apow1, A3 = q->ckn * r->W.apow3;
    r->cf[0] = (T)r->W.cd;
    r->cf[1] = (T)A1;
    r->cf[2] = (T)A3;
    if (lg) {
      lg[0] = r->W.cd;
      lg[1] = q->ckn;
      lg[2] = A1;
      lg[3] = A3;
      lg[4] = r->W.a;
    }
  }
  __device__ __forceinline__ static void store(const PassArgs& P, int lat, const Rec* r) { put(&P.sc[lat], r); }
  __device__ __noinline__ static void put(LatScalars* to, const Rec* r) { store_state(to, r->W); }
};

// RED: 0 = no sums, 1 = sums for the Friedmann kick, 2 = full measurement (one-pass
// launches only).  P.npass > 1: several passes in one cooperative launch
// (ring_pass_begin, ring_pass_end).
template <typename T, int NF, int RED>
__global__ void __launch_bounds__(THREADS, 1) dk_pass_scalar(const __grid_constant__ PassArgs P) {
  constexpr int VX = V16<T>::n;
  constexpr int NA = 2 * NF;
  constexpr int NPOT = ScalarPot<NF>::NPOT;
  constexpr bool FP64 = sizeof(T) == 8;
  // RED = 1 sums: pi^2 after the kick, phi Lap phi (= -(grad^+ phi)^2 summed), V.  The pre-kick sum of
  // pi^2 is the previous kick's post-kick sum (a drift leaves pi unchanged),
  // carried in the lattice scalars.
  constexpr int NACC = RED == 0 ? 1 : (RED == 1 ? 3 : 6 * NF + NPOT);
  // slots a pass reduces: the Friedmann sums, or every measured sum plus the
  // non-finite count (slot NQ - 1)
  constexpr int NUSED = RED == 0 ? 0 : (RED == 1 ? 3 : NQ);

  extern __shared__ __align__(128) unsigned char smem[];
  const Ring R = ring_view(smem, P);
  const int S = R.S;
  volatile int* const flag = R.flag;
  const int* const off = R.off;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sb = P.cta_seg[blockIdx.x], ns = P.cta_seg[blockIdx.x + 1] - sb;
  if (tid == 0) ring_setup<NA>(R, P, sb, ns);
  __syncthreads();
  const int ptot = off[ns];
  int parity = P.parity;
  // passes reading buffer 1 march the CTA's sequence backwards (plane g is
  // plane ptot-1-g of the forward sequence: segments in reverse order, each
  // marched the other way), so that a pass starts on the planes the previous
  // pass wrote last, while they are still in L2
  bool rev = false;

  typedef ScalarUpdate<T, NF, RED> Update;
  const typename Update::Rec* const rec = reinterpret_cast<const typename Update::Rec*>(R.runs);
  auto release = [&](int g, int s) { ring_release<T, NA>(R, g, s, parity, ptot, lane, rev); };
  auto wait_full = [&](int s, uint32_t par) { ring_wait(R, s, par, P.wait_limit_ns); };
  auto stage_ptr = [&](int s) -> const T* { return ring_stage<T>(R, s); };

  // stage and full-barrier phase of the current plane, advanced without divisions
  int s_cur = 0;
  uint32_t p_cur = 0u;
  auto advance = [&](int& s, uint32_t& p) {
    if (++s == S) {
      s = 0;
      p ^= 1u;
    }
  };

  Acc<T> acc[NACC];
  float nonfinite = 0.f;
  int fbuf = 0;
  uint32_t p_drifted = 0u;  // phase of the shared planes' mbarrier (FP64)
#pragma unroll
  for (int k = 0; k < NACC; ++k) acc[k].zero();

  for (int pass = 0; pass < P.npass; ++pass) {
    parity = P.parity ^ (pass & 1);
    rev = parity != 0;
    if (!ring_pass_begin<T, NA, false, NUSED, Update>(R, P, pass, ns, ptot, parity, rev, warp, lane)) goto timeout;
    // a measurement's 14 sums start here, so that they need no registers during the pass's
    // begin, and a plane's output pointer is formed at its stores: spilled otherwise, and 128^3
    // FP32 took 48 us instead of 41, 256^3 145 instead of 138 (FP64 144^3 260, 250)
    if constexpr (RED == 2) {
#pragma unroll
      for (int k = 0; k < NACC; ++k) acc[k].zero();
      nonfinite = 0.f;
    }

    for (int ii = 0; ii < ns; ++ii) {
      const int i = rev ? ns - 1 - ii : ii;
      const SegInfo& si = R.info[i];
      // the last segment of a run on a lattice, in this pass's order
      const bool run_end = rev ? (i == 0 || R.info[i - 1].run != si.run) : si.flush != 0;
      const int dir = rev ? -si.dir : si.dir, nz = si.nz;
      const int N = si.N, BY = si.rows - 2, TX = N / VX;
      const int tx = tid % TX, ty = tid / TX;
      const bool active = ty < BY;  // active threads are 0 .. TX*BY-1
      const int x0 = tx * VX;
      const int y = si.ylo + ty;
      const int arr_elems = (BY + 2) * N;
      const long long NN = (long long)N * N;
      const int g0 = rev ? ptot - off[i + 1] : off[i];
      const T cd = rec[si.run].cf[0], A1 = rec[si.run].cf[1], A3 = rec[si.run].cf[2], q = rec[si.run].cf[3];
      const T hq = T(0.5) * q, A3q = A3 * q;
      const bool drifting = cd != T(0);
      const int own = (ty + 1) * N + x0;
      const int exl = (ty + 1) * N + (x0 == 0 ? N - 1 : x0 - 1), exr = (ty + 1) * N + (x0 + VX == N ? 0 : x0 + VX);

      // own values of a stage, drifted: phi + cd * pi
      auto read_own = [&](const T* st, T (&ph)[NF][VX]) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          ld_vec<T, VX>(ph[f], st + (size_t)(2 * f) * arr_elems + own);
          if (drifting) {
            T pm[VX];
            ld_vec<T, VX>(pm, st + (size_t)(2 * f + 1) * arr_elems + own);
#pragma unroll
            for (int v = 0; v < VX; ++v) ph[f][v] = fmaT(cd, pm[v], ph[f][v]);
          }
        }
      };

      // FP64 (bound by its arithmetic, not by memory): a site's drifted fields are
      // formed once and written back into its stage, where the next plane reads
      // them as y- and x-neighbours; the tile's two halo rows are drifted in place, by
      // the warps without sites where these then have no more FP64 operations than the
      // others (18 a field: 16 elements a lane), else by all; then a proxy fence (bulk
      // copies refill the stage later) and one arrival per warp on an mbarrier, which the
      // warps wait for one plane's kick later.  `drifting` is the same in every thread
      // of the CTA.
      constexpr bool SHARE = FP64;
      const int busy = (TX * BY + 31) & ~31;  // threads of warps with sites
      const bool idle_halo = SHARE && 16 * (THREADS - busy) >= 2 * N;
      const bool share = SHARE && drifting;
      auto share_own = [&](int s, const T (&ph)[NF][VX]) {  // active threads
        T* st = reinterpret_cast<T*>(smem + (size_t)s * P.stage_bytes_max);
#pragma unroll
        for (int f = 0; f < NF; ++f) st_vec<T, VX>(st + (size_t)(2 * f) * arr_elems + own, ph[f]);
      };
      auto share_halo = [&](int s) {  // every thread of the CTA
        if (!flag[0]) {
          T* st = reinterpret_cast<T*>(smem + (size_t)s * P.stage_bytes_max);
          for (int k = idle_halo ? (tid < busy ? 2 * N : tid - busy) : tid; k < 2 * N;
               k += idle_halo ? THREADS - busy : THREADS) {
            const int e = k < N ? k : (BY + 1) * N + (k - N);
#pragma unroll
            for (int f = 0; f < NF; ++f) {
              T* ph = st + (size_t)(2 * f) * arr_elems;
              ph[e] = fmaT(cd, st[(size_t)(2 * f + 1) * arr_elems + e], ph[e]);
            }
          }
          fence_proxy_async_smem();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(R.drifted);
      };
      auto share_wait = [&]() {  // the values shared last are all written
        if (!flag[0] && !mbar_wait_bounded(R.drifted, p_drifted, P.wait_limit_ns)) flag[0] = 1;
        p_drifted ^= 1u;
      };

      // drifted fields of three consecutive planes; the roles below / current /
      // above rotate through b0, b1, b2 (the march is unrolled by three, so the
      // rotation costs no register moves)
      T b0[NF][VX], b1[NF][VX], b2[NF][VX];
      // planes 0 and 1 of the segment
      wait_full(s_cur, p_cur);
      if (active && !flag[0]) read_own(stage_ptr(s_cur), b0);
      release(g0, s_cur);
      advance(s_cur, p_cur);
      wait_full(s_cur, p_cur);
      if (active && !flag[0]) {
        read_own(stage_ptr(s_cur), b1);
        if (share) share_own(s_cur, b1);
      }
      if (share) share_halo(s_cur);
      int s_nxt = s_cur;
      uint32_t p_nxt = p_cur;
      advance(s_nxt, p_nxt);

      // plane j of the segment (stage s_cur), its neighbours below and above
      // (the above plane is read from stage s_nxt into `above`)
      auto plane = [&](int j, const T (&below)[NF][VX], const T (&cur)[NF][VX], T (&above)[NF][VX]) {
        wait_full(s_nxt, p_nxt);
        if (share) share_wait();
        const bool go = active && !flag[0];
        if (go) read_own(stage_ptr(s_nxt), above);
        if (share && j < nz) {
          if (go) share_own(s_nxt, above);
          share_halo(s_nxt);
        }
        if (go) {
          const T* sc = stage_ptr(s_cur);
          T lap[NF][VX], g2[VX];
          bool in_range = true;  // FP64: the integer form holds
#pragma unroll
          for (int v = 0; v < VX; ++v) g2[v] = T(0);
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            const T* ph = sc + (size_t)(2 * f) * arr_elems;
            const T* pm = sc + (size_t)(2 * f + 1) * arr_elems;
            T yl[VX], yh[VX];
            ld_vec<T, VX>(yl, ph + ty * N + x0);
            ld_vec<T, VX>(yh, ph + (ty + 2) * N + x0);
            if (drifting && !SHARE) {
              T ml[VX], mh[VX];
              ld_vec<T, VX>(ml, pm + ty * N + x0);
              ld_vec<T, VX>(mh, pm + (ty + 2) * N + x0);
#pragma unroll
              for (int v = 0; v < VX; ++v) {
                yl[v] = fmaT(cd, ml[v], yl[v]);
                yh[v] = fmaT(cd, mh[v], yh[v]);
              }
            }
            // x-neighbours beyond this thread's sites, read from the stage and
            // drifted like the owner's copy (no shuffle, no divergent edge branch)
            const T left = drifting && !SHARE ? fmaT(cd, pm[exl], ph[exl]) : ph[exl];
            const T right = drifting && !SHARE ? fmaT(cd, pm[exr], ph[exr]) : ph[exr];
            T gf = T(0);
#pragma unroll
            for (int v = 0; v < VX; ++v) {
              const T c = cur[f][v];
              const T xl = v == 0 ? left : cur[f][v - 1];
              const T xr = v == VX - 1 ? right : cur[f][v + 1];
              const T zl = below[f][v], zh = above[f][v];
              if constexpr (sizeof(T) == 8) {
                bool ok;
                lap[f][v] = fix_lap(fix_val(xl), fix_val(xr), fix_val(yl[v]), fix_val(yh[v]), fix_val(zl), fix_val(zh),
                                    fix_val(c), &ok);
                in_range = in_range && ok;
              } else {
                // FP32 keeps each direction's small difference from its own pair sum
                lap[f][v] = ((xl + xr) - T(2) * c) + ((yl[v] + yh[v]) - T(2) * c) +
                            ((zl + zh) - T(2) * c);
              }
              if (RED == 2) {  // forward differences (eq. EK_EG_EV with grad^+)
                const T zp = dir > 0 ? zh : zl;
                const T gx = xr - c, gy = yh[v] - c, gz = zp - c;
                if constexpr (FP64)
                  acc[6 * f + 2].s = fma(gz, gz, fma(gy, gy, fma(gx, gx, acc[6 * f + 2].s)));
                else
                  gf += gx * gx + gy * gy + gz * gz;
              } else if (RED == 1) {
                // sum_n (grad^+ phi)^2 = -sum_n phi Lap phi (summation by parts on the
                // periodic lattice): one FMA on the Laplacian the kick needs anyway
                if constexpr (!FP64) g2[v] = fmaT(c, lap[f][v], g2[v]);
              }
            }
            if constexpr (RED == 2 && !FP64) acc[6 * f + 2].add(gf);
          }
          if constexpr (FP64) {
            // the thread's sites again, in FP64 (one block of all of them: a branch, where a
            // short one would be issued predicated and take its time on the FP64 unit)
            if (!in_range) {
#pragma unroll
              for (int f = 0; f < NF; ++f) {
                const T* ph = sc + (size_t)(2 * f) * arr_elems;
                T yl[VX], yh[VX];
                ld_vec<T, VX>(yl, ph + ty * N + x0);
                ld_vec<T, VX>(yh, ph + (ty + 2) * N + x0);
#pragma unroll
                for (int v = 0; v < VX; ++v)
                  lap[f][v] = fp64_lap(v == 0 ? ph[exl] : cur[f][v - 1], v == VX - 1 ? ph[exr] : cur[f][v + 1], yl[v],
                                       yh[v], below[f][v], above[f][v], cur[f][v]);
              }
            }
          }
          T pn[NF][VX], pic[NF][VX];  // momenta of the current plane, from its stage
#pragma unroll
          for (int f = 0; f < NF; ++f) ld_vec<T, VX>(pic[f], sc + (size_t)(2 * f + 1) * arr_elems + own);
          if constexpr (FP64) {
            // every sum one FMA into its accumulator (FP32 adds a plane's terms first)
#pragma unroll
            for (int v = 0; v < VX; ++v) {
              double fv[NF], k[NF], p[NF], w[NPOT][2], tot[2];
#pragma unroll
              for (int f = 0; f < NF; ++f) {
                fv[f] = cur[f][v];
                k[f] = fma(A1, lap[f][v], pic[f][v]);
              }
              ScalarPot<NF>::kick64(fv, A3, q, A3q, k, p, w, tot);
#pragma unroll
              for (int f = 0; f < NF; ++f) {
                pn[f][v] = p[f];
                if constexpr (RED == 1) {
                  acc[0].s = fma(p[f], p[f], acc[0].s);
                  acc[1].s = fma(fv[f], lap[f][v], acc[1].s);
                }
                if constexpr (RED == 2) {
                  acc[6 * f + 0].s = fma(pic[f][v], pic[f][v], acc[6 * f + 0].s);
                  acc[6 * f + 1].s = fma(p[f], p[f], acc[6 * f + 1].s);
                  acc[6 * f + 3].s += fv[f];
                  acc[6 * f + 4].s = fma(fv[f], fv[f], acc[6 * f + 4].s);
                  acc[6 * f + 5].s += p[f];
                  // (an FP64 comparison would be one more operation on that unit)
                  if ((__double2hiint(p[f]) & 0x7ff00000) == 0x7ff00000) nonfinite += 1.f;
                }
              }
              if constexpr (RED == 1) acc[2].s = fma(tot[0], tot[1], acc[2].s);
              if constexpr (RED == 2) {
#pragma unroll
                for (int t = 0; t < NPOT; ++t) acc[6 * NF + t].s = fma(w[t][0], w[t][1], acc[6 * NF + t].s);
              }
            }
          } else {
            T spost = T(0), vs = T(0), gsum = T(0);
#pragma unroll
            for (int v = 0; v < VX; ++v) {
              T fv[NF], dv[NF], tv[NPOT];
#pragma unroll
              for (int f = 0; f < NF; ++f) fv[f] = cur[f][v];
              ScalarPot<NF>::eval(fv, q, dv, tv);
#pragma unroll
              for (int f = 0; f < NF; ++f) {
                // the small increment last: one rounding at the momentum's size
                pn[f][v] = pic[f][v] + (A1 * lap[f][v] - A3 * dv[f]);
              }
              if (RED == 1) {
#pragma unroll
                for (int f = 0; f < NF; ++f) spost = fmaT(pn[f][v], pn[f][v], spost);
                vs += ScalarPot<NF>::total(fv, hq);
                gsum += g2[v];
              } else if (RED == 2) {
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                  acc[6 * f + 0].add(pic[f][v] * pic[f][v]);
                  acc[6 * f + 1].add(pn[f][v] * pn[f][v]);
                  acc[6 * f + 3].add(fv[f]);
                  acc[6 * f + 4].add(fv[f] * fv[f]);
                  acc[6 * f + 5].add(pn[f][v]);
                  if (!isfinite(pn[f][v])) nonfinite += 1.f;
                }
#pragma unroll
                for (int t = 0; t < NPOT; ++t) acc[6 * NF + t].add(tv[t]);
              }
            }
            if (RED == 1) {
              acc[0].add(spost);
              acc[1].add(gsum);
              acc[2].add(vs);
            }
          }
          if (P.write) {
            T* const out = static_cast<T*>(const_cast<void*>(si.src[parity ^ 1][0])) +
                           (long long)seg_plane_z(si.z0, nz, N, dir, j) * NN + (long long)y * N + x0;
            const long long Vs = si.V;
#pragma unroll
            for (int f = 0; f < NF; ++f) {
              st_vec<T, VX>(out + (2 * f) * Vs, cur[f]);
              st_vec<T, VX>(out + (2 * f + 1) * Vs, pn[f]);
            }
          }
        }
        release(g0 + j, s_cur);
        s_cur = s_nxt;
        p_cur = p_nxt;
        advance(s_nxt, p_nxt);
      };
      for (int j = 1; j <= nz; j += 3) {
        plane(j, b0, b1, b2);
        if (j + 1 > nz) break;
        plane(j + 1, b1, b2, b0);
        if (j + 2 > nz) break;
        plane(j + 2, b2, b0, b1);
      }
      release(g0 + nz + 1, s_cur);
      advance(s_cur, p_cur);

      if (!run_end) continue;

      if constexpr (FP64) {  // the potential's sums were kept without their constant factors
        if constexpr (RED == 1) acc[2].s *= ScalarPot<NF>::kTotalScale;
        if constexpr (RED == 2) {
#pragma unroll
          for (int t = 0; t < NPOT; ++t) acc[6 * NF + t].s *= ScalarPot<NF>::scale(t, q);
        }
      }
      double* rb = R.red + fbuf * CONSUMER_WARPS * NQ;
      fbuf ^= 1;
      if (!ring_flush<NACC, NUSED>(R, P, si, pass, acc, nonfinite, rb, (TX * BY + 31) >> 5, warp, lane)) goto timeout;
    }
    ring_pass_end<NUSED, Update>(R, P, pass, ns, warp, lane);
  }
  return;

timeout:
  // A bounded wait gave up: record it, wait (bounded) for copies still in
  // flight so that none lands in shared memory after exit, and leave.
  if (tid == 0) ring_drain(R, P);
  __syncthreads();
}

// Explicit instantiations, looked up by the host launcher.
template __global__ void dk_pass_scalar<float, 1, 0>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<float, 1, 1>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<float, 1, 2>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<float, 2, 0>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<float, 2, 1>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<float, 2, 2>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<double, 1, 0>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<double, 1, 1>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<double, 1, 2>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<double, 2, 0>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<double, 2, 1>(const __grid_constant__ PassArgs);
template __global__ void dk_pass_scalar<double, 2, 2>(const __grid_constant__ PassArgs);

typedef void (*PassKernel)(const PassArgs);

PassKernel scalar_pass_kernel(int fp32, int nf, int red) {
  static const PassKernel tab[2][2][3] = {
      {{dk_pass_scalar<double, 1, 0>, dk_pass_scalar<double, 1, 1>, dk_pass_scalar<double, 1, 2>},
       {dk_pass_scalar<double, 2, 0>, dk_pass_scalar<double, 2, 1>, dk_pass_scalar<double, 2, 2>}},
      {{dk_pass_scalar<float, 1, 0>, dk_pass_scalar<float, 1, 1>, dk_pass_scalar<float, 1, 2>},
       {dk_pass_scalar<float, 2, 0>, dk_pass_scalar<float, 2, 1>, dk_pass_scalar<float, 2, 2>}}};
  if (nf < 1 || nf > 2 || red < 0 || red > 2) return nullptr;
  return tab[fp32 ? 1 : 0][nf - 1][red];
}

}  // namespace clg
