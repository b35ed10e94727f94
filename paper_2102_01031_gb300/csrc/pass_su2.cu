// pass_su2.cu -- fused drift + kick pass of the SU(2) x U(1) doublet model
// (the gauge content of the CosmoLattice manual's lphi4SU2U1 example: Sec. 4.1
// action, Sec. 4.3 Hamiltonian form in temporal gauge, links, plaquettes and
// covariant derivatives of the U(1) and SU(N) toolkits of Sec. 4.2).
//
// State (35 arrays of one slab, array a at a * V elements):
//   0..3   phi_c, Phi = (phi_0 + i phi_1, phi_2 + i phi_3)/sqrt2 (psi = sqrt2 Phi below)
//   4..7   pi_c
//   8..10  A_i (U(1) link fields, V_i = exp(-i gQ dx A_i)),   11..13 pi_A,i
//   14 + 4 i + k   SU(2) link U_i = u0 - i (u1 s1 + u2 s2 + u3 s3) (s_a Pauli)
//   26 + 3 i + (a - 1)   pi_B,i^a
//
//   drift (deferred from the previous pass):
//       phi_c += cd pi_c,   A_i += cdA pi_A,i,
//       U_i <- exp(-i (gQB dx cdA) pi_B,i^a s_a/2) U_i
//   kick (W_i = V_i U_i, the doublet's hopping link):
//       pi_c     += c_k [ a^{1+alpha} (D^2 psi)_c - a^{3+alpha} 2 lam (|Phi|^2 - v^2) phi_c ]
//       pi_A,i   += c_k [ a^{1+alpha} (f_s/omega_s)^2 (gQ/dx) Im(psi^dag W_i psi(n+i)) + a^{alpha-1} C_i ]
//       pi_B,i^a += c_k [ a^{1+alpha} (f_s/omega_s)^2 (gQB/(2dx)) Im(psi^dag s_a W_i psi(n+i))
//                         - a^{alpha-1} (2/(gQB dx^3)) m_a(U_i S_i) ]
//   with D^2 psi = sum_i [W_i psi(n+i) - 2 psi + W_i^dag(n-i) psi(n-i)]/dx^2, C_i the compact
//   U(1) curl of the U(1) model, S_i the sum of the four staples of U_i(n) and m_a the
//   vector part of a quaternion (Im Tr[s_a M] = -2 m_a).  These are the kernels of one
//   lattice Hamiltonian (kinetic terms, covariant hopping, compact U(1) plaquettes,
//   SU(2) plaquette traces), so that both lattice Gauss laws hold exactly.
//
// Kernel layout.  A work item is a TX x TY tile of x-y sites over a chunk of
// z-planes; the resident CTAs (two per SM) take items in a round-robin that
// keeps neighbouring tiles on the same planes at the same time.  Each plane of
// the tile plus a one-site halo (corners included) is loaded from HBM (all 35
// loads of a site in flight at once), drifted in registers and kept, drifted,
// in a three-plane shared-memory ring (links as one 16-byte quaternion per
// site and direction, the doublet as one quaternion, the three U(1) link
// fields); the drifted fields of the CTA's own sites are written out right
// away.  The kick of plane z then reads every neighbour, staple and plaquette
// it needs from the ring (the stencil reaches n +- x, n +- y, n +- z and the
// diagonal neighbours n + i - j), and re-reads its own momenta, prefetched
// into L1 while the next plane loads.  The two CTAs of an SM overlap one's
// loads with the other's arithmetic.  The last CTA to finish sums the per-CTA
// partial sums in a fixed order and advances the scale factor (tail.cuh).
//
// Bound by the latency of a halo site's loads and the plane's barrier behind them (2320
// instructions a site, 44 % of the issue slots; memory alone takes 350 of 940 us at 192^3).  The kick is
// the kick-then-drift passes' (su2_kick.cuh: each plaquette once, carried along z), one
// barrier a plane, and at alpha = 1 no gauge energies: lphi4SU2U1 192^3 FP32, 5 VV2 steps
// and energies 6457 -> 5992 us, the measurement pass alone 1323 -> 1161 us.
#include "su2_kick.cuh"

namespace clg {

// Bytes of one ring slot: per halo site 3 links + doublet (quaternions) and 3 U(1)
// fields, and for lphi4SU2U1 also the singlet and vphi's two components.
__host__ __device__ constexpr size_t su2_slot_bytes(int TX, int TY, int esz, bool full = false) {
  return ((full ? 22 : 19) * (size_t)(TX + 2) * (TY + 2) * esz + 127) / 128 * 128;
}

// RED: 1 = sums for the Friedmann kicks, SU2_RED_ALPHA1 = the same at alpha = 1 (no gauge
// energies), 2 = full measurement.
// FULL: the lphi4SU2U1 model (Sec. 4.5): also a singlet phi_s and a U(1)-charged
// scalar vphi (charge Qc in units of the doublet's, hopping with exp(-i Qc gQ dx A_i)),
// coupled through V = lam (|Phi|^2 - v^2)^2 + qG |Phi|^2 phi_s^2 + 2 qH |Phi|^2 |vphi|^2:
//   pi_s   += c_k [a^{1+alpha} Lap phi_s - a^{3+alpha} 2 qG |Phi|^2 phi_s]
//   pi_vc  += c_k [a^{1+alpha} (D^2 vphi)_c - a^{3+alpha} 2 qH |Phi|^2 vphi_c]
//   pi_c   (doublet) gains - a^{3+alpha} (qG phi_s^2 + 2 qH |vphi|^2) phi_c
//   pi_A,i gains a^{1+alpha} (f_s/omega_s)^2 Qc (gQ/dx) (vphi_0 u_1 - vphi_1 u_0), u = its hop.
template <typename T, int RED, int TX, bool FULL>
__global__ void __launch_bounds__(256, (RED == 2 || sizeof(T) == 8) ? 1 : 2) dk_pass_su2(const PassArgs P) {
  constexpr int NACC = RED == 1 ? 6 : (RED == SU2_RED_ALPHA1 ? 3 : (FULL ? 29 : 23));
  constexpr int NLD = FULL ? SNARR_FULL : SNARR;  // arrays loaded per halo site
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ double red_s[SU2_NQ][9];
  __shared__ unsigned last_s;
  const LatConst& L = P.lat[0];
  const int N = L.N;
  constexpr int TY = SU2_TY, nth = TX * TY;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int lane = tid & 31, warp = tid >> 5;
  constexpr int HX = TX + 2, HS = HX * (TY + 2);
  const int ntx = N / TX, nty = N / TY;
  const long long NN = (long long)N * N, V = L.V;
  const int parity = P.parity;
  const T* const src = reinterpret_cast<const T*>(L.buf[parity][0]);
  T* const dst = reinterpret_cast<T*>(L.buf[parity ^ 1][0]);
  constexpr size_t slot_b = su2_slot_bytes(TX, TY, sizeof(T), FULL);

  // the deferred drift and the kick's coefficients
  __shared__ Su2Pass<T> coef_s;
  if (warp == 0) su2_coefficients<T>(L, P.sc, P.ck, __ldcg(&P.sc->cd), __ldcg(&P.sc->cdA), lane, &coef_s);
  __syncthreads();
  const T cd = coef_s.cd, cdA = coef_s.cdA, hB = coef_s.hB;
  const Su2Coef<T> cf = coef_s.k;
  const bool drifting = cd != T(0) || cdA != T(0);

  Acc<T> acc[NACC];
#pragma unroll
  for (int k = 0; k < NACC; ++k) acc[k].zero();
  float nonfinite = 0.f;

  // ring slot s: links [3][HS], doublet [HS], U(1) fields [3][HS]
  auto sU = [&](int s, int i) { return reinterpret_cast<Q4<T>*>(smem + s * slot_b) + i * HS; };
  auto sF = [&](int s) { return reinterpret_cast<Q4<T>*>(smem + s * slot_b) + 3 * HS; };
  auto sA = [&](int s, int i) { return reinterpret_cast<T*>(smem + s * slot_b) + 16 * HS + i * HS; };
  // FULL: the singlet (k = 0) and vphi's components (k = 1, 2)
  auto sX = [&](int s, int k) { return reinterpret_cast<T*>(smem + s * slot_b) + 19 * HS + k * HS; };

  // the 35 raw values of halo site k of plane zp, all loads issued before any use
  // (the source buffer is read-only during the pass)
  auto fetch = [&](int k, int x0, int y0, int zp, T (&r)[NLD]) {
    const int hx = k % HX, hy = k / HX;
    int gx = x0 + hx - 1, gy = y0 + hy - 1;
    gx = gx < 0 ? gx + N : (gx >= N ? gx - N : gx);
    gy = gy < 0 ? gy + N : (gy >= N ? gy - N : gy);
    const T* p = src + ((long long)zp * NN + (long long)gy * N + gx);
#pragma unroll
    for (int a = 0; a < NLD; ++a) {
      r[a] = __ldg(p);
      p += V;
    }
  };
  // drift halo site k into ring slot s; own sites written out when `own`
  auto put = [&](int s, int k, int x0, int y0, int zp, bool own, const T (&r)[NLD]) {
    Q4<T> f, u[3];
    T a[3];
    f.w = r[SF];
    f.x = r[SF + 1];
    f.y = r[SF + 2];
    f.z = r[SF + 3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      a[i] = r[SA + i];
      u[i].w = r[SU + 4 * i];
      u[i].x = r[SU + 4 * i + 1];
      u[i].y = r[SU + 4 * i + 2];
      u[i].z = r[SU + 4 * i + 3];
    }
    if (drifting) {
      f.w = fmaT(cd, r[SP], f.w);
      f.x = fmaT(cd, r[SP + 1], f.x);
      f.y = fmaT(cd, r[SP + 2], f.y);
      f.z = fmaT(cd, r[SP + 3], f.z);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        a[i] = fmaT(cdA, r[SPA + i], a[i]);
        // E = exp(-i hB pi.s) = (cos x, sin(x)/x hB pi), x = hB |pi|
        const T p1 = hB * r[SPB + 3 * i], p2 = hB * r[SPB + 3 * i + 1], p3 = hB * r[SPB + 3 * i + 2];
        T c, sc;
        cos_sinc(p1 * p1 + p2 * p2 + p3 * p3, c, sc);
        Q4<T> e;
        e.w = c;
        e.x = sc * p1;
        e.y = sc * p2;
        e.z = sc * p3;
        u[i] = qmul(e, u[i]);
        renorm(u[i]);
      }
    }
    sF(s)[k] = f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      sU(s, i)[k] = u[i];
      sA(s, i)[k] = a[i];
    }
    T xs[3] = {T(0), T(0), T(0)};  // FULL: phi_s, vphi_0, vphi_1, drifted
    if constexpr (FULL) {
      xs[0] = drifting ? fmaT(cd, r[SPS], r[SS]) : r[SS];
      xs[1] = drifting ? fmaT(cd, r[SPC], r[SC]) : r[SC];
      xs[2] = drifting ? fmaT(cd, r[SPC + 1], r[SC + 1]) : r[SC + 1];
#pragma unroll
      for (int m = 0; m < 3; ++m) sX(s, m)[k] = xs[m];
    }
    const int hx = k % HX, hy = k / HX;
    if (own && P.write && hx >= 1 && hx <= TX && hy >= 1 && hy <= TY) {
      T* o = dst + ((long long)zp * NN + (long long)(y0 + hy - 1) * N + (x0 + hx - 1));
      const T vals[19] = {f.w, f.x, f.y, f.z, a[0], a[1], a[2], u[0].w, u[0].x, u[0].y, u[0].z,
                          u[1].w, u[1].x, u[1].y, u[1].z, u[2].w, u[2].x, u[2].y, u[2].z};
#pragma unroll
      for (int m = 0; m < 19; ++m) {  // arrays 0..3, 8..10, 14..25
        const int arr = m < 4 ? SF + m : (m < 7 ? SA + (m - 4) : SU + (m - 7));
        o[arr * V] = vals[m];
      }
      if constexpr (FULL) {
        o[SS * V] = xs[0];
        o[SC * V] = xs[1];
        o[(SC + 1) * V] = xs[2];
      }
    }
  };
  // plane zp of tile (x0, y0) into slot s, drifted
  auto load_plane = [&](int s, int x0, int y0, int zp, bool own) {
    for (int k = tid; k < HS; k += nth) {
      T r0[NLD];
      fetch(k, x0, y0, zp, r0);
      put(s, k, x0, y0, zp, own, r0);
    }
  };

  // work items: (tile, z-chunk), tile = by * ntx + bx, numbered chunk-major; CTA b takes
  // items b, b + gridDim.x, ...  A round of items covers about one chunk of every tile,
  // so neighbouring tiles march the same planes at about the same time and the halo
  // rows and columns a CTA reads come from L2 rather than DRAM.
  const int ntiles = ntx * nty, nzc = L.su2_nzc, nitems = ntiles * nzc;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const int tile = item % ntiles, chunk = item / ntiles;
    const int z0 = (int)((long long)chunk * N / nzc);
    const int nz = (int)((long long)(chunk + 1) * N / nzc) - z0;
    const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
    __syncthreads();  // the previous item's reads of the ring are done
    load_plane(0, x0, y0, (z0 - 1 + N) % N, false);
    load_plane(1, x0, y0, z0, true);
    __syncthreads();
    const int own = (ty + 1) * HX + tx + 1;
    const long long gown = (long long)(y0 + ty) * N + x0 + tx;
    // the site's neighbourhood in slots s and s + 1 of the ring (su2_kick.cuh), its momenta
    // from global memory (prefetched into L1)
    struct Hood {
      const unsigned char *c, *p;
      const T* src;
      long long g, V;
      int own;
      __device__ __forceinline__ const unsigned char* slot(int pl) const { return pl ? p : c; }
      __device__ __forceinline__ Q4<T> u(int pl, int i, int dx, int dy) const {
        return reinterpret_cast<const Q4<T>*>(slot(pl))[i * HS + own + dy * HX + dx];
      }
      __device__ __forceinline__ Q4<T> f(int pl, int dx, int dy) const { return u(pl, 3, dx, dy); }
      __device__ __forceinline__ T a(int pl, int i, int dx, int dy) const {
        return reinterpret_cast<const T*>(slot(pl))[(16 + i) * HS + own + dy * HX + dx];
      }
      __device__ __forceinline__ T x(int pl, int k, int dx, int dy) const { return a(pl, 3 + k, dx, dy); }
      __device__ __forceinline__ T mom(int arr) const { return __ldg(src + arr * V + g); }
    };
    auto hood = [&](int s, long long g) {
      return Hood{smem + s % 3 * slot_b, smem + (s + 1) % 3 * slot_b, src, g, V, own};
    };
    Su2Carry<T> carry = {};
    su2_carry<T, FULL>(hood(0, 0), cf, carry);
    for (int j = 0; j < nz; ++j) {
      const int z = z0 + j;
      const long long g = (long long)z * NN + gown;
      {  // the kick's own momenta move into L1 while the next plane loads
        const T* pp = src + g;
        prefetch_l1(pp + SP * V);
        prefetch_l1(pp + (SP + 1) * V);
        prefetch_l1(pp + (SP + 2) * V);
        prefetch_l1(pp + (SP + 3) * V);
#pragma unroll
        for (int m = 0; m < 3; ++m) prefetch_l1(pp + (SPA + m) * V);
#pragma unroll
        for (int m = 0; m < 9; ++m) prefetch_l1(pp + (SPB + m) * V);
        if constexpr (FULL) {
          prefetch_l1(pp + SPS * V);
          prefetch_l1(pp + SPC * V);
          prefetch_l1(pp + (SPC + 1) * V);
        }
      }
      // plane z + 1 into the slot that held z - 1: its values live on in the carries, and a
      // warp that is still at the kick of z reads the other two slots, so that one barrier
      // a plane is enough
      load_plane((j + 2) % 3, x0, y0, (z + 1) % N, j + 1 < nz);
      __syncthreads();
      auto link = [&](int i, const Q4<T>&, T, T pnA, const T (&pnB)[3]) {
        if (!P.write) return;
        dst[(SPA + i) * V + g] = pnA;
#pragma unroll
        for (int a = 0; a < 3; ++a) dst[(SPB + 3 * i + a) * V + g] = pnB[a];
      };
      Su2Site<T> site;
      su2_kick<T, RED, FULL>(hood(j + 1, g), cf, carry, site, [] {}, link);
      if (P.write) {
#pragma unroll
        for (int c2 = 0; c2 < 4; ++c2) dst[(SP + c2) * V + g] = site.pn[c2];
        if constexpr (FULL) {
          dst[SPS * V + g] = site.pns;
          dst[SPC * V + g] = site.pnc0;
          dst[(SPC + 1) * V + g] = site.pnc1;
        }
      }
      su2_sums<T, RED, FULL>(cf, site, acc, nonfinite);
    }
  }

  su2_pass_end<T, RED, FULL>(P, L, acc, nonfinite, red_s, last_s, tid, lane, warp, nth);
}

typedef void (*PassKernel)(const PassArgs);

// red: 1, 2 or SU2_RED_ALPHA1 (without self-consistent expansion the passes of pass_su2_kd.cu run).
PassKernel su2_pass_kernel(int fp32, int red, int TX, int full) {
  constexpr int A1 = SU2_RED_ALPHA1;
  static const PassKernel tab[2][2][2][3] = {  // [full][TX == 32][fp32][red - 1]
      {{{dk_pass_su2<double, 1, 16, false>, dk_pass_su2<double, 2, 16, false>, dk_pass_su2<double, A1, 16, false>},
        {dk_pass_su2<float, 1, 16, false>, dk_pass_su2<float, 2, 16, false>, dk_pass_su2<float, A1, 16, false>}},
       {{dk_pass_su2<double, 1, 32, false>, dk_pass_su2<double, 2, 32, false>, dk_pass_su2<double, A1, 32, false>},
        {dk_pass_su2<float, 1, 32, false>, dk_pass_su2<float, 2, 32, false>, dk_pass_su2<float, A1, 32, false>}}},
      {{{dk_pass_su2<double, 1, 16, true>, dk_pass_su2<double, 2, 16, true>, dk_pass_su2<double, A1, 16, true>},
        {dk_pass_su2<float, 1, 16, true>, dk_pass_su2<float, 2, 16, true>, dk_pass_su2<float, A1, 16, true>}},
       {{dk_pass_su2<double, 1, 32, true>, dk_pass_su2<double, 2, 32, true>, dk_pass_su2<double, A1, 32, true>},
        {dk_pass_su2<float, 1, 32, true>, dk_pass_su2<float, 2, 32, true>, dk_pass_su2<float, A1, 32, true>}}}};
  static_assert(A1 == 3, "the table's order");
  if (red < 1 || red > 3 || (TX != 16 && TX != 32)) return nullptr;
  return tab[full ? 1 : 0][TX == 32 ? 1 : 0][fp32 ? 1 : 0][red - 1];
}

size_t su2_smem_bytes(int TX, int TY, int esz, int full) { return 3 * su2_slot_bytes(TX, TY, esz, full != 0); }

// ---------------------------------------------------------------------------
// Initial state and the Gauss-law monitor of the doublet model.
// ---------------------------------------------------------------------------

// links at the identity (eqs. Inflc1-2): u0 = 1, the rest zero (caller zeroed the slab)
template <typename T>
__global__ void su2_identity_links_kernel(T* base, long long V) {
  for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < V;
       n += (long long)gridDim.x * blockDim.x)
#pragma unroll
    for (int i = 0; i < 3; ++i) base[(SU + 4 * i) * V + n] = T(1);
}

template <typename T>
__device__ __forceinline__ Q4<double> dq(const T* b, int a, long long V, long long n) {
  Q4<double> r;
  r.w = (double)b[a * V + n];
  r.x = (double)b[(a + 1) * V + n];
  r.y = (double)b[(a + 2) * V + n];
  r.z = (double)b[(a + 3) * V + n];
  return r;
}

// Charge density of generator g (0: U(1); 1..3: SU(2) colour g) at site n:
//   U(1):  (f_s/omega_s)^2 gQ Im[psi^dag pi_psi]
//   SU(2): (f_s/omega_s)^2 (gQB/2) Im[psi^dag s_g pi_psi]
template <typename T>
__device__ double su2_rho(const LatConst& L, const T* b, int g, long long n) {
  const long long V = L.V;
  const Q4<double> f = dq(b, SF, V, n), p = dq(b, SP, V, n);
  double im;
  if (g == 0) im = (f.w * p.x - f.x * p.w) + (f.y * p.z - f.z * p.y);
  else if (g == 1) im = (f.w * p.z - f.x * p.y) + (f.y * p.x - f.z * p.w);
  else if (g == 2) im = (f.y * p.w + f.z * p.x) - (f.w * p.y + f.x * p.z);
  else im = (f.w * p.x - f.x * p.w) - (f.y * p.z - f.z * p.y);
  if (g == 0 && L.model == CL_MODEL_LPHI4_SU2U1)  // vphi's charge density, charge Qc in units of the doublet's
    im += L.Qc * ((double)b[SC * V + n] * (double)b[(SPC + 1) * V + n] -
                  (double)b[(SC + 1) * V + n] * (double)b[SPC * V + n]);
  return L.fo2 * (g == 0 ? L.gQ : 0.5 * L.gQB) * im;
}

template <typename T>
__global__ void su2_rho_kernel(const LatConst* Lc, int parity, int g, double2* rho) {
  const LatConst& L = *Lc;
  const T* b = reinterpret_cast<const T*>(L.buf[parity][0]);
  for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < L.V;
       n += (long long)gridDim.x * blockDim.x)
    rho[n] = make_double2(su2_rho<T>(L, b, g, n), 0.0);
}

// |L - R|, |L + R| summed over the four laws, and max |L - R|, per block.
template <typename T>
__global__ void su2_gauss_monitor_kernel(const LatConst* Lc, int parity, double* part) {
  __shared__ double sh[3][32];
  const LatConst& L = *Lc;
  const T* b = reinterpret_cast<const T*>(L.buf[parity][0]);
  const int N = L.N;
  const long long NN = (long long)N * N, V = L.V;
  double sd = 0.0, ss = 0.0, mx = 0.0;
  for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < V;
       n += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(n % N), y = (int)((n / N) % N), z = (int)(n / NN);
    const long long nm[3] = {x ? n - 1 : n + N - 1, y ? n - N : n + NN - N, z ? n - NN : n + V - NN};
    double lhs[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = 0; i < 3; ++i) {
      const long long m = nm[i];
      lhs[0] += (double)b[(SPA + i) * V + n] - (double)b[(SPA + i) * V + m];
      // (U^dag P U)^a, P = p.s/2 at n - i: rotation of p by the link
      const Q4<double> u = dq(b, SU + 4 * i, V, m);
      Q4<double> pq;
      pq.w = 0.0;
      pq.x = (double)b[(SPB + 3 * i) * V + m];
      pq.y = (double)b[(SPB + 3 * i + 1) * V + m];
      pq.z = (double)b[(SPB + 3 * i + 2) * V + m];
      const Q4<double> r = qmul(qmul(qconj(u), pq), u);
      lhs[1] += (double)b[(SPB + 3 * i) * V + n] - r.x;
      lhs[2] += (double)b[(SPB + 3 * i + 1) * V + n] - r.y;
      lhs[3] += (double)b[(SPB + 3 * i + 2) * V + n] - r.z;
    }
    for (int g2 = 0; g2 < 4; ++g2) {
      const double l = lhs[g2] / L.dx, r = su2_rho<T>(L, b, g2, n);
      const double d = fabs(l - r);
      sd += d;
      ss += fabs(l + r);
      mx = fmax(mx, d);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    sd += __shfl_down_sync(0xffffffffu, sd, o);
    ss += __shfl_down_sync(0xffffffffu, ss, o);
    mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) {
    sh[0][w] = sd;
    sh[1][w] = ss;
    sh[2][w] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, c = 0.0, m = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
      a += sh[0][i];
      c += sh[1][i];
      m = fmax(m, sh[2][i]);
    }
    part[3 * blockIdx.x] = a;
    part[3 * blockIdx.x + 1] = c;
    part[3 * blockIdx.x + 2] = m;
  }
}

__global__ void su2_gauss_final_kernel(const double* part, int nblk, long long V, double* out) {
  if (threadIdx.x | blockIdx.x) return;
  double a = 0.0, b = 0.0, m = 0.0;
  for (int i = 0; i < nblk; ++i) {
    a += part[3 * i];
    b += part[3 * i + 1];
    m = fmax(m, part[3 * i + 2]);
  }
  out[0] = b > 0.0 ? a / b : 0.0;
  out[1] = a / (double)V;
  out[2] = b / (double)V;
  out[3] = m;
}

cudaError_t launch_su2_identity_links(int fp32, void* base, long long V, cudaStream_t st) {
  const int tb = 256;
  const int g = (int)((V + tb - 1) / tb < 65536 ? (V + tb - 1) / tb : 65536);
  if (fp32) su2_identity_links_kernel<float><<<g, tb, 0, st>>>((float*)base, V);
  else su2_identity_links_kernel<double><<<g, tb, 0, st>>>((double*)base, V);
  return cudaGetLastError();
}

cudaError_t launch_su2_rho(int fp32, const LatConst* L, int parity, int g, double2* rho, long long V,
                           cudaStream_t st) {
  const int tb = 256;
  const int gr = (int)((V + tb - 1) / tb < 65536 ? (V + tb - 1) / tb : 65536);
  if (fp32) su2_rho_kernel<float><<<gr, tb, 0, st>>>(L, parity, g, rho);
  else su2_rho_kernel<double><<<gr, tb, 0, st>>>(L, parity, g, rho);
  return cudaGetLastError();
}

cudaError_t launch_su2_gauss_monitor(int fp32, const LatConst* L, int parity, double* part, int nblk,
                                     long long V, cudaStream_t st) {
  if (fp32) su2_gauss_monitor_kernel<float><<<nblk, 256, 0, st>>>(L, parity, part);
  else su2_gauss_monitor_kernel<double><<<nblk, 256, 0, st>>>(L, parity, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  su2_gauss_final_kernel<<<1, 32, 0, st>>>(part, nblk, V, part + 3 * nblk);
  return cudaGetLastError();
}

}  // namespace clg
