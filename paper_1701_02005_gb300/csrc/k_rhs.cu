// Explicit right-hand sides of one RK3 substage (arXiv:1701.02005, Eq. (1)
// momentum with the Coulomb force, Eq. (3) Nernst-Planck for c+ and c-,
// staggered as in Fig. 1; Numerical methods for the time integration).
//
// One thread owns one cell (i, j, k) and produces, for the u point on its
// x-face i, the w point on its z-face k, the v point on its bottom y-face j
// (j >= 1) and the two ion concentrations at its centre:
//   H  = -div(flux) + x/z diffusion + body force        (explicit terms)
//   r  = dt [gam H + zet H_old - alp G p + alp nu L_y q] (Crank-Nicolson RHS)
// H overwrites H_old in place (each thread touches only its own entries).
#include <algorithm>

#include "pnp_common.cuh"

namespace pnp {

template <typename T>
__device__ __forceinline__ double L(const T* p, size_t i) {
  return (double)__ldg(p + i);
}

template <typename TV>
__global__ void __launch_bounds__(128) k_rhs(Fields<TV> f, Geo g, Metrics mt, Phys ph, Stage st) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int k = blockIdx.y * blockDim.y + threadIdx.y;
  const int j = blockIdx.z;
  if (i >= g.nx || k >= g.nz) return;
  const int nx = g.nx, nz = g.nz, nyc = g.nyc;
  const int im = i ? i - 1 : nx - 1, ip = (i + 1 == nx) ? 0 : i + 1;
  const int km = k ? k - 1 : nz - 1, kp = (k + 1 == nz) ? 0 : k + 1;
  const bool has_dn = j > 0, has_up = j < nyc - 1;
  const double idx = g.idx, idz = g.idz;
  const double idx2 = idx * idx, idz2 = idz * idz;
  const size_t c0 = cidx(j, k, i, nz, nx);
  const size_t cxm = cidx(j, k, im, nz, nx), cxp = cidx(j, k, ip, nz, nx);
  const size_t czm = cidx(j, km, i, nz, nx), czp = cidx(j, kp, i, nz, nx);
  const size_t P = (size_t)nz * nx;
  const double idyj = mt.idy[j];

  // ---------------- shared loads ----------------
  const double u0 = L(f.u, c0), uxm = L(f.u, cxm), uxp = L(f.u, cxp), uzm = L(f.u, czm), uzp = L(f.u, czp);
  const double uym = has_dn ? L(f.u, c0 - P) : 0.0, uyp = has_up ? L(f.u, c0 + P) : 0.0;
  const double w0 = L(f.w, c0), wxm = L(f.w, cxm), wxp = L(f.w, cxp), wzm = L(f.w, czm), wzp = L(f.w, czp);
  const double wym = has_dn ? L(f.w, c0 - P) : 0.0, wyp = has_up ? L(f.w, c0 + P) : 0.0;
  // v on the bottom face j and top face j+1 of this cell (wall faces hold zeros)
  const double vb = L(f.v, c0), vt = L(f.v, c0 + P);
  const double Ph0 = L(f.Phi, c0), Phxm = L(f.Phi, cxm), Phxp = L(f.Phi, cxp);
  const double Phzm = L(f.Phi, czm), Phzp = L(f.Phi, czp);
  const double Phym = has_dn ? L(f.Phi, c0 - P) : 0.0, Phyp = has_up ? L(f.Phi, c0 + P) : 0.0;
  const double cp0 = L(f.cp, c0), cm0 = L(f.cm, c0);
  const double rho0 = cp0 - cm0;
  const double p0 = L(f.p, c0);

  // ---------------- u at (x-face i, y-centre j, z-centre k) ----------------
  {
    const double ubp = 0.5 * (u0 + uxp), ubm = 0.5 * (uxm + u0);
    const double ax = (ubp * ubp - ubm * ubm) * idx;
    const double vft = 0.5 * (L(f.v, cidx(j + 1, k, im, nz, nx)) + vt);   // v at (x-face i, y-face j+1)
    const double vfb = 0.5 * (L(f.v, cxm) + vb);                 // v at (x-face i, y-face j)
    const double uft = has_up ? 0.5 * (u0 + uyp) : 0.0;
    const double ufb = has_dn ? 0.5 * (uym + u0) : 0.0;
    const double ay = (vft * uft - vfb * ufb) * idyj;
    const double wfk = 0.5 * (wxm + w0);                        // w at (x-face i, z-face k)
    const double wfkp = 0.5 * (L(f.w, cidx(j, kp, im, nz, nx)) + wzp);   // w at (x-face i, z-face k+1)
    const double az = (wfkp * 0.5 * (u0 + uzp) - wfk * 0.5 * (uzm + u0)) * idz;
    const double lap = (uxp - 2.0 * u0 + uxm) * idx2 + (uzp - 2.0 * u0 + uzm) * idz2;
    const double rhom = L(f.cp, cxm) - L(f.cm, cxm);
    const double fu = -ph.K * 0.5 * (rhom + rho0) * (Ph0 - Phxm) * idx;
    const double H = -(ax + ay + az) + (st.af ? 0.0 : ph.nu * lap) + fu;
    const double ub = f.wall_u ? (double)f.wall_u[(size_t)k * nx + i] : -ph.Uw;
    const double ut = f.wall_u ? (double)f.wall_u[P + (size_t)k * nx + i] : ph.Uw;
    const double Ly = mt.lo_c[j] * ((has_dn ? uym : ub) - u0) + mt.hi_c[j] * ((has_up ? uyp : ut) - u0);
    const double gp = (p0 - L(f.p, cxm)) * idx;
    const double Ho = (double)f.Hu[c0];
    f.ru[c0] = (TV)(st.dt * (st.gam * H + st.zet * Ho - st.alp * gp + st.alp * ph.nu * (st.af ? Ly + lap : Ly)));
    f.Hu[c0] = (TV)H;
  }

  // ---------------- w at (x-centre i, y-centre j, z-face k) ----------------
  {
    const double wbp = 0.5 * (w0 + wzp), wbm = 0.5 * (wzm + w0);
    const double az = (wbp * wbp - wbm * wbm) * idz;
    const double vft = 0.5 * (L(f.v, cidx(j + 1, km, i, nz, nx)) + vt);
    const double vfb = 0.5 * (L(f.v, czm) + vb);
    const double wft = has_up ? 0.5 * (w0 + wyp) : 0.0;
    const double wfb = has_dn ? 0.5 * (wym + w0) : 0.0;
    const double ay = (vft * wft - vfb * wfb) * idyj;
    const double ufi = 0.5 * (uzm + u0);                        // u at (x-face i, z-face k)
    const double ufip = 0.5 * (L(f.u, cidx(j, km, ip, nz, nx)) + uxp);   // u at (x-face i+1, z-face k)
    const double ax = (ufip * 0.5 * (w0 + wxp) - ufi * 0.5 * (wxm + w0)) * idx;
    const double lap = (wxp - 2.0 * w0 + wxm) * idx2 + (wzp - 2.0 * w0 + wzm) * idz2;
    const double rhom = L(f.cp, czm) - L(f.cm, czm);
    const double fw = -ph.K * 0.5 * (rhom + rho0) * (Ph0 - Phzm) * idz;
    const double H = -(ax + ay + az) + (st.af ? 0.0 : ph.nu * lap) + fw;
    const double wb = f.wall_w ? (double)f.wall_w[(size_t)k * nx + i] : 0.0;
    const double wt = f.wall_w ? (double)f.wall_w[P + (size_t)k * nx + i] : 0.0;
    const double Ly = mt.lo_c[j] * ((has_dn ? wym : wb) - w0) + mt.hi_c[j] * ((has_up ? wyp : wt) - w0);
    const double gp = (p0 - L(f.p, czm)) * idz;
    const double Ho = (double)f.Hw[c0];
    f.rw[c0] = (TV)(st.dt * (st.gam * H + st.zet * Ho - st.alp * gp + st.alp * ph.nu * (st.af ? Ly + lap : Ly)));
    f.Hw[c0] = (TV)H;
  }

  // ---------------- v at (x-centre i, y-face j, z-centre k), 1 <= j <= nyc-1 ----------------
  if (has_dn) {
    const double wl = mt.wl[j], wu = mt.wu[j], ihj = mt.ih[j];
    const size_t d0 = c0 - P;   // cell j-1
    const double v0 = vb;
    const double vxm = L(f.v, cxm), vxp = L(f.v, cxp), vzm = L(f.v, czm), vzp = L(f.v, czp);
    const double vym = L(f.v, c0 - P), vyp = vt;
    const double Ui = wl * L(f.u, d0) + wu * u0;                               // u at (x-face i, y-face j)
    const double Uip = wl * L(f.u, cidx(j - 1, k, ip, nz, nx)) + wu * uxp;     // u at (x-face i+1, y-face j)
    const double ax = (Uip * 0.5 * (v0 + vxp) - Ui * 0.5 * (vxm + v0)) * idx;
    const double vbu = 0.5 * (v0 + vyp), vbd = 0.5 * (vym + v0);
    const double ay = (vbu * vbu - vbd * vbd) * ihj;
    const double Wk = wl * L(f.w, d0) + wu * w0;                               // w at (y-face j, z-face k)
    const double Wkp = wl * L(f.w, cidx(j - 1, kp, i, nz, nx)) + wu * wzp;   // w at (y-face j, z-face k+1)
    const double az = (Wkp * 0.5 * (v0 + vzp) - Wk * 0.5 * (vzm + v0)) * idz;
    const double lap = (vxp - 2.0 * v0 + vxm) * idx2 + (vzp - 2.0 * v0 + vzm) * idz2;
    const double rhod = L(f.cp, d0) - L(f.cm, d0);
    const double fv = -ph.K * 0.5 * (rhod + rho0) * (Ph0 - Phym) * ihj;
    const double H = -(ax + ay + az) + (st.af ? 0.0 : ph.nu * lap) + fv;
    const double Ly = mt.lo_f[j] * (vym - v0) + mt.hi_f[j] * (vyp - v0);
    const double gp = (p0 - L(f.p, d0)) * ihj;
    const double Ho = (double)f.Hv[c0];
    f.rv[c0] = (TV)(st.dt * (st.gam * H + st.zet * Ho - st.alp * gp + st.alp * ph.nu * (st.af ? Ly + lap : Ly)));
    f.Hv[c0] = (TV)H;
  }

  // ---------------- c+ and c- at the cell centre (Eq. (3)) ----------------
  {
    const double D = ph.D;
    const double ux_i = u0, ux_ip = uxp;       // u on x-faces i and i+1
    const double wz_k = w0, wz_kp = wzp;       // w on z-faces k and k+1
    const double ihj = mt.ih[j], ihjp = mt.ih[j + 1];
#pragma unroll
    for (int ion = 0; ion < 2; ++ion) {
      const double* c = ion == 0 ? f.cp : f.cm;
      const double s = ion == 0 ? 1.0 : -1.0;
      const double cc = ion == 0 ? cp0 : cm0;
      const double cxm_ = L(c, cxm), cxp_ = L(c, cxp), czm_ = L(c, czm), czp_ = L(c, czp);
      const double cym_ = has_dn ? L(c, c0 - P) : 0.0, cyp_ = has_up ? L(c, c0 + P) : 0.0;
      // face fluxes F = u c_face - D grad c - s D c_face grad Phi
      double ca = 0.5 * (cxm_ + cc), cb = 0.5 * (cc + cxp_);
      const double Fx_i = ux_i * ca - D * (cc - cxm_) * idx - s * D * ca * (Ph0 - Phxm) * idx;
      const double Fx_ip = ux_ip * cb - D * (cxp_ - cc) * idx - s * D * cb * (Phxp - Ph0) * idx;
      ca = 0.5 * (czm_ + cc);
      cb = 0.5 * (cc + czp_);
      const double Fz_k = wz_k * ca - D * (cc - czm_) * idz - s * D * ca * (Ph0 - Phzm) * idz;
      const double Fz_kp = wz_kp * cb - D * (czp_ - cc) * idz - s * D * cb * (Phzp - Ph0) * idz;
      // y faces: advection + migration only (y diffusion is implicit); walls carry no flux
      double Fy_j = 0.0, Fy_jp = 0.0;
      if (has_dn) {
        const double cf = 0.5 * (cym_ + cc);
        Fy_j = vb * cf - s * D * cf * (Ph0 - Phym) * ihj;
      }
      if (has_up) {
        const double cf = 0.5 * (cc + cyp_);
        Fy_jp = vt * cf - s * D * cf * (Phyp - Ph0) * ihjp;
      }
      double H = -((Fx_ip - Fx_i) * idx + (Fy_jp - Fy_j) * idyj + (Fz_kp - Fz_k) * idz);
      double Ly = (has_dn ? mt.lo_c[j] * (cym_ - cc) : 0.0) + (has_up ? mt.hi_c[j] * (cyp_ - cc) : 0.0);
      if (st.af) {   // the x/z diffusion leaves H and joins the implicit operator
        const double lapc = (cxp_ - 2.0 * cc + cxm_) * idx2 + (czp_ - 2.0 * cc + czm_) * idz2;
        H -= D * lapc;
        Ly += lapc;
      }
      double* Hc = ion == 0 ? f.Hcp : f.Hcm;
      double* rc = ion == 0 ? f.rcp : f.rcm;
      const double Ho = Hc[c0];
      rc[c0] = st.dt * (st.gam * H + st.zet * Ho + st.alp * D * Ly);
      Hc[c0] = H;
    }
  }
}

// ---------------------------------------------------------------------------
// The same terms with every face quantity computed once.  The FP64 pipe issues
// one warp instruction per 16 cycles and SM, so operations are what this stencil
// costs, and a cell that forms both of its faces in each direction does a third
// of them twice.  Here a block marches a chunk of y-planes over a TX x TZ tile; a
// thread forms the left x-face, the front z-face and the top y-face of its cell
// (and the centre products), passes the x and z ones to its neighbours through
// shared memory (two buffers, one barrier per plane) and keeps the y ones in
// registers for the next plane.  The right and back faces of the tile's edge are
// formed by its edge threads.  The edge product (w_{i-1} + w_i)(u_{k-1} + u_k)
// serves u's z-flux and w's x-flux.  Factors 1/2 and 1/4 of the averages are part
// of the (exactly scaled) constants, and all constants of a plane come from a
// per-block table.  About 155 FP64 operations per cell (and 5 for the tile's
// edges) against 235: 128x97x128, 0.96 -> 0.50 ms, the FP64 pipe 79% busy.  The tiles
// are as wide as Nx allows, for few x-edges.
// ---------------------------------------------------------------------------
struct MarchPlane {   // constants of plane j (face j and, suffix p, face j + 1)
  double idy4, idy2;                   // 1/(4 dy), 1/(2 dy)
  double ulo, uhi, vlo, vhi, clo, chi; // dt alp nu (ions: D) times the y-couplings of the cells and of the face below
  double wl2, wu2;                     // half the volume weights at the face below
  double ih4, K2ih, aih, Dihp;         // 1/(4 h_j), K/(2 h_j), dt alp / h_j, D / h_{j+1}
};

struct MarchCoef {
  double idx4, idz4, idx2, idz2, idx, idz;   // 1/(4 dx), 1/(2 dx), 1/dx and along z
  double nxx, nzz, nc;                 // nu / dx^2, nu / dz^2 and -2 times their sum (x/z implicit: times dt alp)
  double dxx, dzz, dc;                 // the same with D in the place of nu (x/z implicit only)
  double K2x, K2z;                     // K / (2 dx), K / (2 dz)
  double Dx, Dz, Dx2, Dz2;             // D / dx, D / dz and twice that
  double gdt, zdt, adx, adz, anu, aD;  // dt gam, dt zet, dt alp / dx, dt alp / dz, dt alp nu, dt alp D
  double D, K, Uw, alpdt;
};

template <int TX, int TZ, bool AF>
__global__ void __launch_bounds__(TX* TZ)
    k_rhs_march(Fields<double> f, Geo g, Metrics mt, const __grid_constant__ MarchCoef C, int jc) {
  // faces: x arrays have a column TX (the tile's right edge), z arrays a row TZ
  __shared__ double sE[2][TZ + 1][TX + 1], sVx[2][TZ][TX + 1], sPx[2][TZ][TX + 1], sMx[2][TZ][TX + 1];
  __shared__ double sVz[2][TZ + 1][TX], sPz[2][TZ + 1][TX], sMz[2][TZ + 1][TX];
  __shared__ double sSu[2][TZ][TX], sSw[2][TZ][TX];
  extern __shared__ MarchPlane pl[];
  const int tx = threadIdx.x, tz = threadIdx.y, tid = tz * TX + tx;
  const int nx = g.nx, nz = g.nz, nyc = g.nyc;
  const int i = blockIdx.x * TX + tx, k = blockIdx.y * TZ + tz;
  const int jb = blockIdx.z * jc, je = min(nyc, jb + jc);
  const bool wx = TX < nx, wz = TZ < nz;   // false: the tile spans the period, its last neighbour is its first
  for (int r = tid; r < je - jb; r += TX * TZ) {
    const int j = jb + r;
    MarchPlane q;
    q.idy4 = 0.25 * mt.idy[j];
    q.idy2 = 0.5 * mt.idy[j];
    q.ulo = C.anu * mt.lo_c[j];
    q.uhi = C.anu * mt.hi_c[j];
    q.vlo = C.anu * mt.lo_f[j];
    q.vhi = C.anu * mt.hi_f[j];
    q.clo = C.aD * mt.lo_c[j];
    q.chi = C.aD * mt.hi_c[j];
    q.wl2 = 0.5 * mt.wl[j];
    q.wu2 = 0.5 * mt.wu[j];
    q.ih4 = 0.25 * mt.ih[j];
    q.K2ih = 0.5 * C.K * mt.ih[j];
    q.aih = C.alpdt * mt.ih[j];
    q.Dihp = C.D * mt.ih[j + 1];
    pl[r] = q;
  }
  const int im = i ? i - 1 : nx - 1, ip = i + 1 == nx ? 0 : i + 1;
  const int km = k ? k - 1 : nz - 1, kp = k + 1 == nz ? 0 : k + 1;
  const int P = nz * nx;
  const int o0 = k * nx + i, oxm = k * nx + im, oxp = k * nx + ip, ozm = km * nx + i, ozp = kp * nx + i;
  const int txp = wx ? tx + 1 : (tx + 1) & (TX - 1), tzp = wz ? tz + 1 : (tz + 1) & (TZ - 1);
  // plane pointers advance with j
  size_t pj = (size_t)jb * P;
  auto at = [&](const double* a, int o) { return __ldg(a + pj + o); };
  auto up = [&](const double* a, int o) { return __ldg(a + pj + P + o); };     // plane j + 1
  auto dn = [&](const double* a, int o) { return __ldg(a + pj - P + o); };     // plane j - 1 (j > 0)
  // the cell's values of plane j and what is carried from plane j - 1
  double u0 = at(f.u, o0), w0 = at(f.w, o0), vb = at(f.v, o0), Ph0 = at(f.Phi, o0), cp0 = at(f.cp, o0),
         cm0 = at(f.cm, o0), p0 = at(f.p, o0);
  double vxm = at(f.v, oxm), vzm = at(f.v, ozm);   // v on face j at i - 1, k - 1
  double svx = vxm + vb, svz = vzm + vb;           // v at the edges of face j (x2)
  double ud = 0.0, wd = 0.0, rhoy = 0.0, pd = 0.0; // rhoy: charge at face j (x2)
  double tu = 0.0, tw = 0.0, tv = 0.0;             // y-fluxes of u, w (face j, x4) and of v (centre j - 1, x4)
  double du = 0.0, dw = 0.0, dv = 0.0, dPy = 0.0;  // differences across face j (dv: v_j - v_{j-1})
  double fp = 0.0, fm = 0.0, dp = 0.0, dm = 0.0;   // ion fluxes (x2) and differences at face j
  const bool walls = f.wall_u != nullptr;
  if (jb > 0) {
    ud = dn(f.u, o0);
    wd = dn(f.w, o0);
    pd = dn(f.p, o0);
    const double vd = dn(f.v, o0), Phd = dn(f.Phi, o0), cpd = dn(f.cp, o0), cmd = dn(f.cm, o0);
    const double sp = cpd + cp0, sm = cmd + cm0;
    rhoy = sp - sm;
    tu = svx * (ud + u0);
    tw = svz * (wd + w0);
    const double sv = vd + vb;
    tv = sv * sv;
    du = u0 - ud;
    dw = w0 - wd;
    dv = vb - vd;
    dPy = Ph0 - Phd;
    const double gy = C.D * mt.ih[jb] * dPy;
    fp = sp * (vb - gy);
    fm = sm * (vb + gy);
    dp = cp0 - cpd;
    dm = cm0 - cmd;
  } else {
    du = u0 - (walls ? f.wall_u[o0] : -C.Uw);
    dw = w0 - (walls ? f.wall_w[o0] : 0.0);
  }
  __syncthreads();   // the table
  for (int j = jb; j < je; ++j, pj += P) {
    const MarchPlane& q = pl[j - jb];
    const bool has_dn = j > 0, has_up = j < nyc - 1;
    const int b = (j - jb) & 1;
    // ---- faces of this cell ----
    const double uxm = at(f.u, oxm), uxp = at(f.u, oxp), uzm = at(f.u, ozm), uzp = at(f.u, ozp);
    const double wxm = at(f.w, oxm), wxp = at(f.w, oxp), wzm = at(f.w, ozm), wzp = at(f.w, ozp);
    const double cpx = at(f.cp, oxm), cmx = at(f.cm, oxm), cpz = at(f.cp, ozm), cmz = at(f.cm, ozm);
    const double dPx = Ph0 - at(f.Phi, oxm), dPz = Ph0 - at(f.Phi, ozm);
    // ion flux (x2) through a face: (c + c') (U -+ D dPhi/dn) - 2 D (c' - c)/dn
    auto flux = [&](double sum, double ca, double cb, double E, double dc2) {
      const double adv = sum * E;
      return AF ? adv : adv - dc2 * (cb - ca);
    };
    const double E = (wxm + w0) * (uzm + u0);
    {
      const double a = u0 + uxp, c = w0 + wzp;
      sSu[b][tz][tx] = a * a;
      sSw[b][tz][tx] = c * c;
      sE[b][tz][tx] = E;
    }
    double Vx = 0.0, Vz = 0.0;
    if (has_dn) {
      Vx = (q.wl2 * ud + q.wu2 * u0) * svx;
      Vz = (q.wl2 * wd + q.wu2 * w0) * svz;
      sVx[b][tz][tx] = Vx;
      sVz[b][tz][tx] = Vz;
    }
    const double gx = C.Dx * dPx, gz = C.Dz * dPz;
    const double spx = cpx + cp0, smx = cmx + cm0, spz = cpz + cp0, smz = cmz + cm0;
    const double Px = flux(spx, cpx, cp0, u0 - gx, C.Dx2), Mx = flux(smx, cmx, cm0, u0 + gx, C.Dx2);
    const double Pz = flux(spz, cpz, cp0, w0 - gz, C.Dz2), Mz = flux(smz, cmz, cm0, w0 + gz, C.Dz2);
    sPx[b][tz][tx] = Px;
    sMx[b][tz][tx] = Mx;
    sPz[b][tz][tx] = Pz;
    sMz[b][tz][tx] = Mz;
    if (wx && tx == TX - 1) {   // the x-faces at i + 1
      const double cpn = at(f.cp, oxp), cmn = at(f.cm, oxp);
      const double ge = C.Dx * (at(f.Phi, oxp) - Ph0);
      sE[b][tz][TX] = (w0 + wxp) * (at(f.u, km * nx + ip) + uxp);
      if (has_dn) sVx[b][tz][TX] = (q.wl2 * dn(f.u, oxp) + q.wu2 * uxp) * (vb + at(f.v, oxp));
      sPx[b][tz][TX] = flux(cp0 + cpn, cp0, cpn, uxp - ge, C.Dx2);
      sMx[b][tz][TX] = flux(cm0 + cmn, cm0, cmn, uxp + ge, C.Dx2);
    }
    if (wz && tz == TZ - 1) {   // the z-faces at k + 1
      const double cpn = at(f.cp, ozp), cmn = at(f.cm, ozp);
      const double ge = C.Dz * (at(f.Phi, ozp) - Ph0);
      sE[b][TZ][tx] = (at(f.w, kp * nx + im) + wzp) * (u0 + uzp);
      if (has_dn) sVz[b][TZ][tx] = (q.wl2 * dn(f.w, ozp) + q.wu2 * wzp) * (vb + at(f.v, ozp));
      sPz[b][TZ][tx] = flux(cp0 + cpn, cp0, cpn, wzp - ge, C.Dz2);
      sMz[b][TZ][tx] = flux(cm0 + cmn, cm0, cmn, wzp + ge, C.Dz2);
    }
    // ---- the next plane of this column ----
    const double vt = up(f.v, o0), vxt = up(f.v, oxm), vzt = up(f.v, ozm);   // v on face j + 1
    double u1 = 0.0, w1 = 0.0, Ph1 = 0.0, cp1 = 0.0, cm1 = 0.0, p1 = 0.0;
    if (has_up) {
      u1 = up(f.u, o0);
      w1 = up(f.w, o0);
      Ph1 = up(f.Phi, o0);
      cp1 = up(f.cp, o0);
      cm1 = up(f.cm, o0);
      p1 = up(f.p, o0);
    }
    const double sxt = vxt + vt, szt = vzt + vt;
    __syncthreads();   // this plane's faces (the buffer's last readers are a barrier behind)
    // ---- u ----
    {
      const double tt = has_up ? sxt * (u0 + u1) : 0.0;
      const double dt = (has_up ? u1 : walls ? f.wall_u[P + o0] : C.Uw) - u0;
      double left;
      if (wx && tx == 0) {
        const double a = uxm + u0;
        left = a * a;
      } else {
        left = sSu[b][tz][(tx - 1) & (TX - 1)];
      }
      double lap = C.nc * u0;
      lap += C.nxx * (uxm + uxp);
      lap += C.nzz * (uzm + uzp);
      double H = -C.K2x * ((spx - smx) * dPx);
      if (!AF) H += lap;
      H -= C.idx4 * (sSu[b][tz][tx] - left);
      H -= q.idy4 * (tt - tu);
      H -= C.idz4 * (sE[b][tzp][tx] - E);
      double r = C.gdt * H;
      if (C.zdt != 0.0) r += C.zdt * f.Hu[pj + o0];
      r -= C.adx * (p0 - at(f.p, oxm));
      r += q.uhi * dt;
      r -= q.ulo * du;
      if (AF) r += lap;
      f.ru[pj + o0] = r;
      f.Hu[pj + o0] = H;
      tu = tt;
      du = dt;
    }
    // ---- w ----
    {
      const double tt = has_up ? szt * (w0 + w1) : 0.0;
      const double dt = (has_up ? w1 : walls ? f.wall_w[P + o0] : 0.0) - w0;
      double front;
      if (wz && tz == 0) {
        const double a = wzm + w0;
        front = a * a;
      } else {
        front = sSw[b][(tz - 1) & (TZ - 1)][tx];
      }
      double lap = C.nc * w0;
      lap += C.nxx * (wxm + wxp);
      lap += C.nzz * (wzm + wzp);
      double H = -C.K2z * ((spz - smz) * dPz);
      if (!AF) H += lap;
      H -= C.idz4 * (sSw[b][tz][tx] - front);
      H -= q.idy4 * (tt - tw);
      H -= C.idx4 * (sE[b][tz][txp] - E);
      double r = C.gdt * H;
      if (C.zdt != 0.0) r += C.zdt * f.Hw[pj + o0];
      r -= C.adz * (p0 - at(f.p, ozm));
      r += q.uhi * dt;
      r -= q.ulo * dw;
      if (AF) r += lap;
      f.rw[pj + o0] = r;
      f.Hw[pj + o0] = H;
      tw = tt;
      dw = dt;
    }
    // ---- v on the face below ----
    {
      const double sv = vb + vt, tt = sv * sv, dt = vt - vb;
      if (has_dn) {
        double lap = C.nc * vb;
        lap += C.nxx * (vxm + at(f.v, oxp));
        lap += C.nzz * (vzm + at(f.v, ozp));
        double H = -q.K2ih * (rhoy * dPy);
        if (!AF) H += lap;
        H -= C.idx * (sVx[b][tz][txp] - Vx);
        H -= q.ih4 * (tt - tv);
        H -= C.idz * (sVz[b][tzp][tx] - Vz);
        double r = C.gdt * H;
        if (C.zdt != 0.0) r += C.zdt * f.Hv[pj + o0];
        r -= q.aih * (p0 - pd);
        r += q.vhi * dt;
        r -= q.vlo * dv;
        if (AF) r += lap;
        f.rv[pj + o0] = r;
        f.Hv[pj + o0] = H;
      }
      tv = tt;
      dv = dt;
    }
    // ---- ions ----
    {
      const double dPt = has_up ? Ph1 - Ph0 : 0.0, gy = q.Dihp * dPt;
      double lx = 0.0, mx = 0.0;
      if (AF) {
        lx = C.dc * cp0 + C.dxx * (cpx + at(f.cp, oxp)) + C.dzz * (cpz + at(f.cp, ozp));
        mx = C.dc * cm0 + C.dxx * (cmx + at(f.cm, oxp)) + C.dzz * (cmz + at(f.cm, ozp));
      }
      const double sp = cp0 + cp1, sm = cm0 + cm1;
      {
        const double tt = has_up ? sp * (vt - gy) : 0.0, dt = has_up ? cp1 - cp0 : 0.0;
        double H = -C.idx2 * (sPx[b][tz][txp] - Px);
        H -= q.idy2 * (tt - fp);
        H -= C.idz2 * (sPz[b][tzp][tx] - Pz);
        double r = C.gdt * H;
        if (C.zdt != 0.0) r += C.zdt * f.Hcp[pj + o0];
        r += q.chi * dt;
        r -= q.clo * dp;
        if (AF) r += lx;
        f.rcp[pj + o0] = r;
        f.Hcp[pj + o0] = H;
        fp = tt;
        dp = dt;
      }
      {
        const double tt = has_up ? sm * (vt + gy) : 0.0, dt = has_up ? cm1 - cm0 : 0.0;
        double H = -C.idx2 * (sMx[b][tz][txp] - Mx);
        H -= q.idy2 * (tt - fm);
        H -= C.idz2 * (sMz[b][tzp][tx] - Mz);
        double r = C.gdt * H;
        if (C.zdt != 0.0) r += C.zdt * f.Hcm[pj + o0];
        r += q.chi * dt;
        r -= q.clo * dm;
        if (AF) r += mx;
        f.rcm[pj + o0] = r;
        f.Hcm[pj + o0] = H;
        fm = tt;
        dm = dt;
      }
      dPy = dPt;
      rhoy = sp - sm;
    }
    ud = u0;
    wd = w0;
    svx = sxt;
    svz = szt;
    pd = p0;
    u0 = u1;
    w0 = w1;
    Ph0 = Ph1;
    cp0 = cp1;
    cm0 = cm1;
    p0 = p1;
    vb = vt;
    vxm = vxt;
    vzm = vzt;
  }
}

static cudaError_t launch_rhs_march(const Fields<double>& f, const Geo& g, const Metrics& m, const Phys& ph,
                                    const Stage& st, cudaStream_t s) {
  MarchCoef C{};
  C.idx4 = 0.25 * g.idx;
  C.idz4 = 0.25 * g.idz;
  C.idx2 = 0.5 * g.idx;
  C.idz2 = 0.5 * g.idz;
  C.idx = g.idx;
  C.idz = g.idz;
  const double xz = st.af ? st.dt * st.alp : 1.0;
  C.nxx = xz * ph.nu * (g.idx * g.idx);
  C.nzz = xz * ph.nu * (g.idz * g.idz);
  C.nc = -2.0 * (C.nxx + C.nzz);
  C.dxx = xz * ph.D * (g.idx * g.idx);
  C.dzz = xz * ph.D * (g.idz * g.idz);
  C.dc = -2.0 * (C.dxx + C.dzz);
  C.K2x = 0.5 * ph.K * g.idx;
  C.K2z = 0.5 * ph.K * g.idz;
  C.Dx = ph.D * g.idx;
  C.Dz = ph.D * g.idz;
  C.Dx2 = 2.0 * C.Dx;
  C.Dz2 = 2.0 * C.Dz;
  C.gdt = st.dt * st.gam;
  C.zdt = st.dt * st.zet;
  C.alpdt = st.dt * st.alp;
  C.adx = C.alpdt * g.idx;
  C.adz = C.alpdt * g.idz;
  C.anu = C.alpdt * ph.nu;
  C.aD = C.alpdt * ph.D;
  C.D = ph.D;
  C.K = ph.K;
  C.Uw = ph.Uw;
  auto go = [&](auto kern, int TX, int TZ) {
    const int tiles = (g.nx / TX) * (g.nz / TZ);
    int sms = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // chunks of up to eight planes (a chunk's first face costs a seventh of a
    // plane), shorter where that leaves an SM fewer than eight blocks
    const int jc = std::min(8, std::max(1, (int)((long long)g.nyc * tiles / (8 * sms))));
    const dim3 grd((unsigned)(g.nx / TX), (unsigned)(g.nz / TZ), (unsigned)((g.nyc + jc - 1) / jc));
    kern<<<grd, dim3(TX, TZ), sizeof(MarchPlane) * jc, s>>>(f, g, m, C, jc);
    return cudaGetLastError();
  };
  if (g.nx >= 128) return st.af ? go(k_rhs_march<128, 2, true>, 128, 2) : go(k_rhs_march<128, 2, false>, 128, 2);
  if (g.nx >= 64) return st.af ? go(k_rhs_march<64, 4, true>, 64, 4) : go(k_rhs_march<64, 4, false>, 64, 4);
  return st.af ? go(k_rhs_march<32, 4, true>, 32, 4) : go(k_rhs_march<32, 4, false>, 32, 4);
}

template <typename TV>
cudaError_t launch_rhs(const Fields<TV>& f, const Geo& g, const Metrics& m, const Phys& ph,
                       const Stage& st, cudaStream_t s) {
  if constexpr (sizeof(TV) == sizeof(double))
    if (g.nx >= 32 && g.lc_rhs_bx != 16) return launch_rhs_march(f, g, m, ph, st, s);   // nz >= 4: a power of two
  const int bx = g.lc_rhs_bx ? g.lc_rhs_bx : 32, by = 128 / bx;
  dim3 blk(bx, by, 1);
  dim3 grd((g.nx + bx - 1) / bx, (g.nz + by - 1) / by, g.nyc);
  k_rhs<TV><<<grd, blk, 0, s>>>(f, g, m, ph, st);
  return cudaGetLastError();
}

template cudaError_t launch_rhs<double>(const Fields<double>&, const Geo&, const Metrics&, const Phys&,
                                        const Stage&, cudaStream_t);
}  // namespace pnp
