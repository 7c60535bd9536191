// Initial condition, diagnostics and data movement for libpnp.
//
// Diagnostics follow the Numerical-methods definitions of arXiv:1701.02005:
// wall shear tau_w = (1/Re) d<u>/dy from the plane-averaged profile, total
// ion numbers (conserved: zero wall flux, Fig. 1 caption), net charge, max
// divergence (Eq. (2)).  All sums are FP64 with a fixed reduction order
// (deterministic across runs for a given grid).
#include <algorithm>
#include <mutex>

#include "pnp_common.cuh"
#include "pnp_df.cuh"
#include "pnp_mixed.cuh"

namespace pnp {

cudaError_t allow_smem(const void* kern, size_t smem) {
  if (smem <= 40 * 1024) return cudaSuccess;   // 48 KB with the kernel's static part need no asking
  static std::mutex one;
  const std::lock_guard<std::mutex> hold(one);
  cudaFuncAttributes a;
  const cudaError_t e = cudaFuncGetAttributes(&a, kern);
  if (e != cudaSuccess || (size_t)a.maxDynamicSharedSizeBytes >= smem) return e;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// SplitMix64 (Steele, Lea & Flood 2014) used as a counter-based generator:
// output n of the stream seeded by `seed` is mix(seed + (n + 1) * gamma).
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t n) {
  uint64_t x = seed + (n + 1ull) * 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// Uniform value in [-1, 1) for counter (field << 40) + index.
__device__ __forceinline__ double uniform_pm1(uint64_t seed, uint64_t field, uint64_t index) {
  const uint64_t b = splitmix64(seed, (field << 40) + index) >> 11;
  return (double)b * 0x1p-53 * 2.0 - 1.0;
}

template <typename TV>
__global__ void k_init_centres(Fields<TV> f, Geo g, Metrics m, Phys ph, int ic_kind, double cb, double kappa,
                               uint64_t seed, double amp) {
  const size_t n = (size_t)g.nyc * g.nz * g.nx;
  const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const int j = (int)(c / ((size_t)g.nz * g.nx));
  const double y = m.yc[j];
  double u = ph.Uw * y, w = 0.0;
  if (amp != 0.0) {
    const double env = amp * (1.0 - y * y);
    u = u + env * uniform_pm1(seed, 0, c);
    w = w + env * uniform_pm1(seed, 2, c);
  }
  double cp = 1.0, cm = 1.0;
  if (ic_kind == PNP_IC_PB && ph.V != 0.0) {
    // superposed Gouy-Chapman layers of the walls at y = +1 (+V) and y = -1 (-V)
    const double t = tanh(0.25 * ph.V);
    const double Pgc = 4.0 * atanh(t * exp(-(1.0 - y) * kappa)) - 4.0 * atanh(t * exp(-(1.0 + y) * kappa));
    cp = cb * exp(-Pgc);
    cm = cb * exp(Pgc);
  }
  f.u[c] = (TV)u;
  f.w[c] = (TV)w;
  f.p[c] = (TV)0;
  f.Hu[c] = (TV)0;
  f.Hw[c] = (TV)0;
  f.cp[c] = cp;
  f.cm[c] = cm;
  f.Hcp[c] = 0.0;
  f.Hcm[c] = 0.0;
}

template <typename TV>
__global__ void k_init_faces(Fields<TV> f, Geo g, const double* __restrict__ yf, uint64_t seed, double amp) {
  const size_t n = (size_t)g.ny * g.nz * g.nx;
  const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const int j = (int)(c / ((size_t)g.nz * g.nx));
  double v = 0.0;
  if (amp != 0.0 && j > 0 && j < g.ny - 1) {
    const double y = yf[j];
    v = amp * (1.0 - y * y) * uniform_pm1(seed, 1, c);
  }
  f.v[c] = (TV)v;
  f.Hv[c] = (TV)0;
  f.rv[c] = (TV)0;
}

template <typename TV>
cudaError_t launch_init_fields(const Fields<TV>& f, const Geo& g, const Metrics& m, const Phys& ph, int ic_kind,
                               double cb, double kappa, uint64_t seed, double amp, const double* yf,
                               cudaStream_t s) {
  const size_t nc = (size_t)g.nyc * g.nz * g.nx, nv = (size_t)g.ny * g.nz * g.nx;
  const int T = 256;
  k_init_centres<TV><<<(unsigned)((nc + T - 1) / T), T, 0, s>>>(f, g, m, ph, ic_kind, cb, kappa, seed, amp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_init_faces<TV><<<(unsigned)((nv + T - 1) / T), T, 0, s>>>(f, g, yf, seed, amp);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Diagnostics: per-block partial sums in a fixed order, then one block.
// Slots: 0 sum u(j=0), 1 sum u(j=nyc-1), 2 sum c+ dy, 3 sum c- dy, 4 max|div|,
// 5 sum (u^2 + w^2) dy + v^2 h, 6 count of non-finite values, 7 min(c+, c-),
// 8 max advective rate |u_c|/dx + |v_c|/dy + |w_c|/dz (cell-centred velocities;
// times dt it is the CFL number), 9 max |Phi difference| between neighbouring
// cells (x, z and interior y faces), 10 / 11 sum of the stored explicit ion
// terms H_c+ dy, H_c- dy (by the discrete divergence theorem minus the net
// ion flux through the two wall faces, per unit dx dz), 12 max migration rate
// over D: |dPhi_x|/dx^2 + |dPhi_y|/(h dy) + |dPhi_z|/dz^2 (the drift speed
// D |grad Phi| over the cell size), 13 max (c+ + c-) (times D / (2 lam^2) the
// dielectric relaxation rate).
// ---------------------------------------------------------------------------
constexpr int kDiagSlots = 14;
constexpr int kDiagThreads = 256;
constexpr int kDiagPairs = 15;   // paired (8-byte) inputs per cell pair of the mixed diagnostics
// its dynamic shared memory: two staging slots per thread, or the reduction buffer after the sweep
constexpr size_t kDiagMixedSmem = (size_t)2 * (kDiagPairs * 8 + 2 * 4) * kDiagThreads;

__device__ __forceinline__ bool diag_is_max(int q) { return q == 4 || q == 8 || q == 9 || q == 12 || q == 13; }

__device__ __forceinline__ void block_reduce(double* sh, double* vals, int tid) {
  // tree reduction of kDiagSlots values per thread; op: sum, except the maxima (4, 8, 9, 12, 13) and the minimum (7)
  for (int q = 0; q < kDiagSlots; ++q) sh[q * kDiagThreads + tid] = vals[q];
  __syncthreads();
  for (int st = kDiagThreads / 2; st > 0; st >>= 1) {
    if (tid < st) {
      for (int q = 0; q < kDiagSlots; ++q) {
        double a = sh[q * kDiagThreads + tid], b = sh[q * kDiagThreads + tid + st];
        sh[q * kDiagThreads + tid] = diag_is_max(q) ? fmax(a, b) : (q == 7 ? fmin(a, b) : a + b);
      }
    }
    __syncthreads();
  }
}

template <typename TV>
__global__ void __launch_bounds__(kDiagThreads) k_diag_partial(Fields<TV> f, Geo g, Metrics m, double* partial) {
  __shared__ double sh[kDiagSlots * kDiagThreads];
  double acc[kDiagSlots] = {0, 0, 0, 0, 0, 0, 0, 1e300, 0, 0, 0, 0, 0, 0};
  const size_t P = (size_t)g.nz * g.nx;
  const size_t nc = (size_t)g.nyc * P, nv = (size_t)g.ny * P;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += stride) {
    const int j = (int)(c / P);
    const int rem = (int)(c - (size_t)j * P);
    const int k = rem / g.nx, i = rem - k * g.nx;
    const int ip = (i + 1 == g.nx) ? 0 : i + 1, kp = (k + 1 == g.nz) ? 0 : k + 1;
    const double u = (double)f.u[c], w = (double)f.w[c];
    const double cp = f.cp[c], cm = f.cm[c];
    const double dy = 1.0 / m.idy[j];
    if (j == 0) acc[0] += u;
    if (j == g.nyc - 1) acc[1] += u;
    acc[2] += cp * dy;
    acc[3] += cm * dy;
    const double div = ((double)f.u[cidx(j, k, ip, g.nz, g.nx)] - u) * g.idx +
                       ((double)f.v[c + P] - (double)f.v[c]) * m.idy[j] +
                       ((double)f.w[cidx(j, kp, i, g.nz, g.nx)] - w) * g.idz;
    acc[4] = fmax(acc[4], fabs(div));
    acc[5] += (u * u + w * w) * dy;
    const double ue = (double)f.u[cidx(j, k, ip, g.nz, g.nx)], wn = (double)f.w[cidx(j, kp, i, g.nz, g.nx)];
    const double rate = fabs(0.5 * (u + ue)) * g.idx + fabs(0.5 * ((double)f.v[c] + (double)f.v[c + P])) * m.idy[j] +
                        fabs(0.5 * (w + wn)) * g.idz;
    acc[8] = fmax(acc[8], rate);
    const double p = (double)f.p[c], Ph = f.Phi[c];
    const double dpx = fabs(f.Phi[cidx(j, k, ip, g.nz, g.nx)] - Ph), dpz = fabs(f.Phi[cidx(j, kp, i, g.nz, g.nx)] - Ph);
    const double dpy = j + 1 < g.nyc ? fabs(f.Phi[c + P] - Ph) : 0.0;
    acc[9] = fmax(acc[9], fmax(fmax(dpx, dpz), dpy));
    acc[12] = fmax(acc[12], dpx * g.idx * g.idx + dpy * m.ih[j + 1] * m.idy[j] + dpz * g.idz * g.idz);
    acc[13] = fmax(acc[13], cp + cm);
    acc[10] += f.Hcp[c] * dy;
    acc[11] += f.Hcm[c] * dy;
    if (!isfinite(u) || !isfinite(w) || !isfinite(cp) || !isfinite(cm) || !isfinite(p) || !isfinite(Ph) ||
        !isfinite(div))
      acc[6] += 1.0;
    acc[7] = fmin(acc[7], fmin(cp, cm));
  }
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < nv; c += stride) {
    const int j = (int)(c / P);
    const double v = (double)f.v[c];
    acc[5] += v * v / m.ih[j];
    if (!isfinite(v)) acc[6] += 1.0;
  }
  block_reduce(sh, acc, threadIdx.x);
  if (threadIdx.x == 0)
    for (int q = 0; q < kDiagSlots; ++q) partial[(size_t)blockIdx.x * kDiagSlots + q] = sh[q * kDiagThreads];
}

// Two df values side by side, one per lane of a float2, for the packed FP32
// instructions (each lane rounded to nearest, never contracted): the same
// error-free transforms as pnp_df.cuh, lane by lane.
struct dfl2 {
  float2 h, l;
};
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) {   // a - b, one rounding
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p_abs(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ dfl2 p_two_sum(float2 a, float2 b) {
  const float2 s = p_add(a, b), bb = p_sub(s, a);
  return {s, p_add(p_sub(a, p_sub(s, bb)), p_sub(b, bb))};
}
__device__ __forceinline__ dfl2 p_fast_two_sum(float2 a, float2 b) {
  const float2 s = p_add(a, b);
  return {s, p_sub(b, p_sub(s, a))};
}
__device__ __forceinline__ dfl2 p_add_fast(dfl2 x, dfl2 y) {
  const dfl2 s = p_two_sum(x.h, y.h);
  return p_fast_two_sum(s.h, p_add(s.l, p_add(x.l, y.l)));
}
__device__ __forceinline__ dfl2 p_prod(float2 a, float2 b) {
  const float2 p = p_mul(a, b);
  return {p, p_fma(a, b, p_mul(p, make_float2(-1.f, -1.f)))};
}

// Mixed precision: the same partial sums straight from the FP32 fields and the
// df ion state c = c_ref + S + L, with no FP64 copy of the state and no FP64
// arithmetic per cell.  A block takes a contiguous range of x-rows, so a
// thread's rows share their plane j for long runs: per run it sums u^2 + w^2,
// v^2 (exact squares) and the ion fluctuations S + L in df on the FP32 pipe and
// weights the run's sums by dy_j and h_j (df pairs) once.  The per-thread sums
// go to FP64 once and the block reduces them in FP64 in a fixed order; the
// reference part of the ion numbers, sum_j c_ref(j) dy_j over the plane, is
// added on the host.  The divergence is summed in df from exact differences
// (TwoSum) times df coefficients, so that its small value keeps its FP64
// accuracy; the minimum concentration is FP32; a cell is counted non-finite
// when any input read for it is.  Each thread stages its next cell pair's
// inputs in its own shared-memory slot by cp.async while it sums the current
// pair.  Nx and Nz are powers of two.
__global__ void __launch_bounds__(kDiagThreads, 2) k_diag_partial_mixed(Fields<float> f, Shadows sh,
                                                                        const float* __restrict__ cref_p,
                                                                        const float* __restrict__ cref_m,
                                                                        const float* __restrict__ dPref,
                                                                        const float2* __restrict__ wgt, Geo g,
                                                                        double* partial) {
  // dynamic shared memory: the threads' staging slots during the sweep, the
  // block reduction's buffer after it
  extern __shared__ __align__(16) unsigned char diag_smem[];
  double* shr = reinterpret_cast<double*>(diag_smem);
  float2* st2 = reinterpret_cast<float2*>(diag_smem);                                            // [2][kDiagPairs][threads]
  float* st1 = reinterpret_cast<float*>(diag_smem + (size_t)2 * kDiagPairs * kDiagThreads * 8);  // [2][2][threads]
  const int tid = threadIdx.x;
  dfl sum[7] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};   // 0-3, 5, 10, 11
  float maxdiv = 0.f, bad = 0.f, cmin = 3.0e38f, maxrate = 0.f, maxdphi = 0.f, maxmig = 0.f, maxcsum = 0.f;
  const int nx = g.nx, nz = g.nz, lnz = __ffs(nz) - 1;
  const size_t P = (size_t)nz * nx;
  const int rows = g.nyc * nz, per = (rows + gridDim.x - 1) / gridDim.x;
  const int r0 = blockIdx.x * per, r1 = min(rows, r0 + per);
  // two cells per thread (paired 8-byte copies); the block's threads cover
  // `rpp` rows at a time, each thread keeping to one row in rpp and taking
  // `nib` cell pairs of it
  const int tpr = min((int)blockDim.x, nx / 2), rpp = (int)blockDim.x / tpr, nib = nx / (2 * tpr);
  const int sub = tid / tpr, tx = tid - sub * tpr;
  // 1/dx, 1/dz as df pairs (per thread, once)
  const float idxh = (float)g.idx, idzh = (float)g.idz;
  const dfl idx{idxh, (float)(g.idx - (double)idxh)}, idz{idzh, (float)(g.idz - (double)idzh)};
  const float2 idxh2 = make_float2(idx.h, idx.h), idxl2 = make_float2(idx.l, idx.l);
  const float2 idzh2 = make_float2(idz.h, idz.h), idzl2 = make_float2(idz.l, idz.l);
  // work item q of this thread: row r, first cell i
  auto item = [&](int q, int& r, int& i) {
    const int a = q / nib, b = q - a * nib;
    r = r0 + sub + rpp * a;
    i = 2 * tx + 2 * tpr * b;
    return sub < rpp && r < r1;
  };
  // the item's inputs into this thread's staging slot (only this thread reads
  // them: no barrier); one commit group per item
  auto issue = [&](int slot, int r, int i) {
    const int j = r >> lnz, kp = ((r & (nz - 1)) + 1) & (nz - 1);
    const size_t c = (size_t)r * nx + i, ckp = ((size_t)j * nz + kp) * nx + i;
    const size_t ce = (size_t)r * nx + ((i + 2) & (nx - 1));
    const float* src[kDiagPairs] = {f.u + c,   f.w + c,    f.p + c,    sh.phi + c, f.v + c,    f.v + c + P,
                                    f.w + ckp, sh.phi + ckp, sh.cp + c, sh.cpL + c, sh.cm + c, sh.cmL + c,
                                    sh.Hcp + c, sh.Hcm + c, sh.phi + c + P};
    const int npair = j + 1 < g.nyc ? kDiagPairs : kDiagPairs - 1;   // no plane above the last one
#pragma unroll
    for (int k = 0; k < kDiagPairs; ++k) {
      if (k >= npair) continue;
      const unsigned d = (unsigned)__cvta_generic_to_shared(st2 + ((size_t)slot * kDiagPairs + k) * kDiagThreads + tid);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src[k]) : "memory");
    }
    const float* one[2] = {f.u + ce, sh.phi + ce};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const unsigned d = (unsigned)__cvta_generic_to_shared(st1 + ((size_t)slot * 2 + k) * kDiagThreads + tid);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(one[k]) : "memory");
    }
  };
  // the current run of rows in plane jr: sums still to be weighted
  int jr = (r0 + sub) >> lnz;
  // the run's sums, one df value per lane (even and odd cells of the pairs)
  const dfl2 z2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  dfl2 ruw = z2, rv = z2, rcp = z2, rcm = z2, ru = z2, rhp = z2, rhm = z2;
  bool any = false;
  auto flush = [&]() {
    const float2 dyw = wgt[jr], hw = wgt[g.ny + jr];
    const dfl dy{dyw.x, dyw.y}, h{hw.x, hw.y};
    auto lanes = [](dfl2 x) { return df_add(dfl{x.h.x, x.l.x}, dfl{x.h.y, x.l.y}); };
    sum[4] = df_add(sum[4], df_add(df_mul(lanes(ruw), dy), df_mul(lanes(rv), h)));
    sum[2] = df_add(sum[2], df_mul(lanes(rcp), dy));
    sum[3] = df_add(sum[3], df_mul(lanes(rcm), dy));
    sum[5] = df_add(sum[5], df_mul(lanes(rhp), dy));
    sum[6] = df_add(sum[6], df_mul(lanes(rhm), dy));
    if (jr == 0) sum[0] = df_add(sum[0], lanes(ru));
    if (jr == g.nyc - 1) sum[1] = df_add(sum[1], lanes(ru));
    ruw = rv = rcp = rcm = ru = rhp = rhm = z2;
  };
  int r = 0, i = 0;
  bool have = item(0, r, i);
  if (have) issue(0, r, i);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int q = 0; have; ++q) {
    int rn = 0, in = 0;
    const bool hn = item(q + 1, rn, in);
    if (hn) issue((q + 1) & 1, rn, in);   // the next item's copies fly while this one is summed
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");   // this item's copies (this thread's own)
    const int j = r >> lnz;
    if (j != jr) {
      flush();
      jr = j;
    }
    any = true;
    const bool wall_row = j == 0 || j == g.nyc - 1;   // the only rows whose sum of u is kept
    const float2 iyw = wgt[2 * g.ny + j];
    const dfl iy{iyw.x, iyw.y};
    const float crp = cref_p[j], crm = cref_m[j];
    const bool top = j + 1 < g.nyc;
    const float dpy = top ? dPref[j + 1] : 0.f;   // Phi_ref step across face j+1 (interior faces)
    const float ihy = top ? 1.f / wgt[g.ny + j + 1].x : 0.f;   // 1 / h of that face
    const float2* s2 = st2 + (size_t)(q & 1) * kDiagPairs * kDiagThreads + tid;
    const float* s1 = st1 + (size_t)(q & 1) * 2 * kDiagThreads + tid;
    const float2 u = s2[0], w = s2[kDiagThreads], p = s2[2 * kDiagThreads], ph = s2[3 * kDiagThreads];
    const float2 v0 = s2[4 * kDiagThreads], v1 = s2[5 * kDiagThreads], wn = s2[6 * kDiagThreads];
    const float2 phn = s2[7 * kDiagThreads], Sp = s2[8 * kDiagThreads], Lp = s2[9 * kDiagThreads];
    const float2 Sm = s2[10 * kDiagThreads], Lm = s2[11 * kDiagThreads], Hp = s2[12 * kDiagThreads];
    const float2 Hm = s2[13 * kDiagThreads];
    const float2 phu = top ? s2[14 * kDiagThreads] : make_float2(0.f, 0.f);
    const float ue2 = s1[0], phe2 = s1[kDiagThreads];
    // the pair's two cells side by side in packed FP32 (lane x: cell i, lane y:
    // cell i + 1), with their neighbours east (+x), north (+z) and above (+y)
    const float2 ue = make_float2(u.y, ue2), phe = make_float2(ph.y, phe2);
    const float2 m1 = make_float2(-1.f, -1.f), zero = make_float2(0.f, 0.f);
    if (wall_row) ru = p_add_fast(ru, dfl2{u, zero});
    ruw = p_add_fast(ruw, p_add_fast(p_prod(u, u), p_prod(w, w)));
    rv = p_add_fast(rv, p_prod(v0, v0));
    rcp = p_add_fast(rcp, dfl2{Sp, Lp});
    rcm = p_add_fast(rcm, dfl2{Sm, Lm});
    rhp = p_add_fast(rhp, dfl2{Hp, zero});
    rhm = p_add_fast(rhm, dfl2{Hm, zero});
    // the divergence of the stored fields in df: exact differences (TwoSum),
    // exact leading products (TwoProduct) and the cross terms with the df
    // coefficients, the three leading parts summed by TwoSum, the rest in FP32
    const float2 iyh = make_float2(iy.h, iy.h), iyl = make_float2(iy.l, iy.l);
    const dfl2 a1 = p_two_sum(ue, p_mul(u, m1)), a2 = p_two_sum(v1, p_mul(v0, m1)), a3 = p_two_sum(wn, p_mul(w, m1));
    const dfl2 p1 = p_prod(a1.h, idxh2), p2 = p_prod(a2.h, iyh), p3 = p_prod(a3.h, idzh2);
    const dfl2 q1 = p_two_sum(p1.h, p2.h), q2 = p_two_sum(q1.h, p3.h);
    float2 lo = p_add(p_add(p1.l, p2.l), p3.l);
    lo = p_fma(a1.h, idxl2, lo);
    lo = p_fma(a1.l, idxh2, lo);
    lo = p_fma(a2.h, iyl, lo);
    lo = p_fma(a2.l, iyh, lo);
    lo = p_fma(a3.h, idzl2, lo);
    lo = p_fma(a3.l, idzh2, lo);
    const float2 dv = p_add(q2.h, p_add(lo, p_add(q1.l, q2.l)));
    maxdiv = fmaxf(maxdiv, fmaxf(fabsf(dv.x), fabsf(dv.y)));
    // non-finite inputs: x - x is 0 for a finite x and NaN otherwise (dv is
    // non-finite when u, ue, v0, v1, w or wn is); a cell counts once
    const float2 nf = p_add(p_add(p_sub(dv, dv), p_sub(Sp, Sp)), p_add(p_add(p_sub(Sm, Sm), p_sub(p, p)), p_sub(ph, ph)));
    bad += (nf.x != 0.f ? 1.f : 0.f) + (nf.y != 0.f ? 1.f : 0.f);
    const float2 ctp = p_add(make_float2(crp, crp), Sp), ctm = p_add(make_float2(crm, crm), Sm);
    cmin = fminf(cmin, fminf(fminf(ctp.x, ctp.y), fminf(ctm.x, ctm.y)));
    const float2 cs = p_add(ctp, ctm);
    maxcsum = fmaxf(maxcsum, fmaxf(cs.x, cs.y));
    const float2 hf = make_float2(0.5f, 0.5f);
    const float2 rate = p_fma(p_abs(p_mul(hf, p_add(u, ue))), idxh2,
                              p_fma(p_abs(p_mul(hf, p_add(v0, v1))), make_float2(iyw.x, iyw.x),
                                    p_mul(p_abs(p_mul(hf, p_add(w, wn))), idzh2)));
    maxrate = fmaxf(maxrate, fmaxf(rate.x, rate.y));
    const float2 dpx = p_abs(p_sub(phe, ph)), dpz = p_abs(p_sub(phn, ph));
    const float2 dpyc = top ? p_abs(p_add(make_float2(dpy, dpy), p_sub(phu, ph))) : zero;
    maxdphi = fmaxf(maxdphi, fmaxf(fmaxf(fmaxf(dpx.x, dpx.y), fmaxf(dpz.x, dpz.y)), fmaxf(dpyc.x, dpyc.y)));
    const float2 mig = p_fma(p_mul(dpx, idxh2), idxh2,
                             p_fma(p_mul(dpyc, make_float2(ihy, ihy)), make_float2(iyw.x, iyw.x),
                                   p_mul(p_mul(dpz, idzh2), idzh2)));
    maxmig = fmaxf(maxmig, fmaxf(mig.x, mig.y));
    r = rn;
    i = in;
    have = hn;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();   // the staging slots become the reduction's buffer
  if (any) flush();
  // the top wall face of v
  const size_t nc = (size_t)g.nyc * P;
  const float2 hw = wgt[g.ny + g.nyc];
  for (size_t c = nc + (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < nc + P; c += (size_t)gridDim.x * blockDim.x) {
    const float v = f.v[c];
    sum[4] = df_add(sum[4], df_mul(df_prod(v, v), dfl{hw.x, hw.y}));
    if (!isfinite(v)) bad += 1.f;
  }
  auto d = [](dfl x) { return (double)x.h + (double)x.l; };
  double acc[kDiagSlots] = {d(sum[0]), d(sum[1]), d(sum[2]), d(sum[3]), (double)maxdiv, d(sum[4]), (double)bad,
                            (double)cmin, (double)maxrate, (double)maxdphi, d(sum[5]), d(sum[6]), (double)maxmig,
                            (double)maxcsum};
  block_reduce(shr, acc, threadIdx.x);
  if (threadIdx.x == 0)
    for (int q = 0; q < kDiagSlots; ++q) partial[(size_t)blockIdx.x * kDiagSlots + q] = shr[q * kDiagThreads];
}

// Final reduction and the device status word: a non-finite value, a negative
// concentration, an advective CFL number (rate x dt, dt > 0 the last step's
// size) above cfl_max, or a potential step between neighbouring cells above
// dphi_max, in that order of precedence.
__global__ void __launch_bounds__(kDiagThreads) k_diag_final(const double* partial, int npartial, double* out,
                                                            int* status, DiagLimits lim) {
  __shared__ double sh[kDiagSlots * kDiagThreads];
  double acc[kDiagSlots] = {0, 0, 0, 0, 0, 0, 0, 1e300, 0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < npartial; b += blockDim.x) {
    for (int q = 0; q < kDiagSlots; ++q) {
      const double v = partial[(size_t)b * kDiagSlots + q];
      acc[q] = diag_is_max(q) ? fmax(acc[q], v) : (q == 7 ? fmin(acc[q], v) : acc[q] + v);
    }
  }
  block_reduce(sh, acc, threadIdx.x);
  if (threadIdx.x == 0) {
    for (int q = 0; q < kDiagSlots; ++q) out[q] = sh[q * kDiagThreads];
    int st = PNP_OK;
    if (sh[6 * kDiagThreads] > 0.0) st = PNP_ERR_NONFINITE;
    else if (sh[7 * kDiagThreads] < 0.0) st = PNP_ERR_NEGATIVE_C;
    else if (lim.dt > 0.0 && sh[8 * kDiagThreads] * lim.dt > lim.cfl_max) st = PNP_ERR_CFL;
    else if (sh[9 * kDiagThreads] > lim.dphi_max) st = PNP_ERR_DPHI;
    *status = st;
  }
}

template <typename TV>
cudaError_t launch_diagnostics(const Fields<TV>& f, const Geo& g, const Metrics& m, const Phys& ph,
                               double* partial, int npartial, double* out, int* status, const DiagLimits& lim,
                               cudaStream_t s) {
  (void)ph;
  k_diag_partial<TV><<<npartial, kDiagThreads, 0, s>>>(f, g, m, partial);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_diag_final<<<1, kDiagThreads, 0, s>>>(partial, npartial, out, status, lim);
  return cudaGetLastError();
}

cudaError_t launch_diagnostics_mixed(const Fields<float>& f, const Shadows& sh, const float* cref_p,
                                     const float* cref_m, const float* dPref, const float2* wgt, const Geo& g,
                                     double* partial, int npartial, double* out, int* status,
                                     const DiagLimits& lim, cudaStream_t s) {
  // one resident wave: two 256-thread blocks per SM (up to 128 registers a thread:
  // two cells each, the double-float sums of the row runs kept in registers)
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int nb = std::max(1, std::min(npartial, 2 * sms));
  static_assert(kDiagMixedSmem >= (size_t)kDiagSlots * kDiagThreads * sizeof(double), "reduction buffer");
  e = cudaFuncSetAttribute(k_diag_partial_mixed, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDiagMixedSmem);
  if (e != cudaSuccess) return e;
  k_diag_partial_mixed<<<nb, kDiagThreads, kDiagMixedSmem, s>>>(f, sh, cref_p, cref_m, dPref, wgt, g, partial);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_diag_final<<<1, kDiagThreads, 0, s>>>(partial, nb, out, status, lim);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
template <typename TA, typename TB>
__global__ void k_convert(const TA* __restrict__ a, TB* __restrict__ b, size_t n) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (TB)a[i];
}

template <typename TA, typename TB>
cudaError_t launch_convert(const TA* a, TB* b, size_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int T = 256;
  k_convert<TA, TB><<<(unsigned)((n + T - 1) / T), T, 0, s>>>(a, b, n);
  return cudaGetLastError();
}

// Plane mean of q over plane `plane` (block per plane when plane < 0).
template <typename TQ>
__global__ void k_mean_profile(const TQ* __restrict__ q, size_t P, double* out) {
  __shared__ double sh[256];
  const int j = blockIdx.x;
  double acc = 0.0;
  for (size_t c = threadIdx.x; c < P; c += blockDim.x) acc += (double)q[(size_t)j * P + c];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if (threadIdx.x < st) sh[threadIdx.x] += sh[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[j] = sh[0] / (double)P;
}

template <typename TQ>
cudaError_t launch_mean_profile(const TQ* q, int nplanes, int plane_size, double* out, cudaStream_t s) {
  k_mean_profile<TQ><<<nplanes, 256, 0, s>>>(q, (size_t)plane_size, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Statistics: plane means of q and q^2 for u, v, w, c+, c-, Phi of the current
// state, added to the accumulators acc[(2 q + 0 | 1) ny + j] (one block per
// plane, fixed reduction order).  The mixed path reads the FP32 velocities,
// the double-float ion state c = c_ref + S + L and Phi = Phi_ref + phi'; every
// per-cell value is formed and squared in FP64.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_stats_sample(StatSrc src, Geo g, double* __restrict__ acc) {
  __shared__ double sh[12 * 256];
  const int j = blockIdx.x;
  const size_t P = (size_t)g.nz * g.nx;
  double a[12];
#pragma unroll
  for (int q = 0; q < 12; ++q) a[q] = 0.0;
  auto vel = [&](const void* p, size_t c) {
    return src.vel_f32 ? (double)static_cast<const float*>(p)[c] : static_cast<const double*>(p)[c];
  };
  for (size_t r = threadIdx.x; r < P; r += blockDim.x) {
    const size_t c = (size_t)j * P + r;
    const double v = vel(src.v, c);
    a[2] += v;
    a[3] += v * v;
    if (j < g.nyc) {
      const double u = vel(src.u, c), w = vel(src.w, c);
      double cp, cm, ph;
      if (src.mixed) {
        cp = src.cref_p[j] + ((double)src.cpS[c] + (double)src.cpL[c]);
        cm = src.cref_m[j] + ((double)src.cmS[c] + (double)src.cmL[c]);
        ph = src.phi_ref[j] + (double)src.phiS[c];
      } else {
        cp = src.cp[c];
        cm = src.cm[c];
        ph = src.Phi[c];
      }
      a[0] += u; a[1] += u * u;
      a[4] += w; a[5] += w * w;
      a[6] += cp; a[7] += cp * cp;
      a[8] += cm; a[9] += cm * cm;
      a[10] += ph; a[11] += ph * ph;
    }
  }
  for (int q = 0; q < 12; ++q) sh[q * 256 + threadIdx.x] = a[q];
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if (threadIdx.x < st)
      for (int q = 0; q < 12; ++q) sh[q * 256 + threadIdx.x] += sh[q * 256 + threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x < 12) {
    const int q = threadIdx.x;   // slot order u, u2, v, v2, w, w2, c+, c+2, c-, c-2, Phi, Phi2
    const bool cell = q < 2 || q >= 4;
    if (!cell || j < g.nyc) acc[(size_t)q * g.ny + j] += sh[q * 256] / (double)P;
  }
}

cudaError_t launch_stats_sample(const StatSrc& src, const Geo& g, double* acc, cudaStream_t s) {
  k_stats_sample<<<g.ny, 256, 0, s>>>(src, g, acc);
  return cudaGetLastError();
}

// FP64 FMA throughput probe: 8 independent dependency chains per thread.
__global__ void k_fp64_probe(double* out, int iters) {
  double x0 = threadIdx.x * 1e-3, x1 = x0 + 1, x2 = x0 + 2, x3 = x0 + 3;
  double x4 = x0 + 4, x5 = x0 + 5, x6 = x0 + 6, x7 = x0 + 7;
  const double a = 0.999, b = 1e-3;
  for (int i = 0; i < iters; ++i) {
    x0 = fma(x0, a, b); x1 = fma(x1, a, b); x2 = fma(x2, a, b); x3 = fma(x3, a, b);
    x4 = fma(x4, a, b); x5 = fma(x5, a, b); x6 = fma(x6, a, b); x7 = fma(x7, a, b);
  }
  out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = x0 + x1 + x2 + x3 + x4 + x5 + x6 + x7;
}

cudaError_t launch_fp64_probe(double* out, int iters, int blocks, cudaStream_t s) {
  k_fp64_probe<<<blocks, 256, 0, s>>>(out, iters);
  return cudaGetLastError();
}

template cudaError_t launch_init_fields<double>(const Fields<double>&, const Geo&, const Metrics&, const Phys&, int,
                                                double, double, uint64_t, double, const double*, cudaStream_t);
template cudaError_t launch_init_fields<float>(const Fields<float>&, const Geo&, const Metrics&, const Phys&, int,
                                               double, double, uint64_t, double, const double*, cudaStream_t);
// ---------------------------------------------------------------------------
// Wall potentials that vary along the walls (the walls may carry any
// potential): Phi = V y + off + lift + phi, lift the charge-free potential between
// the walls' variations.
// ---------------------------------------------------------------------------
// What the wall values leave on the right of the first and last cell planes' rows.
__global__ void k_wall_rows(double* __restrict__ src, const double* __restrict__ B, const double* __restrict__ T,
                            double Bm, double Tm, double cb, double ct, int P) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= P) return;
  src[r] = cb * (B[r] - Bm);
  src[P + r] = ct * (T[r] - Tm);
}

cudaError_t launch_wall_rows(double* src, const double* B, const double* T, double Bm, double Tm, double cb, double ct,
                             const Geo& g, cudaStream_t s) {
  const int P = g.nz * g.nx;
  k_wall_rows<<<(P + 255) / 256, 256, 0, s>>>(src, B, T, Bm, Tm, cb, ct, P);
  return cudaGetLastError();
}

__global__ void k_lift_copy(double* __restrict__ lift64, float* __restrict__ lift32, double off, size_t n) {
  const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const double v = lift64[c];
  lift32[c] = (float)v;
  if (off != 0.0) lift64[c] = v + off;
}

cudaError_t launch_lift_copy(double* lift64, float* lift32, double off, size_t n, cudaStream_t s) {
  k_lift_copy<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(lift64, lift32, off, n);
  return cudaGetLastError();
}

template cudaError_t launch_diagnostics<double>(const Fields<double>&, const Geo&, const Metrics&, const Phys&,
                                                double*, int, double*, int*, const DiagLimits&, cudaStream_t);
template cudaError_t launch_diagnostics<float>(const Fields<float>&, const Geo&, const Metrics&, const Phys&,
                                               double*, int, double*, int*, const DiagLimits&, cudaStream_t);
template cudaError_t launch_convert<double, double>(const double*, double*, size_t, cudaStream_t);
template cudaError_t launch_convert<double, float>(const double*, float*, size_t, cudaStream_t);
template cudaError_t launch_convert<float, double>(const float*, double*, size_t, cudaStream_t);
template cudaError_t launch_mean_profile<double>(const double*, int, int, double*, cudaStream_t);
template cudaError_t launch_mean_profile<float>(const float*, int, int, double*, cudaStream_t);

}  // namespace pnp
