// Kalman re-fit of tracks (the paper's "fitting" step, Sec. 5): one thread
// per track, state and covariance in registers, from the seed prior placed at
// the first hit over the track's hits layer by layer.  The result is the
// state after the last hit, before its scattering, and the summed chi2 of the
// predicted residuals.
//
// Conditioning: where a track crosses a layer close to tangentially (the
// looper at the end of its reach), the propagation Jacobian grows like
// 1/cos(alpha) and the predicted covariance gains a large, nearly rank-one
// term that the update then removes again; FP32 loses the posterior there.
// A first FP32 pass fits every track and stops a track at the first of its
// crossings with cos(alpha) below CAREFUL_COS; a second pass takes the listed
// tracks on from there, running such steps' propagation and update in double
// precision (a small fraction of tracks: loopers near their maximum radius).
// On a detector with endcap disks, a plane step along more than half a
// radian of the helix (a looper reaching a disk) flags its track the same
// way (PLANE_CAREFUL_PSI).
#include <algorithm>

#include "kf_internal.h"

namespace kfg {

namespace {

constexpr float CAREFUL_COS = 0.5f;
constexpr int FIT_THREADS = 128;  // threads per block of the FP32 pass

// One Kalman step on an endcap disk in scalar type T (the plane, the (r-phi, r)
// measurement, the disk's scattering and loss).
template <class T>
__device__ __forceinline__ int disk_step(const DevGeom& g, T (&p)[6], T (&C)[21], bool first, bool last, int L,
                                         float mx, float my, float& chi2) {
  if (!first && !propagate_plane<T, true>(p, C, (T)plane_z(g, L), field_kb<T>(g, p))) return KF_FIT_NO_CROSS;
  DiskFrameT<T> d;
  make_frame_disk<T>(p, C, (T)g.vr, (T)g.vrr, d);
  T r0, r1;
  if (!residual_disk<T>(p, d.f, (T)mx, (T)my, r0, r1)) return KF_FIT_FAR_SIDE;
  chi2 += (float)chi2_of<T>(d.f, r0, r1);
  kf_update_disk<T>(p, C, d, r0, r1);
  if (!last) {
    add_ms_disk<T>(p, C, (T)g.disk_x0);
    add_eloss_ool<T, true, true>(p, C, (T)g.disk_eloss);
  }
  return KF_FIT_OK;
}

// add_ms in double with its quotients resolved: with w = |q/pT| sin(theta),
// 0.0136/(beta p) = 0.0136 w sqrt(1 + m^2 w^2), and Var(phi) = Var(theta) /
// sin^2(theta) without the sine.  One quotient and three roots instead of six
// and three: a double-precision quotient takes its unit about 700 clocks.
__device__ __forceinline__ void add_ms_double(const double (&p)[6], double (&C)[21], double x0) {
  if (p[3] == 0.0 || x0 <= 0.0) return;
  double sth, cth, sph, cph;
  sincos(p[5], &sth, &cth);
  sincos(p[4], &sph, &cph);
  const double cd = fma(cph, p[0], sph * p[1]) * rsqrt(fma(p[0], p[0], p[1] * p[1]));
  const double t = x0 / fabs(sth * cd);
  const double w = fabs(p[3]) * sth;
  const double tp = 0.0136 * fabs(p[3]) * sqrt(fma(MPION * MPION * w, w, 1.0)) * sqrt(t) * fma(0.038, log(t), 1.0);
  const double tt = tp * sth;
  C[S6(4, 4)] = fma(tp, tp, C[S6(4, 4)]);
  C[S6(5, 5)] = fma(tt, tt, C[S6(5, 5)]);
}

// One Kalman step in scalar type T: propagate (unless first), update with the
// corrected hit, scatter unless last.  Returns a KF_FIT_* status.  The fit
// takes the library's sine and cosine throughout (ACC).
template <class T, bool DISK>
__device__ __forceinline__ int fit_step(const DevGeom& g, float (&pf)[6], float (&Cf)[21], bool first,
                                        bool last, int L, float mx, float my, float mz, float& chi2) {
  T p[6], C[21];
#pragma unroll
  for (int k = 0; k < 6; ++k) p[k] = (T)pf[k];
#pragma unroll
  for (int k = 0; k < 21; ++k) C[k] = (T)Cf[k];
  if (DISK && is_disk(g, L)) {
    const int rc = disk_step<T>(g, p, C, first, last, L, mx, my, chi2);
    if (rc != KF_FIT_OK) return rc;
#pragma unroll
    for (int k = 0; k < 6; ++k) pf[k] = (float)p[k];
#pragma unroll
    for (int k = 0; k < 21; ++k) Cf[k] = (float)C[k];
    return KF_FIT_OK;
  }
  if (!first && propagate<T, true>(p, C, (T)g.radius[L], field_kb<T>(g, p), T(INFINITY)) != 1)
    return KF_FIT_NO_CROSS;
  FrameT<T> f;
  make_frame<T>(p, C, (T)g.vr, (T)g.vz, f);
  T r0, r1;
  if (!residual<T>(p, f, (T)mx, (T)my, (T)mz, r0, r1)) return KF_FIT_FAR_SIDE;
  chi2 += (float)chi2_of<T>(f, r0, r1);
  kf_update<T>(p, C, f, r0, r1);
  if (!last) {
    if constexpr (sizeof(T) == 8) add_ms_double(p, C, x0_at<T>(g, L, p[2]));
    else add_ms<T, true>(p, C, x0_at<T>(g, L, p[2]));
    add_eloss_ool<T, false, true>(p, C, (T)g.eloss[L]);
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) pf[k] = (float)p[k];
#pragma unroll
  for (int k = 0; k < 21; ++k) Cf[k] = (float)C[k];
  return KF_FIT_OK;
}

// A double-precision step onto a barrel layer (not a track's first) by a whole
// warp on one track: every lane holds the state and calls this with the same
// arguments.  A double-precision instruction takes its unit 64 clocks for a
// warp, whatever its active lanes, so that the step's time is its number of
// instructions: the sines and cosines of both angles, the quotients, the
// series of the helix functions, the Jacobian's entries, the rows of J C J^T
// and of the gain and the update are each one instruction sequence over as
// many lanes.  The operations and their order are fit_step's, element by
// element (a term with a structural zero or one of J adds exactly), so that a
// track's fit does not depend on how many others were listed.  The careful pass
// of a 2,500-track event: 90 us in one lane per track, 68 so.
struct CoopMem {
  double C[36], J[36], T[36], a0[6], k0[6], k1[6], p[6];
  float f[27];
};
__device__ __forceinline__ double lane_of(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __noinline__ int fit_step_coop(const DevGeom& g, float (&pf)[6], float (&Cf)[21], bool last, int L,
                                          float mx, float my, float mz, float& chi2, CoopMem& m) {
  const int lane = threadIdx.x & 31;
  // the lane's element (i, j), i <= j, of a symmetric 6x6 (lanes 0-20)
  const int e = min(lane, 20);
  const int ei = e < 6 ? 0 : e < 11 ? 1 : e < 15 ? 2 : e < 18 ? 3 : e < 20 ? 4 : 5;
  const int ej = e - (ei == 0 ? 0 : ei == 1 ? 5 : ei == 2 ? 9 : ei == 3 ? 12 : ei == 4 ? 14 : 15);
  const int ij = ei * 6 + ej, ji = ej * 6 + ei;
  // state in: one conversion per element
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 6; ++k) m.f[k] = pf[k];
#pragma unroll
    for (int k = 0; k < 21; ++k) m.f[6 + k] = Cf[k];
  }
  __syncwarp();
  {
    const double pe = (double)m.f[min(lane, 5)], ce = (double)m.f[6 + e];
    if (lane < 6) m.p[lane] = pe;
    if (lane < 21) m.C[ij] = m.C[ji] = ce;
  }
  __syncwarp();
  const double x = m.p[0], y = m.p[1], z = m.p[2], kap = m.p[3], phi = m.p[4], th = m.p[5];
  const double R = (double)g.radius[L];
  const double p6[6] = {x, y, z, kap, phi, th};
  const double kb = field_kb<double>(g, p6);
  double sv, cv;
  sincos((lane & 1) ? th : phi, &sv, &cv);
  const double sf = lane_of(sv, 0), cf = lane_of(cv, 0), sth = lane_of(sv, 1), cth = lane_of(cv, 1);
  // path length: the outward crossing of path_length, or that function
  const double h = kb * kap;
  const double ab = (lane & 1) ? fma(y, cf, -x * sf) : fma(x, cf, y * sf);
  const double b = lane_of(ab, 0), a = lane_of(ab, 1);
  const double r0 = sqrt(fma(x, x, y * y));
  const double dR2 = (R - r0) * (R + r0);
  const double A = b * h, B = fma(a, h, 1.0), E = 0.5 * h * h * dR2, den = fma(2.0, B, -E);
  const double D = fma(A, A, E * den);
  const bool outward = E > 0.0 && b > 0.0 && den > 0.0 && A != 0.0 && !(D < 0.0) && h != 0.0;
  const double sq = sqrt(outward ? D : 0.0);
  // quotients: lane 0 tan(psi / 2), lane 1 1/h, lane 2 cot(theta)
  const double qn = lane == 0 ? E : lane == 1 ? 1.0 : cth;
  const double qd = lane == 0 ? fma(b, h, h > 0.0 ? sq : -sq) : lane == 1 ? h : sth;
  const double quo = qn / (outward || lane > 1 ? qd : 1.0);
  const double cot = lane_of(quo, 2);
  double s = 2.0 * atan(lane_of(quo, 0)) * lane_of(quo, 1);
  if (!outward && !path_length<double>(x, y, h, cf, sf, R, s)) return KF_FIT_NO_CROSS;
  // helix functions: lanes 0-3 sc, cc, f1, f2
  const double psi = h * s;
  double sc, cc, f1, f2;
  if (fabs(psi) < 0.5) {
    const int k = lane & 3;
    const double c0 = k == 0 ? 1.0 / 362880.0 : k == 1 ? 1.0 / 3628800.0 : k == 2 ? -1.0 / 3991680.0 : 1.0 / 403200.0;
    const double c1 = k == 0 ? -1.0 / 5040.0 : k == 1 ? -1.0 / 40320.0 : k == 2 ? 1.0 / 45360.0 : -1.0 / 5760.0;
    const double c2 = k == 0 ? 1.0 / 120.0 : k == 1 ? 1.0 / 720.0 : k == 2 ? -1.0 / 840.0 : 1.0 / 144.0;
    const double c3 = k == 0 ? -1.0 / 6.0 : k == 1 ? -1.0 / 24.0 : k == 2 ? 1.0 / 30.0 : -1.0 / 8.0;
    const double c4 = k == 0 ? 1.0 : k == 1 ? 0.5 : k == 2 ? -1.0 / 3.0 : 0.5;
    const double c5 = k == 0   ? -1.0 / 39916800.0
                      : k == 1 ? -1.0 / 479001600.0
                      : k == 2 ? 12.0 / 6227020800.0
                               : -11.0 / 479001600.0;
    const double q = psi * psi;
    const double q5 = q * q * q * q * q, w = k == 1 || k == 2 ? psi : 1.0;
    const double v = fma(w * q5, c5, w * fma(q, fma(q, fma(q, fma(q, c0, c1), c2), c3), c4));
    sc = lane_of(v, 0);
    cc = lane_of(v, 1);
    f1 = lane_of(v, 2);
    f2 = lane_of(v, 3);
  } else {
    helix_fns<double>(psi, sc, cc, f1, f2);
  }
  const double Sx = s * sc, Cx = s * cc;
  const double dx = fma(cf, Sx, -sf * Cx), dy = fma(sf, Sx, cf * Cx);
  const double xn = x + dx, yn = y + dy, zn = fma(s, cot, z);
  const double cpsi = fma(-psi, cc, 1.0), spsi = psi * sc;
  const double cp = fma(cf, cpsi, -sf * spsi), sp = fma(sf, cpsi, cf * spsi);
  const double s2 = s * s, dSdh = s2 * f1, dCdh = s2 * f2;
  const double Fx3 = kb * fma(cf, dSdh, -sf * dCdh), Fy3 = kb * fma(sf, dSdh, cf * dCdh);
  // lane 0: -1 / (dg/ds), lane 1: -s / sin^2(theta)
  const double q2 = (lane & 1 ? -s : -1.0) / (lane & 1 ? sth * sth : fma(xn, cp, yn * sp));
  const double inv = lane_of(q2, 0), J25 = lane_of(q2, 1);
  // ds/d(x, y, q/pT, phi) in lanes 0-3, then J's value entries: lane 4 r + c,
  // rows x, y, z, phi, columns x, y, q/pT, phi
  const int c4 = lane & 3, r4 = (lane >> 2) & 3;
  const double gx = c4 == 0 ? 1.0 : c4 == 1 ? 0.0 : c4 == 2 ? Fx3 : -dy;
  const double gy = c4 == 0 ? 0.0 : c4 == 1 ? 1.0 : c4 == 2 ? Fy3 : dx;
  const double ds = fma(xn, gx, yn * gy) * inv;
  const double coef = r4 == 0 ? cp : r4 == 1 ? sp : r4 == 2 ? cot : h;
  const double base = r4 == 0 ? gx : r4 == 1 ? gy : r4 == 2 ? 0.0 : c4 == 2 ? kb * s : c4 == 3 ? 1.0 : 0.0;
  const double Je = fma(coef, ds, base);
  const int jr = r4 == 3 ? 4 : r4, jc = c4 < 2 ? c4 : c4 + 1;
  if (lane < 16) m.J[jr * 6 + jc] = Je;
  else if (lane < 24) {  // columns z and theta
    const int r = (lane - 16) >> 1, c = (lane & 1) ? 5 : 2;
    m.J[(r == 3 ? 4 : r) * 6 + c] = r == 2 ? (c == 2 ? 1.0 : J25) : 0.0;
  }
  __syncwarp();
  // C <- J C J^T: lanes 0-23 the rows 0, 1, 2, 4 of T = J C, then every
  // element from T and J (rows 3 and 5 of J are unit rows)
  {
    const int r = lane < 24 ? lane / 6 : 0, i = r == 3 ? 4 : r, k = lane < 24 ? lane - 6 * r : 0;
    double t = m.J[i * 6] * m.C[k];
#pragma unroll
    for (int q = 1; q < 6; ++q) t = fma(m.J[i * 6 + q], m.C[q * 6 + k], t);
    if (lane < 24) m.T[i * 6 + k] = t;
  }
  __syncwarp();
  {
    const bool ui = ei == 3 || ei == 5, uj = ej == 3 || ej == 5;
    // T's row, J's row: the order in which transport takes them (2, 0, 1, 4)
    const bool swap = ui || (ej == 2 && ei < 2);
    const int ra = swap ? ej : ei, rb = swap ? ei : ej;
    const int rj = rb == 3 || rb == 5 ? 0 : rb, rt = ui && uj ? 0 : ra;
    double v = m.T[rt * 6] * m.J[rj * 6];
#pragma unroll
    for (int q = 1; q < 6; ++q) v = fma(m.T[rt * 6 + q], m.J[rj * 6 + q], v);
    if (ui && uj) v = m.C[ij];
    else if (ui || uj) v = m.T[ra * 6 + rb];
    __syncwarp();
    if (lane < 21) m.C[ij] = m.C[ji] = v;
  }
  __syncwarp();
  // measurement frame, residual, chi2
  const double ir = 1.0 / sqrt(fma(xn, xn, yn * yn));
  const double cu = xn * ir, su = yn * ir;
  const int i6 = min(lane, 5);
  const double a0 = fma(-su, m.C[i6 * 6], cu * m.C[i6 * 6 + 1]), a1 = m.C[i6 * 6 + 2];
  const double s00 = fma(-su, lane_of(a0, 0), fma(cu, lane_of(a0, 1), (double)g.vr));
  const double s01 = lane_of(a0, 2), s11 = m.C[14] + (double)g.vz;
  const double idet = 1.0 / fma(s00, s11, -s01 * s01);
  const double si00 = s11 * idet, si01 = -s01 * idet, si11 = s00 * idet;
  const double hx = (double)mx, hy = (double)my, hz = (double)mz;
  if (fma(hx, xn, hy * yn) <= 0.0) return KF_FIT_FAR_SIDE;
  const double res0 = fma(-su, hx - xn, cu * (hy - yn)), res1 = hz - zn;
  chi2 += (float)fma(si00 * res0, res0, fma(2.0 * si01 * res0, res1, si11 * res1 * res1));
  // gain and update
  const double k0 = fma(a0, si00, a1 * si01), k1 = fma(a0, si01, a1 * si11);
  const double pq = i6 == 0 ? xn : i6 == 1 ? yn : i6 == 2 ? zn : i6 == 3 ? kap : i6 == 4 ? fma(h, s, phi) : th;
  const double pu = fma(k0, res0, fma(k1, res1, pq));
  if (lane < 6) {
    m.a0[lane] = a0;
    m.k0[lane] = k0;
    m.k1[lane] = k1;
    m.p[lane] = pu;
  }
  __syncwarp();
  double ce = m.C[ij] - fma(m.k0[ei], m.a0[ej], m.k1[ei] * m.C[ej * 6 + 2]);
  double pe = m.p[i6];
  if (!last) {
    const double pp[6] = {m.p[0], m.p[1], m.p[2], m.p[3], m.p[4], m.p[5]};
    const double x0 = x0_at<double>(g, L, pp[2]);
    if (pp[3] != 0.0 && x0 > 0.0) {
      sincos((lane & 1) ? pp[5] : pp[4], &sv, &cv);
      const double sph = lane_of(sv, 0), cph = lane_of(cv, 0), st = lane_of(sv, 1);
      const double cd = fma(cph, pp[0], sph * pp[1]) * rsqrt(fma(pp[0], pp[0], pp[1] * pp[1]));
      const double t = x0 / fabs(st * cd);
      const double w = fabs(pp[3]) * st;
      const double root = sqrt((lane & 1) ? t : fma(MPION * MPION * w, w, 1.0));
      const double tp = 0.0136 * fabs(pp[3]) * lane_of(root, 0) * lane_of(root, 1) * fma(0.038, log(t), 1.0);
      const double tt = tp * st;
      if (lane == 18) ce = fma(tp, tp, ce);  // phi, phi
      if (lane == 20) ce = fma(tt, tt, ce);  // theta, theta
    }
    if (g.eloss[L] > 0.f) {
      __syncwarp();
      if (lane < 21) m.C[ij] = ce;
      __syncwarp();
      double pl[6] = {pp[0], pp[1], pp[2], pp[3], pp[4], pp[5]}, Cl[21];
#pragma unroll
      for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = i; j < 6; ++j) Cl[S6(i, j)] = m.C[i * 6 + j];
      add_eloss_ool<double, false, true>(pl, Cl, (double)g.eloss[L]);
      __syncwarp();
      if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
          for (int j = i; j < 6; ++j) m.C[i * 6 + j] = Cl[S6(i, j)];
        m.p[3] = pl[3];
      }
      __syncwarp();
      ce = m.C[ij];
      pe = m.p[i6];
    }
  }
  // state out
  __syncwarp();
  if (lane < 6) m.f[lane] = (float)pe;
  const float cef = (float)ce;
  if (lane < 21) m.f[6 + lane] = cef;
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 6; ++k) pf[k] = m.f[k];
#pragma unroll
  for (int k = 0; k < 21; ++k) Cf[k] = m.f[6 + k];
  __syncwarp();
  return KF_FIT_OK;
}

// The fit's track order, per window of ORDER_WINDOW consecutive tracks: by
// decreasing hit count (tracks removed as duplicates count 0), so that a
// warp's tracks run about the same number of steps, while the per-track
// reads and writes of a window stay close together in time (they meet in L2).
// The order within a hit count is not fixed; no result depends on it.
constexpr int ORDER_WINDOW = 4096, ORDER_THREADS = 512, ORDER_BINS = 64;

__device__ __forceinline__ int order_key(const FitParams& P, int t) {
  if (P.keep && P.keep_in_main && !P.keep[t]) return 0;
  return min(max(P.n_list[t], 0), ORDER_BINS - 1);
}

// One block per window (the first one also empties the careful pass's lists):
// counts per hit count, an exclusive prefix over the
// counts from the longest down, then each track's position (one shared-memory
// atomic per hit count and warp).
__global__ void __launch_bounds__(ORDER_THREADS) k_fit_order(const FitParams P) {
  static_assert(ORDER_BINS == 64, "two bins per lane");
  __shared__ unsigned cnt[ORDER_BINS], cur[ORDER_BINS];
  if (blockIdx.x == 0 && threadIdx.x == 0) *P.careful_count = *P.dbl_count = 0u;
  const int w0 = blockIdx.x * ORDER_WINDOW;
  const int w1 = min(P.ns, w0 + ORDER_WINDOW);
  for (int b = threadIdx.x; b < ORDER_BINS; b += blockDim.x) cnt[b] = 0u;
  __syncthreads();
  for (int t = w0 + threadIdx.x; t < w1; t += blockDim.x) atomicAdd(&cnt[order_key(P, t)], 1u);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {  // lane j: bins 63 - 2j and 62 - 2j
    const unsigned a = cnt[63 - 2 * lane], b = cnt[62 - 2 * lane];
    unsigned incl = a + b;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    cur[63 - 2 * lane] = incl - a - b;
    cur[62 - 2 * lane] = incl - b;
  }
  __syncthreads();
  for (int r = 0; r < ORDER_WINDOW; r += ORDER_THREADS) {
    const int t = w0 + r + threadIdx.x;
    const int key = t < w1 ? order_key(P, t) : ORDER_BINS;  // ORDER_BINS: no track
    const unsigned same = __match_any_sync(0xffffffffu, key);
    if (key < ORDER_BINS) {
      const int leader = __ffs(same) - 1;
      unsigned pos = 0;
      if (lane == leader) pos = atomicAdd(&cur[key], (unsigned)__popc(same));
      pos = __shfl_sync(same, pos, leader) + __popc(same & ((1u << lane) - 1u));
      P.order[w0 + pos] = t;
    }
  }
}

// A track the FP32 pass leaves to the careful pass at step k: the state before
// that step, the chi2 so far and k wait in the track's own output places.
__device__ __forceinline__ void leave_to_careful(const FitParams& P, int i, int t, int k, const float (&p)[6],
                                                 const float (&C)[21], float chi2) {
#pragma unroll
  for (int q = 0; q < 6; ++q) P.fit_p[(size_t)q * P.ns + t] = p[q];
#pragma unroll
  for (int q = 0; q < 21; ++q) P.fit_C[(size_t)q * P.ns + t] = C[q];
  P.fit_chi2[t] = chi2;
  P.fit_status[t] = k;
  P.careful_list[atomicAdd(P.careful_count, 1u)] = i;
  if (P.careful_flag) P.careful_flag[t] = (unsigned char)min(k + 1, 255);
}

// Track at position i of the fit's order; checkpoints go to column i.
// Returns, in the careful pass, whether a crossing of the track has
// cos(alpha) < ADJOINT_CAREFUL_COS (its adjoint then needs double steps).
// DISK: the detector has endcap disks (hits on surfaces >= n_layers take the
// plane step; they carry no alignment).
// coop (careful pass): the whole warp works on this track; lane 0 writes.
template <bool CAREFUL, bool DISK>
__device__ __forceinline__ bool fit_track(const FitParams& P, int i, int t, CoopMem* coop = nullptr) {
  const bool writes = !CAREFUL || !coop || (threadIdx.x & 31) == 0;
  if (!CAREFUL && P.careful_flag) P.careful_flag[t] = 0;  // set below if the track is left to the careful pass
  // removed as a duplicate: zero outputs (the careful pass reads the final
  // flags; the main pass only when they are written before it)
  if (P.keep && (CAREFUL || P.keep_in_main) && !P.keep[t]) {
    if (!writes) return false;
#pragma unroll
    for (int k = 0; k < 6; ++k) P.fit_p[(size_t)k * P.ns + t] = 0.f;
#pragma unroll
    for (int k = 0; k < 21; ++k) P.fit_C[(size_t)k * P.ns + t] = 0.f;
    P.fit_chi2[t] = 0.f;
    P.fit_status[t] = KF_FIT_SKIPPED;
    return false;
  }
  const DevGeom& g = P.g;
  // the prior, or (careful pass) the state the FP32 pass stopped at before step k0
  const float* const p0 = CAREFUL ? P.fit_p : P.sp;
  const float* const C0 = CAREFUL ? P.fit_C : P.sc;
  float p[6], C[21];
#pragma unroll
  for (int k = 0; k < 6; ++k) p[k] = p0[(size_t)k * P.ns + t];
#pragma unroll
  for (int k = 0; k < 21; ++k) C[k] = C0[(size_t)k * P.ns + t];
  const int k0 = CAREFUL ? P.fit_status[t] : 0;
  // a loose prior: the careful pass runs the first steps in double (a track
  // left at a later step had no loose prior)
  const bool loose = k0 == 0 && loose_prior(C, g);
  if (!CAREFUL && loose) {
    leave_to_careful(P, i, t, 0, p, C, 0.f);
    return false;
  }
  const int hoff = P.hit_off[P.seed_event[t]];
  const int n = P.n_list[t];
  const int* lst = P.lists + (size_t)t * P.max_len;
  float chi2 = CAREFUL ? P.fit_chi2[t] : 0.f;
  int status = KF_FIT_OK;
  bool adj_dbl = false;
#pragma unroll 1
  for (int k = k0; k < n && status == KF_FIT_OK; ++k) {
    if (P.ckpt && writes && k % P.ckpt_stride == 0 && k / P.ckpt_stride < P.ckpt_slices) {  // state before hit k
      float* c = P.ckpt + (size_t)(k / P.ckpt_stride) * 27 * P.ns + i;
#pragma unroll
      for (int q = 0; q < 6; ++q) c[(size_t)q * P.ns] = p[q];
#pragma unroll
      for (int q = 0; q < 21; ++q) c[(size_t)(6 + q) * P.ns] = C[q];
    }
    const int hi = hoff + lst[k];
    const int L = P.hlayer[hi];
    const bool disk = DISK && is_disk(g, L);
    float mx, my, mz;
    if (disk) {
      mx = P.hx[hi];
      my = P.hy[hi];
      mz = P.hz[hi];
    } else {
      corrected_hit(P.align[L], P.hx[hi], P.hy[hi], P.hz[hi], mx, my, mz);
    }
    if (!CAREFUL && disk) {
      if (k > 0 && plane_careful(g, p, plane_z(g, L))) {  // a long arc onto the disk: the careful pass
        leave_to_careful(P, i, t, k, p, C, chi2);
        return false;
      }
      status = disk_step<float>(g, p, C, k == 0, k + 1 == n, L, mx, my, chi2);
    } else if (!CAREFUL) {
      if (k > 0) {
        float q[6], J[6][6], cosa = 1.f;
        if (prop_jacobian<float, true>(p, g.radius[L], field_kb<float>(g, p), INFINITY, q, J, &cosa) != 1) {
          status = KF_FIT_NO_CROSS;
          break;
        }
        if (cosa < CAREFUL_COS) {
          leave_to_careful(P, i, t, k, p, C, chi2);
          return false;
        }
        transport<float>(J, C);
#pragma unroll
        for (int q_ = 0; q_ < 6; ++q_) p[q_] = q[q_];
      }
      Frame f;
      make_frame<float>(p, C, g.vr, g.vz, f);
      float r0, r1;
      if (!residual<float>(p, f, mx, my, mz, r0, r1)) { status = KF_FIT_FAR_SIDE; break; }
      chi2 += chi2_of<float>(f, r0, r1);
      kf_update<float>(p, C, f, r0, r1);
      if (k + 1 < n) {
        add_ms<float, true>(p, C, x0_at<float>(g, L, p[2]));
        add_eloss_ool<float, false, true>(p, C, g.eloss[L]);
      }
    } else {
      bool careful = false;
      if (k > 0 && !disk) {
        float zc, cosa;
        if (!crossing(p, g.radius[L], field_kb<float>(g, p), zc, cosa)) { status = KF_FIT_NO_CROSS; break; }
        careful = cosa < CAREFUL_COS;
        adj_dbl = adj_dbl || cosa < ADJOINT_CAREFUL_COS;
      } else if (k > 0) {  // a long arc onto a disk: in double here and in the adjoint
        careful = plane_careful(g, p, plane_z(g, L));
        adj_dbl = adj_dbl || careful;
      }
      if (loose && k < LOOSE_STEPS) careful = true;  // the first steps against a loose prior
      if (coop && careful && k > 0 && !disk)
        status = fit_step_coop(g, p, C, k + 1 == n, L, mx, my, mz, chi2, *coop);
      else
        status = careful ? fit_step<double, DISK>(g, p, C, k == 0, k + 1 == n, L, mx, my, mz, chi2)
                         : fit_step<float, DISK>(g, p, C, k == 0, k + 1 == n, L, mx, my, mz, chi2);
    }
  }
  if (CAREFUL && coop) __syncwarp();  // every lane has read the track's places
  if (!writes) return adj_dbl;
#pragma unroll
  for (int k = 0; k < 6; ++k) P.fit_p[(size_t)k * P.ns + t] = p[k];
#pragma unroll
  for (int k = 0; k < 21; ++k) P.fit_C[(size_t)k * P.ns + t] = C[k];
  P.fit_chi2[t] = chi2;
  P.fit_status[t] = status;
  return adj_dbl;
}

template <bool DISK>
__global__ void __launch_bounds__(FIT_THREADS) k_fit(const FitParams P) {
  const int i = blockIdx.x * FIT_THREADS + threadIdx.x;
  if (i < P.ns) fit_track<false, DISK>(P, i, P.order[i]);
}

// Second pass over the flagged tracks, one warp per block.  Its double steps
// are bound by the SM's FP64 rate (about 2 FMA per clock and SM, whatever the
// number of active lanes) and by the divergence of a warp's tracks, so the
// list is dealt evenly to the blocks: with fewer tracks than blocks, one track
// per warp.  Taken on from the FP32 pass's last state (one to three steps a
// track instead of all of them), the fit of 180,000 tracks of 30 events
// (loads included) went from 551 to 426 us, that of one 2,500-track event
// with its finding from 825 to 716 us.  A track whose adjoint needs double steps gets CAREFUL_DBL_BIT in
// its entry and is listed in dbl_list.
template <bool DISK>
__global__ void __launch_bounds__(32) k_fit_careful(const FitParams P) {
  const unsigned n = *P.careful_count;
  const unsigned spread = min(gridDim.x, (unsigned)P.careful_spread);
  const unsigned per = min(32u, (n + spread - 1) / spread);  // tracks per warp and round
  __shared__ CoopMem mem;
  const bool whole = per == 1;  // the whole warp on one track
  if (!whole && threadIdx.x >= per) return;
#pragma unroll 1
  for (unsigned j = blockIdx.x * per + (whole ? 0u : threadIdx.x); j < n; j += gridDim.x * per) {
    const unsigned v = (unsigned)P.careful_list[j];
    const int pos = (int)(v & ~CAREFUL_DBL_BIT);
    const bool dbl = fit_track<true, DISK>(P, pos, P.order[pos], whole ? &mem : nullptr);
    if (whole && threadIdx.x != 0) continue;
    P.careful_list[j] = (int)(dbl ? (v | CAREFUL_DBL_BIT) : (v & ~CAREFUL_DBL_BIT));
    if (dbl) P.dbl_list[atomicAdd(P.dbl_count, 1u)] = pos;  // packed, so that few blocks hold them
  }
}

__global__ void __launch_bounds__(256) k_fit_unkept(const FitParams P) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= P.ns || P.keep[t]) return;
#pragma unroll
  for (int k = 0; k < 6; ++k) P.fit_p[(size_t)k * P.ns + t] = 0.f;
#pragma unroll
  for (int k = 0; k < 21; ++k) P.fit_C[(size_t)k * P.ns + t] = 0.f;
  P.fit_chi2[t] = 0.f;
  P.fit_status[t] = KF_FIT_SKIPPED;
}

}  // namespace

cudaError_t launch_fit_unkept(const FitParams& P, cudaStream_t st) {
  if (P.ns <= 0 || !P.keep) return cudaSuccess;
  k_fit_unkept<<<(P.ns + 255) / 256, 256, 0, st>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_fit_main(const FitParams& P, cudaStream_t st) {
  if (P.ns <= 0) return cudaSuccess;
  k_fit_order<<<(P.ns + ORDER_WINDOW - 1) / ORDER_WINDOW, ORDER_THREADS, 0, st>>>(P);
  const int blocks = (P.ns + FIT_THREADS - 1) / FIT_THREADS;
  if (P.g.n_disks > 0) k_fit<true><<<blocks, FIT_THREADS, 0, st>>>(P);
  else k_fit<false><<<blocks, FIT_THREADS, 0, st>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_fit_careful(const FitParams& P, cudaStream_t st) {
  if (P.ns <= 0) return cudaSuccess;
  FitParams Q = P;
  Q.careful_spread = 2 * P.num_sms;
  const int blocks = careful_blocks(P.ns, 32, Q.careful_spread, P.num_sms);
  if (P.g.n_disks > 0) k_fit_careful<true><<<blocks, 32, 0, st>>>(Q);
  else k_fit_careful<false><<<blocks, 32, 0, st>>>(Q);
  return cudaGetLastError();
}

cudaError_t launch_fit(const FitParams& P, cudaStream_t st) {
  cudaError_t e = launch_fit_main(P, st);
  if (e == cudaSuccess) e = launch_fit_careful(P, st);
  return e;
}

}  // namespace kfg
