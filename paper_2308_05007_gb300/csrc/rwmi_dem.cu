// rwmi_dem.cu -- free DEM of the metaball particles (Section 2.2, Eqs. 4-11): sphero-metaball
// contact geometry, linear spring-dashpot normal force, the Eq. 5 tangential spring with its
// Coulomb limit, and the Eq. 4 integration.
//
// This translation unit is built without FMA contraction (-fmad=false) and takes IEEE division
// and square roots, so every binary64 operation rounds exactly as written. With the fluid force
// switched off the trajectories then follow the CPU oracle's bit for bit, which the GPU tests
// check; the formulas and their readings are the oracle's.
//
// For up to 128 particles every DEM step of an LBM step is one launch of one thread-block cluster
// (dem_cluster_kernel, cluster barriers between the two phases); beyond that a DEM step is two
// launches:
//   dem_contacts_kernel   one thread per pair slot (i < j) and per wall slot (particle, face):
//                         reach test, Newton-Raphson geometry, force law; writes the slot's
//                         force and torques (zero when apart) and its spring and Newton point;
//   dem_integrate_kernel  one thread per particle: sums its slots in a fixed order (pairs by
//                         partner index, then faces), adds the fluid force and gravity, advances
//                         velocity, origin, spin and orientation.
// The launches follow each other on one stream.
#include "rwmi_internal.cuh"

namespace rwmi {
namespace {

constexpr int NEWTON_NEW = 24;        // Newton iterations (at most) from the deterministic start
constexpr int NEWTON_CONT = 6;        // ... from the previous DEM step's point (pair within reach then)
constexpr int SURFACE_ITERS = 24;     // bracketed Newton iterations for Eq. 8's q
constexpr int SURFACE_HALVINGS = 16;  // halvings of the first-order q looking for an inside point

__device__ void quat_matrix(const double* q, double R[3][3]) {
  const double w = q[0], x = q[1], y = q[2], z = q[3];
  R[0][0] = 1.0 - 2.0 * (y * y + z * z);
  R[0][1] = 2.0 * (x * y - w * z);
  R[0][2] = 2.0 * (x * z + w * y);
  R[1][0] = 2.0 * (x * y + w * z);
  R[1][1] = 1.0 - 2.0 * (x * x + z * z);
  R[1][2] = 2.0 * (y * z - w * x);
  R[2][0] = 2.0 * (x * z - w * y);
  R[2][1] = 2.0 * (y * z + w * x);
  R[2][2] = 1.0 - 2.0 * (x * x + y * y);
}

// Internal (zoomed) control points of particle p about origin org: positions and weights
__device__ int internal_points(const DemArgs& a, int p, const double org[3], double* cw, double* kw) {
  double R[3][3];
  quat_matrix(a.st + 13 * p + 3, R);
  const double s = a.zoom[p];
  const ParticleDesc& d = a.desc[p];
  int n = 0;
  for (int i = d.c0; i < d.c1 && n < DEM_MAX_CP; ++i, ++n) {
    const float4 cb = a.cbody[i];
    const double b[3] = {s * (double)cb.x, s * (double)cb.y, s * (double)cb.z};
    for (int e = 0; e < 3; ++e) cw[3 * n + e] = org[e] + R[e][0] * b[0] + R[e][1] * b[1] + R[e][2] * b[2];
    kw[n] = s * s * (double)cb.w;
  }
  return n;
}

// Eq. 3 with gradient and Hessian (xx yy zz xy xz yz) at x
__device__ double mb_eval(const double* cw, const double* kw, int n, const double x[3], double g[3], double H[6]) {
  double f = 0.0;
  for (int e = 0; e < 3; ++e) g[e] = 0.0;
  for (int m = 0; m < 6; ++m) H[m] = 0.0;
  for (int i = 0; i < n; ++i) {
    const double r[3] = {x[0] - cw[3 * i], x[1] - cw[3 * i + 1], x[2] - cw[3 * i + 2]};
    const double r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
    const double inv2 = 1.0 / r2, k = kw[i];
    const double fi = k * inv2;
    f += fi;
    const double c1 = -2.0 * fi * inv2;
    const double c2 = 8.0 * fi * inv2 * inv2;
    for (int e = 0; e < 3; ++e) g[e] += c1 * r[e];
    H[0] += c1 + c2 * r[0] * r[0];
    H[1] += c1 + c2 * r[1] * r[1];
    H[2] += c1 + c2 * r[2] * r[2];
    H[3] += c2 * r[0] * r[1];
    H[4] += c2 * r[0] * r[2];
    H[5] += c2 * r[1] * r[2];
  }
  return f;
}

__device__ bool solve3(const double A[3][3], const double b[3], double d[3]) {
  const double det = A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1])
                   - A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0])
                   + A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]);
  if (!(fabs(det) > 1e-300)) return false;
  d[0] = (b[0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) - A[0][1] * (b[1] * A[2][2] - A[1][2] * b[2])
          + A[0][2] * (b[1] * A[2][1] - A[1][1] * b[2])) / det;
  d[1] = (A[0][0] * (b[1] * A[2][2] - A[1][2] * b[2]) - b[0] * (A[1][0] * A[2][2] - A[1][2] * A[2][0])
          + A[0][2] * (A[1][0] * b[2] - b[1] * A[2][0])) / det;
  d[2] = (A[0][0] * (A[1][1] * b[2] - b[1] * A[2][1]) - A[0][1] * (A[1][0] * b[2] - b[1] * A[2][0])
          + b[0] * (A[1][0] * A[2][1] - A[1][1] * A[2][0])) / det;
  return true;
}

// Newton step, at most one lattice unit long; false when singular or converged (step < 1e-12)
__device__ bool newton_update(const double A[3][3], const double G[3], double x[3]) {
  const double b[3] = {-G[0], -G[1], -G[2]};
  double d[3];
  if (!solve3(A, b, d)) return false;
  const double len = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  const double sc = len > 1.0 ? 1.0 / len : 1.0;
  for (int e = 0; e < 3; ++e) x[e] += sc * d[e];
  return len > 1e-12;
}

// Eq. 8: x_c = x_m + q grad f(x_m) with f(x_c) = 1, the crossing nearest to x_m (first-order
// Taylor q, bracket by halving to an inside point, bracketed Newton in q)
__device__ void surface_along(const double* c, const double* k, int n, const double xm[3], double xc[3]) {
  double g[3], gx[3], H[6], x[3];
  const double f = mb_eval(c, k, n, xm, g, H);
  const double q1 = (1.0 - f) / (g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
  double lo = 0.0, hi = q1, q = q1;
  bool inside = false;
  for (int h = 0; h <= SURFACE_HALVINGS; ++h) {
    for (int e = 0; e < 3; ++e) x[e] = xm[e] + hi * g[e];
    if (mb_eval(c, k, n, x, gx, H) >= 1.0) { inside = true; break; }
    hi = 0.5 * hi;
  }
  if (inside) {
    q = hi;
    for (int it = 0; it < SURFACE_ITERS; ++it) {
      for (int e = 0; e < 3; ++e) x[e] = xm[e] + q * g[e];
      const double fx = mb_eval(c, k, n, x, gx, H);
      if (fx == 1.0) break;
      if (fx > 1.0) hi = q; else lo = q;
      const double dq = gx[0] * g[0] + gx[1] * g[1] + gx[2] * g[2];
      double qn = fabs(dq) > 1e-300 ? q - (fx - 1.0) / dq : 0.5 * (lo + hi);
      if (!(qn > lo && qn < hi)) qn = 0.5 * (lo + hi);
      if (qn == q) break;
      q = qn;
    }
  }
  for (int e = 0; e < 3; ++e) xc[e] = xm[e] + q * g[e];
}

// Eqs. 7-9 for one pair; xm: start (cont) and result. Returns delta; writes n (0 -> 1), x_cp.
__device__ double pair_geom(const double* c0, const double* k0, int n0, const double* c1, const double* k1, int n1,
                            double Rs0, double Rs1, bool cont, double xm[3], double nrm[3], double xcp[3]) {
  if (!cont) {
    int ba = 0, bb = 0;
    double best = INFINITY;
    for (int a = 0; a < n0; ++a)
      for (int b = 0; b < n1; ++b) {
        const double d[3] = {c1[3 * b] - c0[3 * a], c1[3 * b + 1] - c0[3 * a + 1], c1[3 * b + 2] - c0[3 * a + 2]};
        const double gap = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]) - sqrt(k0[a]) - sqrt(k1[b]);
        if (gap < best) { best = gap; ba = a; bb = b; }
      }
    const double ra = sqrt(k0[ba]), rb = sqrt(k1[bb]), w = ra / (ra + rb);
    for (int e = 0; e < 3; ++e) xm[e] = c0[3 * ba + e] + w * (c1[3 * bb + e] - c0[3 * ba + e]);
  }
  const int iters = cont ? NEWTON_CONT : NEWTON_NEW;
  for (int it = 0; it < iters; ++it) {
    double g0[3], g1[3], H0[6], H1[6];
    mb_eval(c0, k0, n0, xm, g0, H0);
    mb_eval(c1, k1, n1, xm, g1, H1);
    const double G[3] = {g0[0] + g1[0], g0[1] + g1[1], g0[2] + g1[2]};
    const double A[3][3] = {{H0[0] + H1[0], H0[3] + H1[3], H0[4] + H1[4]},
                            {H0[3] + H1[3], H0[1] + H1[1], H0[5] + H1[5]},
                            {H0[4] + H1[4], H0[5] + H1[5], H0[2] + H1[2]}};
    if (!newton_update(A, G, xm)) break;
  }
  double xc0[3], xc1[3];
  surface_along(c0, k0, n0, xm, xc0);
  surface_along(c1, k1, n1, xm, xc1);
  const double d[3] = {xc1[0] - xc0[0], xc1[1] - xc0[1], xc1[2] - xc0[2]};
  const double dist = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  const double delta = Rs0 + Rs1 - dist;
  for (int e = 0; e < 3; ++e) nrm[e] = dist > 0.0 ? d[e] / dist : 0.0;
  for (int e = 0; e < 3; ++e) xcp[e] = xc0[e] + (Rs0 - 0.5 * delta) * nrm[e];
  return delta;
}

// Eqs. 10-11 for the face `side` of walled axis ax at 0 or L; n into the box
__device__ double wall_geom(const double* c, const double* k, int n, int ax, int side, double L, double Rs, bool cont,
                            double xm[3], double nrm[3], double xcp[3]) {
  const double sg = side ? -1.0 : 1.0;
  if (!cont) {
    int bi = 0;
    double best = INFINITY;
    for (int i = 0; i < n; ++i) {
      const double reach = side ? -(c[3 * i + ax] + sqrt(k[i])) : c[3 * i + ax] - sqrt(k[i]);
      if (reach < best) { best = reach; bi = i; }
    }
    for (int e = 0; e < 3; ++e) xm[e] = c[3 * bi + e];
    xm[ax] -= sg * sqrt(k[bi]);
  }
  int b = (ax + 1) % 3, cc = (ax + 2) % 3;
  if (b > cc) { const int t = b; b = cc; cc = t; }
  const int iters = cont ? NEWTON_CONT : NEWTON_NEW;
  for (int it = 0; it < iters; ++it) {
    double g[3], H6[6];
    const double f = mb_eval(c, k, n, xm, g, H6);
    const double H[3][3] = {{H6[0], H6[3], H6[4]}, {H6[3], H6[1], H6[5]}, {H6[4], H6[5], H6[2]}};
    const double G[3] = {g[b], g[cc], f - 1.0};
    const double A[3][3] = {{H[b][0], H[b][1], H[b][2]}, {H[cc][0], H[cc][1], H[cc][2]}, {g[0], g[1], g[2]}};
    if (!newton_update(A, G, xm)) break;
  }
  double xcw[3];
  for (int e = 0; e < 3; ++e) { xcw[e] = xm[e]; nrm[e] = 0.0; }
  xcw[ax] = side ? L : 0.0;
  nrm[ax] = sg;
  const double dist = (xm[ax] - xcw[ax]) * sg;
  const double delta = Rs - dist;
  for (int e = 0; e < 3; ++e) xcp[e] = xcw[e] + 0.5 * delta * nrm[e];
  return delta;
}

__device__ void point_velocity(const DemArgs& a, int p, const double org[3], const double x[3], double v[3]) {
  const double* st = a.st + 13 * p;
  const double r[3] = {x[0] - org[0], x[1] - org[1], x[2] - org[2]};
  const double* w = st + 10;
  v[0] = st[7] + (w[1] * r[2] - w[2] * r[1]);
  v[1] = st[8] + (w[2] * r[0] - w[0] * r[2]);
  v[2] = st[9] + (w[0] * r[1] - w[1] * r[0]);
}

// Normal spring-dashpot and Eq. 5 on body i; n from i towards the other body
__device__ void contact_force(const DemArgs& a, double delta, const double n[3], const double vi[3],
                              const double vj[3], double* xi, double F[3]) {
  const double vr[3] = {vj[0] - vi[0], vj[1] - vi[1], vj[2] - vi[2]};
  const double vn = vr[0] * n[0] + vr[1] * n[1] + vr[2] * n[2];
  double Fn = a.kn * delta - a.etan * vn;
  if (Fn < 0.0) Fn = 0.0;
  const double vt[3] = {vr[0] - vn * n[0], vr[1] - vn * n[1], vr[2] - vn * n[2]};
  const double xn = xi[0] * n[0] + xi[1] * n[1] + xi[2] * n[2];
  for (int e = 0; e < 3; ++e) xi[e] = (xi[e] - xn * n[e]) + vt[e] * a.dt;
  double Ft[3];
  for (int e = 0; e < 3; ++e) Ft[e] = a.kt * xi[e] + a.etat * vt[e];
  const double mag = sqrt(Ft[0] * Ft[0] + Ft[1] * Ft[1] + Ft[2] * Ft[2]);
  const double lim = a.mus * Fn;
  if (mag > lim) {
    const double sc = lim / mag;
    for (int e = 0; e < 3; ++e) {
      Ft[e] = Ft[e] * sc;
      xi[e] = a.kt > 0.0 ? (Ft[e] - a.etat * vt[e]) / a.kt : 0.0;
    }
  }
  for (int e = 0; e < 3; ++e) F[e] = Ft[e] - Fn * n[e];
}

__device__ void cross3(const double u[3], const double v[3], double w[3]) {
  w[0] = u[1] * v[2] - u[2] * v[1];
  w[1] = u[2] * v[0] - u[0] * v[2];
  w[2] = u[0] * v[1] - u[1] * v[0];
}

__device__ void clear3(double* v) { v[0] = v[1] = v[2] = 0.0; }

// One pair slot (i < j)
__device__ void pair_slot(const DemArgs& a, int i, int j) {
  const size_t pr = (size_t)i * a.P + j;
  double* F = a.pF + 3 * pr;
  double* Ti = a.pTi + 3 * pr;
  double* Tj = a.pTj + 3 * pr;
  double* xi = a.xi + 3 * pr;
  {   // binary32 reach prefilter: bound spheres apart by more than a margin cannot touch
    const float4 pi = a.posf[i], pj = a.posf[j];
    const float dv[3] = {pj.x - pi.x, pj.y - pi.y, pj.z - pi.z};
    float d2 = 0.0f;
    for (int e = 0; e < 3; ++e) {
      float dd = dv[e];
      if (!a.wall[e]) dd -= (float)a.n[e] * rintf(dd / (float)a.n[e]);
      d2 += dd * dd;
    }
    const float reach = pi.w + pj.w + 0.01f;
    if (d2 > reach * reach) {   // the slot's forces are read only while in contact
      if (a.act[pr]) { a.act[pr] = 0; clear3(xi); }
      return;
    }
  }
  clear3(F); clear3(Ti); clear3(Tj);
  const double* si = a.st + 13 * i;
  const double* sj = a.st + 13 * j;
  double oj[3];
  for (int e = 0; e < 3; ++e) {   // minimum image of j's origin seen from i's
    double d = sj[e] - si[e];
    if (!a.wall[e]) d -= (double)a.n[e] * floor(d / (double)a.n[e] + 0.5);
    oj[e] = si[e] + d;
  }
  const double d[3] = {oj[0] - si[0], oj[1] - si[1], oj[2] - si[2]};
  const double reach = (double)a.desc[i].rb + (double)a.desc[j].rb;
  if (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] >= reach * reach) {
    a.act[pr] = 0;
    clear3(xi);
    return;
  }
  double c0[3 * DEM_MAX_CP], k0[DEM_MAX_CP], c1[3 * DEM_MAX_CP], k1[DEM_MAX_CP];
  const int n0 = internal_points(a, i, si, c0, k0);
  const int n1 = internal_points(a, j, oj, c1, k1);
  double nrm[3], xcp[3];
  double xm[3] = {a.xm[3 * pr], a.xm[3 * pr + 1], a.xm[3 * pr + 2]};
  const double delta = pair_geom(c0, k0, n0, c1, k1, n1, a.Rs[i], a.Rs[j], a.act[pr] != 0, xm, nrm, xcp);
  for (int e = 0; e < 3; ++e) a.xm[3 * pr + e] = xm[e];
  if (!(delta > 0.0)) {
    a.act[pr] = 0;
    clear3(xi);
    return;
  }
  a.act[pr] = 1;
  double vi[3], vj[3];
  point_velocity(a, i, si, xcp, vi);
  point_velocity(a, j, oj, xcp, vj);
  contact_force(a, delta, nrm, vi, vj, xi, F);
  const double ri[3] = {xcp[0] - si[0], xcp[1] - si[1], xcp[2] - si[2]};
  const double rj[3] = {xcp[0] - oj[0], xcp[1] - oj[1], xcp[2] - oj[2]};
  const double Fj[3] = {-F[0], -F[1], -F[2]};
  cross3(ri, F, Ti);
  cross3(rj, Fj, Tj);
}

// One wall slot: particle p, face f = 2 axis + side
__device__ void wall_slot(const DemArgs& a, int p, int f) {
  const size_t wi = 6 * (size_t)p + f;
  const int ax = f >> 1, side = f & 1;
  double* F = a.wF + 3 * wi;
  double* T = a.wT + 3 * wi;
  double* xi = a.xiw + 3 * wi;
  {   // binary32 reach prefilter
    const float4 pf = a.posf[p];
    const float c = ax == 0 ? pf.x : ax == 1 ? pf.y : pf.z;
    const float gapf = side ? (float)a.n[ax] - c : c;
    if (!a.wall[ax] || gapf > pf.w + 0.01f) {
      if (a.actw[wi]) { a.actw[wi] = 0; clear3(xi); }
      return;
    }
  }
  clear3(F); clear3(T);
  const double* sp = a.st + 13 * p;
  const double L = (double)a.n[ax];
  const double gap = side ? L - sp[ax] : sp[ax];
  if (!a.wall[ax] || gap >= (double)a.desc[p].rb) {
    a.actw[wi] = 0;
    clear3(xi);
    return;
  }
  double c[3 * DEM_MAX_CP], k[DEM_MAX_CP];
  const int n = internal_points(a, p, sp, c, k);
  double nrm[3], xcp[3];
  double xm[3] = {a.xmw[3 * wi], a.xmw[3 * wi + 1], a.xmw[3 * wi + 2]};
  const double delta = wall_geom(c, k, n, ax, side, L, a.Rs[p], a.actw[wi] != 0, xm, nrm, xcp);
  for (int e = 0; e < 3; ++e) a.xmw[3 * wi + e] = xm[e];
  if (!(delta > 0.0)) {
    a.actw[wi] = 0;
    clear3(xi);
    return;
  }
  a.actw[wi] = 1;
  double vi[3];
  const double vw[3] = {0.0, 0.0, 0.0};
  point_velocity(a, p, sp, xcp, vi);
  const double nw[3] = {-nrm[0], -nrm[1], -nrm[2]};
  contact_force(a, delta, nw, vi, vw, xi, F);
  const double r[3] = {xcp[0] - sp[0], xcp[1] - sp[1], xcp[2] - sp[2]};
  cross3(r, F, T);
}

__global__ void __launch_bounds__(64) dem_contacts_kernel(DemArgs a, int npairs) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < npairs) {
    int i = 0, rem = k;   // slot k -> pair (i, j), rows of P - 1 - i entries
    while (rem >= a.P - 1 - i) { rem -= a.P - 1 - i; ++i; }
    pair_slot(a, i, i + 1 + rem);
  } else if (k < npairs + 6 * a.P) {
    const int w = k - npairs;
    wall_slot(a, w / 6, w % 6);
  }
}

__device__ void integrate_particle(const DemArgs& a, int p);

__global__ void dem_integrate_kernel(DemArgs a) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < a.P) integrate_particle(a, p);
}

// Force and torque of pair slot (p, j) added to particle p's sums.
__device__ __forceinline__ void add_pair(const DemArgs& a, int p, int j, double F[3], double T[3]) {
  if (j < p) {
    const size_t pr = (size_t)j * a.P + p;
    for (int e = 0; e < 3; ++e) { F[e] = F[e] - a.pF[3 * pr + e]; T[e] = T[e] + a.pTj[3 * pr + e]; }
  } else {
    const size_t pr = (size_t)p * a.P + j;
    for (int e = 0; e < 3; ++e) { F[e] = F[e] + a.pF[3 * pr + e]; T[e] = T[e] + a.pTi[3 * pr + e]; }
  }
}

// Particle p by one DEM step from the sums F, T of its pair slots in contact.
__device__ void advance_particle(const DemArgs& a, int p, double F[3], double T[3]) {
  for (int f = 0; f < 6; ++f)
    if (a.actw[6 * (size_t)p + f])
      for (int e = 0; e < 3; ++e) {
        F[e] = F[e] + a.wF[3 * (6 * (size_t)p + f) + e];
        T[e] = T[e] + a.wT[3 * (6 * (size_t)p + f) + e];
      }
  const double m = a.mass[p];
  for (int e = 0; e < 3; ++e) {
    if (a.Fe) { F[e] = F[e] + a.Fe[6 * p + e]; T[e] = T[e] + a.Fe[6 * p + 3 + e]; }
    F[e] = F[e] + m * a.g[e];
  }
  double* st = a.st + 13 * p;
  const double dt = a.dt;
  for (int e = 0; e < 3; ++e) {   // translation: symplectic Euler
    st[7 + e] = st[7 + e] + dt * (F[e] / m);
    st[e] = st[e] + dt * st[7 + e];
  }
  double R[3][3];   // rotation: I_w = R I_b R^T, w += dt I_w^-1 (T - w x I_w w)
  quat_matrix(st + 3, R);
  const double* I6 = a.Ib + 6 * p;
  const double Ib[3][3] = {{I6[0], I6[3], I6[4]}, {I6[3], I6[1], I6[5]}, {I6[4], I6[5], I6[2]}};
  double RI[3][3], Iw[3][3];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) RI[r][c] = R[r][0] * Ib[0][c] + R[r][1] * Ib[1][c] + R[r][2] * Ib[2][c];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) Iw[r][c] = RI[r][0] * R[c][0] + RI[r][1] * R[c][1] + RI[r][2] * R[c][2];
  double* w = st + 10;
  const double Lw[3] = {Iw[0][0] * w[0] + Iw[0][1] * w[1] + Iw[0][2] * w[2],
                        Iw[1][0] * w[0] + Iw[1][1] * w[1] + Iw[1][2] * w[2],
                        Iw[2][0] * w[0] + Iw[2][1] * w[1] + Iw[2][2] * w[2]};
  double gyro[3], dw[3];
  cross3(w, Lw, gyro);
  const double rhs[3] = {T[0] - gyro[0], T[1] - gyro[1], T[2] - gyro[2]};
  if (solve3(Iw, rhs, dw))
    for (int e = 0; e < 3; ++e) w[e] = w[e] + dt * dw[e];
  double* q = st + 3;   // orientation: q += dt/2 (0, w) q, normalised
  const double qw = q[0], qv[3] = {q[1], q[2], q[3]};
  double wxq[3];
  cross3(w, qv, wxq);
  const double h = 0.5 * dt;
  const double nq[4] = {qw - h * (w[0] * qv[0] + w[1] * qv[1] + w[2] * qv[2]),
                        qv[0] + h * (qw * w[0] + wxq[0]),
                        qv[1] + h * (qw * w[1] + wxq[1]),
                        qv[2] + h * (qw * w[2] + wxq[2])};
  const double nn = sqrt(nq[0] * nq[0] + nq[1] * nq[1] + nq[2] * nq[2] + nq[3] * nq[3]);
  for (int e = 0; e < 4; ++e) q[e] = nq[e] / nn;
  a.posf[p] = make_float4((float)st[0], (float)st[1], (float)st[2], a.desc[p].rb);
}

__device__ void integrate_particle(const DemArgs& a, int p) {
  double F[3] = {0.0, 0.0, 0.0}, T[3] = {0.0, 0.0, 0.0};
  // slots not in contact hold no force: adding their zeros would change no bit, so they are skipped
  for (int j = 0; j < a.P; ++j)
    if (j != p && a.act[j < p ? (size_t)j * a.P + p : (size_t)p * a.P + j]) add_pair(a, p, j, F, T);
  advance_particle(a, p, F, T);
}

// ---- every DEM step of one LBM step in one thread-block cluster ------------------------------
// A DEM step is chains of binary64 operations, and one such warp instruction holds its quarter
// of an SM for 64 cycles whatever the warp's active lanes (measured, dependent or not), so the cost
// is the number of binary64 instructions per warp. One thread per slot and per particle (512
// threads of one block) issued vector components, sums over control points, Hessian entries and
// cofactors one after the other: 221 us per LBM step for 50 particles of a 120 x 120 x 180 box
// with nothing in contact, about 600 us with its floor covered. Here the slots in reach are
// compacted, a pair takes one warp (a half per particle), a face or a particle half a warp, with
// lanes for the components of vectors and matrices, the control points, the ten sums of Eq. 3 and its
// derivatives and the determinants; slots and particles spread over the SMs of a cluster. Every value
// is formed by the same operations in the same order as in the functions above (sums over
// control points by one lane in index order; x - y as x + (-y)), so the results are theirs bit for
// bit.
constexpr int DEM_CLUSTER = 8, DEM_THREADS = 256, DEM_WARPS = DEM_THREADS / 32;
constexpr int DEM_FUSED_MAX_P = 128;

struct HalfWarp {          // shared scratch of half a warp
  double t[DEM_MAX_CP][6];  // per control point: k/r^2, its first and second derivative factors, r
  double o[10];             // f, gradient, Hessian
};

// Where a half warp's lane finds itself: mask of the half's lanes, lane within it, the component e
// it holds of a vector (lanes 0-2; the others repeat them), scratch; and the control point it holds
// (n in all).
struct Half {
  unsigned mask;
  int hl, e, n;
  HalfWarp* s;
  double c[3], k;
};
__device__ __forceinline__ double from(const Half& w, double v, int lane) { return __shfl_sync(w.mask, v, lane, 16); }
__device__ __forceinline__ double comp3(const double* v, int e) { return e == 0 ? v[0] : e == 1 ? v[1] : v[2]; }
__device__ __forceinline__ void gather3(const Half& w, double v, double out[3]) {
  for (int e = 0; e < 3; ++e) out[e] = from(w, v, e);
}
// u . v of lane components
__device__ __forceinline__ double lane_dot(const Half& w, double u, double v) {
  double p[3];
  gather3(w, u * v, p);
  return p[0] + p[1] + p[2];
}
// component e of u x v
__device__ __forceinline__ double lane_cross(const Half& w, double u, double v) {
  const int e1 = w.e == 2 ? 0 : w.e + 1, e2 = w.e == 0 ? 2 : w.e - 1;
  return from(w, u, e1) * from(w, v, e2) - from(w, u, e2) * from(w, v, e1);
}
// quat_matrix: lane 3 r + c < 9 forms R[r][c]
__device__ __forceinline__ double lane_rotation(const Half& w, const double* q, int r, int c) {
  const bool diag = r == c;
  const int r1 = r == 2 ? 0 : r + 1, r2 = r == 0 ? 2 : r - 1;   // cyclic neighbours of the axis
  const double m0 = q[1 + (diag ? r1 : r)], m1 = diag ? m0 : q[1 + c];
  const double n0 = diag ? q[1 + r2] : q[0], n1 = diag ? n0 : q[1 + (3 - r - c)];
  const double u = m0 * m1, v = n0 * n1;
  const double two = 2.0 * (u + (!diag && c == r1 ? -v : v));
  return diag ? 1.0 - two : two;
}

__device__ void half_points(const DemArgs& a, Half& w, int p, const double org[3]) {
  const int l = w.hl < 9 ? w.hl : 0;
  const double Rl = lane_rotation(w, a.st + 13 * p + 3, l / 3, l % 3);
  const double z = a.zoom[p];
  const ParticleDesc& d = a.desc[p];
  w.n = min(d.c1 - d.c0, DEM_MAX_CP);
  const float4 cb = w.hl < w.n ? a.cbody[d.c0 + w.hl] : make_float4(0.f, 0.f, 0.f, 0.f);
  const double b[3] = {z * (double)cb.x, z * (double)cb.y, z * (double)cb.z};
  for (int e = 0; e < 3; ++e)
    w.c[e] = org[e] + from(w, Rl, 3 * e) * b[0] + from(w, Rl, 3 * e + 1) * b[1] + from(w, Rl, 3 * e + 2) * b[2];
  w.k = z * z * (double)cb.w;
}

// mb_eval: lane i < n forms control point i's terms, lane m < 10 sums one of the ten results over
// the points in order
__device__ double half_eval(const Half& w, const double x[3], double g[3], double H[6]) {
  HalfWarp& s = *w.s;
  if (w.hl < w.n) {
    const double r[3] = {x[0] - w.c[0], x[1] - w.c[1], x[2] - w.c[2]};
    const double r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
    const double inv2 = 1.0 / r2;
    const double fi = w.k * inv2;
    double* t = s.t[w.hl];
    t[0] = fi;
    t[1] = -2.0 * fi * inv2;
    t[2] = 8.0 * fi * inv2 * inv2;
    t[3] = r[0]; t[4] = r[1]; t[5] = r[2];
  }
  __syncwarp(w.mask);
  const int m = w.hl;   // 0: f, 1-3: g, 4-6: H xx yy zz, 7-9: H xy xz yz
  const int ia = m < 4 ? (m + 2) % 3 : m < 7 ? m - 4 : m < 9 ? 0 : 1, ib = m < 7 ? ia : m == 7 ? 1 : 2;
  double acc = 0.0;
  for (int i = 0; i < w.n; ++i) {
    const double* t = s.t[i];
    const double p = (m < 4 ? t[1] : t[2]) * t[3 + ia], p2 = p * t[3 + ib], d = t[1] + p2;
    acc += m == 0 ? t[0] : m < 4 ? p : m < 7 ? d : p2;
  }
  if (m < 10) s.o[m] = acc;
  __syncwarp(w.mask);
  const double f = s.o[0];
  for (int e = 0; e < 3; ++e) g[e] = s.o[1 + e];
  for (int e = 0; e < 6; ++e) H[e] = s.o[4 + e];
  __syncwarp(w.mask);
  return f;
}

// solve3: lane q & 3 = 0 forms the determinant, 1-3 that with column q - 1 replaced by b; returns
// lane e's component of the solution in d
__device__ bool half_solve3(const Half& w, const double A[3][3], const double b[3], double& d) {
  const int q = w.hl & 3;
  double M[3][3];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) M[r][c] = c + 1 == q ? b[r] : A[r][c];
  const double v = M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1])
                 - M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0])
                 + M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
  const double det = from(w, v, 0);
  if (!(fabs(det) > 1e-300)) return false;
  d = from(w, v / det, w.e + 1);
  return true;
}

// newton_update. Its length is compared as a square: the correctly rounded root of s exceeds 1 where
// s > 1 + 2^-52, and 1e-12 where s > 0x1.357c299a88ea8p-80 (the largest double whose root does not).
__device__ bool half_newton(const Half& w, const double A[3][3], const double G[3], double x[3]) {
  const double b[3] = {-G[0], -G[1], -G[2]};
  double d;
  if (!half_solve3(w, A, b, d)) return false;
  const double s = lane_dot(w, d, d);
  double step = d;
  if (s > 0x1.0000000000001p+0) step = 1.0 / sqrt(s) * d;
  gather3(w, comp3(x, w.e) + step, x);
  return s > 0x1.357c299a88ea8p-80;
}

__device__ void half_surface_along(const Half& w, const double xm[3], double xc[3]) {
  double g[3], gx[3], H[6], x[3];
  const double f = half_eval(w, xm, g, H);
  const double xme = comp3(xm, w.e), ge = comp3(g, w.e);
  const double q1 = (1.0 - f) / lane_dot(w, ge, ge);
  double lo = 0.0, hi = q1, q = q1;
  bool inside = false;
  for (int h = 0; h <= SURFACE_HALVINGS; ++h) {
    gather3(w, xme + hi * ge, x);
    if (half_eval(w, x, gx, H) >= 1.0) { inside = true; break; }
    hi = 0.5 * hi;
  }
  if (inside) {
    q = hi;
    for (int it = 0; it < SURFACE_ITERS; ++it) {
      gather3(w, xme + q * ge, x);
      const double fx = half_eval(w, x, gx, H);
      if (fx == 1.0) break;
      if (fx > 1.0) hi = q; else lo = q;
      const double dq = lane_dot(w, comp3(gx, w.e), ge);
      double qn = fabs(dq) > 1e-300 ? q - (fx - 1.0) / dq : 0.5 * (lo + hi);
      if (!(qn > lo && qn < hi)) qn = 0.5 * (lo + hi);
      if (qn == q) break;
      q = qn;
    }
  }
  gather3(w, xme + q * ge, xc);
}

// point_velocity, lane components: v + w x (x - org) of particle p
__device__ __forceinline__ double lane_point_velocity(const DemArgs& a, const Half& w, int p, double r) {
  const double* st = a.st + 13 * p;
  return st[7 + w.e] + lane_cross(w, st[10 + w.e], r);
}

// contact_force, lane components
__device__ double lane_contact_force(const DemArgs& a, const Half& w, double delta, double n, double vi, double vj,
                                     double& xi) {
  const double vr = vj - vi;
  const double vn = lane_dot(w, vr, n);
  double Fn = a.kn * delta - a.etan * vn;
  if (Fn < 0.0) Fn = 0.0;
  const double vt = vr - vn * n;
  const double xn = lane_dot(w, xi, n);
  xi = (xi - xn * n) + vt * a.dt;
  double Ft = a.kt * xi + a.etat * vt;
  const double mag = sqrt(lane_dot(w, Ft, Ft));
  const double lim = a.mus * Fn;
  if (mag > lim) {
    const double sc = lim / mag;
    Ft = Ft * sc;
    xi = a.kt > 0.0 ? (Ft - a.etat * vt) / a.kt : 0.0;
  }
  return Ft - Fn * n;
}

// pair_slot after its prefilter, by one warp (lanes 0-15: particle i, 16-31: particle j)
__device__ void warp_pair_slot(const DemArgs& a, int i, int j, Half& w) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, h = lane >> 4;
  const size_t pr = (size_t)i * a.P + j;
  const double* si = a.st + 13 * i;
  const double* sj = a.st + 13 * j;
  const double sie = si[w.e];
  double de = sj[w.e] - sie;   // minimum image of j's origin seen from i's
  const int wall = w.e == 0 ? a.wall[0] : w.e == 1 ? a.wall[1] : a.wall[2];
  const double len = (double)(w.e == 0 ? a.n[0] : w.e == 1 ? a.n[1] : a.n[2]);
  if (!wall) de -= len * floor(de / len + 0.5);
  const double oje = sie + de;
  const double dd = oje - sie;
  const double reach = (double)a.desc[i].rb + (double)a.desc[j].rb;
  const bool near = !(lane_dot(w, dd, dd) >= reach * reach);
  const bool cont = a.act[pr] != 0;
  double xm[3] = {a.xm[3 * pr], a.xm[3 * pr + 1], a.xm[3 * pr + 2]};
  double xi = a.xi[3 * pr + w.e];
  double F = 0.0, Ti = 0.0, Tj = 0.0;
  bool touch = false;
  if (near) {
    double org[3];
    gather3(w, h ? oje : sie, org);
    half_points(a, w, h ? j : i, org);
    const int n0 = __shfl_sync(full, w.n, 0), n1 = __shfl_sync(full, w.n, 16);
    if (!cont) {   // the closest pair of control points, weighted by radius (first in order on ties)
      double best = INFINITY;
      int at = 0x7fffffff;
      const double rk = sqrt(w.k);
      for (int base = 0; base < n0 * n1; base += 32) {
        const int l = base + lane, ia = min(l / n1, n0 - 1), ib = l - (l / n1) * n1;
        double d[3];
        for (int e = 0; e < 3; ++e) d[e] = __shfl_sync(full, w.c[e], 16 + ib) - __shfl_sync(full, w.c[e], ia);
        const double gap = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]) - __shfl_sync(full, rk, ia) -
                           __shfl_sync(full, rk, 16 + ib);
        if (l < n0 * n1 && gap < best) { best = gap; at = l; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(full, best, o);
        const int oa = __shfl_xor_sync(full, at, o);
        if (ob < best || (ob == best && oa < at)) { best = ob; at = oa; }
      }
      if (at == 0x7fffffff) at = 0;
      const int ba = at / n1, bb = 16 + at - ba * n1;
      const double ra = __shfl_sync(full, rk, ba), rb = __shfl_sync(full, rk, bb), wr = ra / (ra + rb);
      for (int e = 0; e < 3; ++e) {
        const double ca = __shfl_sync(full, w.c[e], ba), cb = __shfl_sync(full, w.c[e], bb);
        xm[e] = ca + wr * (cb - ca);
      }
    }
    const int iters = cont ? NEWTON_CONT : NEWTON_NEW;
    for (int it = 0; it < iters; ++it) {
      double g[3], H[6], G[3], S[6];
      half_eval(w, xm, g, H);
      for (int e = 0; e < 3; ++e) G[e] = g[e] + __shfl_xor_sync(full, g[e], 16);
      for (int e = 0; e < 6; ++e) S[e] = H[e] + __shfl_xor_sync(full, H[e], 16);
      const double A[3][3] = {{S[0], S[3], S[4]}, {S[3], S[1], S[5]}, {S[4], S[5], S[2]}};
      if (!half_newton(w, A, G, xm)) break;   // the same in both halves
    }
    double xc[3];
    half_surface_along(w, xm, xc);
    __syncwarp();
    const double xc0 = __shfl_sync(full, comp3(xc, w.e), w.e), d = __shfl_sync(full, comp3(xc, w.e), 16 + w.e) - xc0;
    const double dist = sqrt(lane_dot(w, d, d));
    const double Rs0 = a.Rs[i], Rs1 = a.Rs[j];
    const double delta = Rs0 + Rs1 - dist;
    touch = delta > 0.0;
    if (touch) {
      const double nrm = dist > 0.0 ? d / dist : 0.0;
      const double xcp = xc0 + (Rs0 - 0.5 * delta) * nrm;
      const double ri = xcp - sie, rj = xcp - oje;
      const double vi = lane_point_velocity(a, w, i, ri), vj = lane_point_velocity(a, w, j, rj);
      F = lane_contact_force(a, w, delta, nrm, vi, vj, xi);
      Ti = lane_cross(w, ri, F);
      Tj = lane_cross(w, rj, -F);
    }
  }
  __syncwarp();
  if (lane == 0) a.act[pr] = touch ? 1 : 0;
  if (lane < 3) {
    if (near) a.xm[3 * pr + lane] = comp3(xm, lane);
    a.xi[3 * pr + lane] = touch ? xi : 0.0;
    a.pF[3 * pr + lane] = F;
    a.pTi[3 * pr + lane] = Ti;
    a.pTj[3 * pr + lane] = Tj;
  }
}

// wall_slot after its prefilter, by half a warp: particle p, face f = 2 axis + side
__device__ void half_wall_slot(const DemArgs& a, int p, int f, Half& w) {
  const size_t wi = 6 * (size_t)p + f;
  const int ax = f >> 1, side = f & 1;
  const double* sp = a.st + 13 * p;
  const double L = (double)a.n[ax];
  const double gap = side ? L - sp[ax] : sp[ax];
  const bool near = a.wall[ax] && !(gap >= (double)a.desc[p].rb);
  const bool cont = a.actw[wi] != 0;
  double xm[3] = {a.xmw[3 * wi], a.xmw[3 * wi + 1], a.xmw[3 * wi + 2]};
  double xi = a.xiw[3 * wi + w.e];
  double F = 0.0, T = 0.0;
  bool touch = false;
  if (near) {
    half_points(a, w, p, sp);
    const double sg = side ? -1.0 : 1.0;
    if (!cont) {   // the control point reaching closest to the face (first in order on ties)
      const double rk = sqrt(w.k), ca = comp3(w.c, ax);
      const double reach = side ? -(ca + rk) : ca - rk;
      double best = INFINITY;
      int bi = 0x7fffffff;
      if (w.hl < w.n && reach < best) { best = reach; bi = w.hl; }
      for (int o = 8; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(w.mask, best, o, 16);
        const int oi = __shfl_xor_sync(w.mask, bi, o, 16);
        if (ob < best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (bi == 0x7fffffff) bi = 0;
      const double rb = from(w, rk, bi);
      for (int e = 0; e < 3; ++e) {
        xm[e] = from(w, w.c[e], bi);
        if (e == ax) xm[e] -= sg * rb;
      }
    }
    const int iters = cont ? NEWTON_CONT : NEWTON_NEW;
    for (int it = 0; it < iters; ++it) {
      double g[3], H[6];
      const double fx = half_eval(w, xm, g, H);
      const double G[3] = {ax == 0 ? g[1] : g[0], ax == 2 ? g[1] : g[2], fx - 1.0};
      // rows of the Hessian of the two axes along the face
      const double A[3][3] = {{ax == 0 ? H[3] : H[0], ax == 0 ? H[1] : H[3], ax == 0 ? H[5] : H[4]},
                              {ax == 2 ? H[3] : H[4], ax == 2 ? H[1] : H[5], ax == 2 ? H[5] : H[2]},
                              {g[0], g[1], g[2]}};
      if (!half_newton(w, A, G, xm)) break;
    }
    const double wall = side ? L : 0.0;
    const double dist = (comp3(xm, ax) - wall) * sg;
    const double delta = a.Rs[p] - dist;
    touch = delta > 0.0;
    if (touch) {
      const double nrm = w.e == ax ? sg : 0.0;
      const double xcp = (w.e == ax ? wall : comp3(xm, w.e)) + 0.5 * delta * nrm;
      const double r = xcp - sp[w.e];
      const double vi = lane_point_velocity(a, w, p, r);
      F = lane_contact_force(a, w, delta, -nrm, vi, 0.0, xi);
      T = lane_cross(w, r, F);
    }
  }
  __syncwarp(w.mask);
  if (w.hl == 0) a.actw[wi] = touch ? 1 : 0;
  if (w.hl < 3) {
    if (near) a.xmw[3 * wi + w.hl] = comp3(xm, w.hl);
    a.xiw[3 * wi + w.hl] = touch ? xi : 0.0;
    a.wF[3 * wi + w.hl] = F;
    a.wT[3 * wi + w.hl] = T;
  }
}

// integrate_particle by half a warp: lanes 0-2 hold the force sums, 3-5 the torque sums
__device__ void half_integrate(const DemArgs& a, int p, const unsigned char* partner, int np, const Half& w) {
  const bool tor = w.hl >= 3 && w.hl < 6;
  double S = 0.0;
  for (int k = 0; k < np; ++k) {
    const int j = partner[k];
    const size_t at = 3 * (j < p ? (size_t)j * a.P + p : (size_t)p * a.P + j) + w.e;
    const double v = tor ? (j < p ? a.pTj[at] : a.pTi[at]) : a.pF[at];
    S = S + (!tor && j < p ? -v : v);
  }
  for (int f = 0; f < 6; ++f)
    if (a.actw[6 * (size_t)p + f]) {
      const size_t at = 3 * (6 * (size_t)p + f) + w.e;
      S = S + (tor ? a.wT[at] : a.wF[at]);
    }
  const double m = a.mass[p], dt = a.dt;
  if (a.Fe) S = S + a.Fe[6 * p + (tor ? 3 : 0) + w.e];
  const double F = S + m * (w.e == 0 ? a.g[0] : w.e == 1 ? a.g[1] : a.g[2]);   // lanes 0-2
  const double T = from(w, S, 3 + w.e);
  double* st = a.st + 13 * p;
  double q[4];
  for (int e = 0; e < 4; ++e) q[e] = st[3 + e];
  // translation: symplectic Euler
  const double vel = st[7 + w.e] + dt * (F / m);
  const double pos = st[w.e] + dt * vel;
  // rotation: I_w = R I_b R^T, w += dt I_w^-1 (T - w x I_w w); lane 3 r + c < 9 holds entry (r, c)
  const int l = w.hl < 9 ? w.hl : 0, r = l / 3, c = l - 3 * r;
  const double R = lane_rotation(w, q, r, c);
  const double* I6 = a.Ib + 6 * p;   // xx yy zz xy xz yz
  const double I0 = I6[c == 0 ? 0 : 2 + c], I1 = I6[c == 0 ? 3 : c == 1 ? 1 : 5], I2 = I6[c == 2 ? 2 : 4 + c];
  const double RI = from(w, R, 3 * r) * I0 + from(w, R, 3 * r + 1) * I1 + from(w, R, 3 * r + 2) * I2;
  const double Iwl = from(w, RI, 3 * r) * from(w, R, 3 * c) + from(w, RI, 3 * r + 1) * from(w, R, 3 * c + 1) +
                     from(w, RI, 3 * r + 2) * from(w, R, 3 * c + 2);
  double Iw[3][3];
  for (int e = 0; e < 9; ++e) Iw[e / 3][e % 3] = from(w, Iwl, e);
  double spin = st[10 + w.e], ws[3];
  gather3(w, spin, ws);
  const double Lw = (w.e == 0 ? Iw[0][0] : w.e == 1 ? Iw[1][0] : Iw[2][0]) * ws[0] +
                    (w.e == 0 ? Iw[0][1] : w.e == 1 ? Iw[1][1] : Iw[2][1]) * ws[1] +
                    (w.e == 0 ? Iw[0][2] : w.e == 1 ? Iw[1][2] : Iw[2][2]) * ws[2];
  double rhs[3], dw;
  gather3(w, T - lane_cross(w, spin, Lw), rhs);
  if (half_solve3(w, Iw, rhs, dw)) spin = spin + dt * dw;
  gather3(w, spin, ws);
  // orientation: q += dt/2 (0, w) q, normalised; lane 0: qw - h (w.q), lanes 1-3: q_e + h (qw w + w x q)_e
  const double h = 0.5 * dt;
  const int i = w.hl & 3, e0 = i == 0 ? 0 : i - 1, e1 = e0 == 2 ? 0 : e0 + 1, e2 = e0 == 0 ? 2 : e0 - 1;
  const double m0 = i == 0 ? ws[0] * q[1] : q[0] * comp3(ws, e0);
  const double m1 = comp3(ws, e1) * comp3(q + 1, i == 0 ? e1 : e2);   // i = 0: w1 q1; else w_{e1} q_{e2}
  const double m2 = comp3(ws, e2) * comp3(q + 1, i == 0 ? e2 : e1);
  const double t = i == 0 ? m0 + m1 : m1 + -m2;
  const double u = i == 0 ? t + m2 : m0 + t;
  const double hu = h * u;
  const double nql = (i == 0 ? q[0] : comp3(q + 1, e0)) + (i == 0 ? -hu : hu);
  const double sq = nql * nql;
  const double nn = sqrt(from(w, sq, 0) + from(w, sq, 1) + from(w, sq, 2) + from(w, sq, 3));
  const double qn = nql / nn;
  __syncwarp(w.mask);   // the state has been read
  if (w.hl < 3) {
    st[w.hl] = pos;
    st[7 + w.hl] = vel;
    st[10 + w.hl] = spin;
  }
  if (w.hl < 4) st[3 + w.hl] = qn;
  double o[3];
  gather3(w, pos, o);
  if (w.hl == 0) a.posf[p] = make_float4((float)o[0], (float)o[1], (float)o[2], a.desc[p].rb);
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
}

__global__ void __cluster_dims__(DEM_CLUSTER, 1, 1) __launch_bounds__(DEM_THREADS, 1)
dem_cluster_kernel(DemArgs a, int substeps) {
  constexpr int MAX_LOCAL = (DEM_FUSED_MAX_P + DEM_CLUSTER - 1) / DEM_CLUSTER;
  __shared__ HalfWarp s_half[2 * DEM_WARPS];
  __shared__ uint16_t s_pairs[(DEM_FUSED_MAX_P * DEM_FUSED_MAX_P + DEM_CLUSTER - 1) / DEM_CLUSTER];
  __shared__ uint16_t s_walls[(6 * DEM_FUSED_MAX_P + DEM_CLUSTER - 1) / DEM_CLUSTER];
  __shared__ unsigned char s_partner[MAX_LOCAL][DEM_FUSED_MAX_P];
  __shared__ int s_np, s_nw;
  const int P = a.P, rank = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, half = lane >> 4;
  Half w;
  w.mask = 0xffffu << (16 * half);
  w.hl = lane & 15;
  w.e = w.hl % 3;
  w.n = 0;
  w.s = s_half + 2 * warp + half;
  for (int step = 0; step < substeps; ++step) {
    if (threadIdx.x == 0) { s_np = 0; s_nw = 0; }
    __syncthreads();
    // slots within binary32 reach (bound spheres apart by more than a margin cannot touch), dealt
    // out to the blocks one by one; slots that left reach are cleared
    for (int k = threadIdx.x * DEM_CLUSTER + rank; k < P * P + 6 * P; k += DEM_THREADS * DEM_CLUSTER) {
      if (k < P * P) {
        const int i = k / P, j = k - i * P;
        if (i >= j) continue;
        const float4 pi = a.posf[i], pj = a.posf[j];
        const float dv[3] = {pj.x - pi.x, pj.y - pi.y, pj.z - pi.z};
        float d2 = 0.0f;
        for (int e = 0; e < 3; ++e) {
          float dd = dv[e];
          if (!a.wall[e]) dd -= (float)a.n[e] * rintf(dd / (float)a.n[e]);
          d2 += dd * dd;
        }
        const float reach = pi.w + pj.w + 0.01f;
        if (d2 > reach * reach) {
          if (a.act[k]) { a.act[k] = 0; clear3(a.xi + 3 * (size_t)k); }
        } else {
          s_pairs[atomicAdd(&s_np, 1)] = (uint16_t)k;
        }
      } else {
        const int wi = k - P * P, p = wi / 6, ax = (wi - 6 * p) >> 1, side = wi & 1;
        const float4 pf = a.posf[p];
        const float c = ax == 0 ? pf.x : ax == 1 ? pf.y : pf.z;
        const float gapf = side ? (float)a.n[ax] - c : c;
        if (!a.wall[ax] || gapf > pf.w + 0.01f) {
          if (a.actw[wi]) { a.actw[wi] = 0; clear3(a.xiw + 3 * (size_t)wi); }
        } else {
          s_walls[atomicAdd(&s_nw, 1)] = (uint16_t)wi;
        }
      }
    }
    __syncthreads();
    for (int k = warp; k < s_np; k += DEM_WARPS) {
      const int pr = s_pairs[k];
      warp_pair_slot(a, pr / P, pr % P, w);
    }
    // faces from the last warp on, so that they land beside the fewest pairs
    for (int k = 2 * (DEM_WARPS - 1 - warp) + half; k < s_nw; k += 2 * DEM_WARPS) {
      const int wi = s_walls[k];
      half_wall_slot(a, wi / 6, wi % 6, w);
    }
    __syncwarp();   // the halves of a warp may have left the loop apart
    cluster_barrier();
    // this block's particles, two per warp: their partners in contact by index, then the integration
    const int local = (P - rank + DEM_CLUSTER - 1) / DEM_CLUSTER;
    for (int l0 = 2 * warp; l0 < local; l0 += 2 * DEM_WARPS) {
      int np = 0;
      for (int k = 0; k < 2 && l0 + k < local; ++k) {
        const int p = (l0 + k) * DEM_CLUSTER + rank;
        int n = 0;
        for (int base = 0; base < P; base += 32) {
          const int j = base + lane;
          const bool on = j < P && j != p && a.act[j < p ? j * P + p : p * P + j];
          const unsigned bal = __ballot_sync(0xffffffffu, on);
          if (on) s_partner[l0 + k][n + __popc(bal & ((1u << lane) - 1u))] = (unsigned char)j;
          n += __popc(bal);
        }
        if (half == k) np = n;
      }
      __syncwarp();
      if (l0 + half < local) half_integrate(a, (l0 + half) * DEM_CLUSTER + rank, s_partner[l0 + half], np, w);
      __syncwarp();
    }
    cluster_barrier();
  }
}

// zoom s_p = 1 - R_s,p / R_c,p with R_c,p = max_i (|c_i| + sqrt(k_i)) over the body frame
__global__ void dem_init_kernel(DemArgs a) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.P) return;
  double r = 0.0;
  for (int i = a.desc[p].c0; i < a.desc[p].c1; ++i) {
    const float4 cb = a.cbody[i];
    const double x = (double)cb.x, y = (double)cb.y, z = (double)cb.z;
    const double e = sqrt(x * x + y * y + z * z) + sqrt((double)cb.w);
    if (e > r) r = e;
  }
  a.zoom[p] = 1.0 - a.Rs[p] / r;
  const double* st = a.st + 13 * p;
  a.posf[p] = make_float4((float)st[0], (float)st[1], (float)st[2], a.desc[p].rb);
}

// Mass properties from the metaball: body-frame sample points (i + 1/2) h, h = 1/4, out to the
// bound radius (N points per half-axis), inside when the binary32 sum reaches 1; integer sums in
// units of h/2 per particle: count, coordinates (3), products (xx yy zz xy xz yz). One block per
// particle; the sums are exact, so their order does not matter.
__global__ void dem_mass_sums_kernel(DemArgs a, unsigned long long* sums) {
  const int p = blockIdx.x;
  const ParticleDesc& d = a.desc[p];
  const int N = (int)ceil((double)d.rb / 0.25) + 1;
  const int side = 2 * N;
  const long long total = (long long)side * side * side;
  long long v[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (long long m = threadIdx.x; m < total; m += blockDim.x) {
    const int i = (int)(m % side) - N, j = (int)((m / side) % side) - N, k = (int)(m / ((long long)side * side)) - N;
    const int ca = 2 * i + 1, cb = 2 * j + 1, cc = 2 * k + 1;
    const float x = (float)ca * 0.125f, y = (float)cb * 0.125f, z = (float)cc * 0.125f;
    float f = 0.0f;
    for (int q = d.c0; q < d.c1; ++q) {
      const float4 c = a.cbody[q];
      const float dx = x - c.x, dy = y - c.y, dz = z - c.z;
      const float xx = dx * dx, yy = dy * dy, zz = dz * dz;
      float r2 = xx + yy;
      r2 = r2 + zz;
      f = f + c.w / r2;
    }
    if (f >= 1.0f) {
      v[0] += 1; v[1] += ca; v[2] += cb; v[3] += cc;
      v[4] += (long long)ca * ca; v[5] += (long long)cb * cb; v[6] += (long long)cc * cc;
      v[7] += (long long)ca * cb; v[8] += (long long)ca * cc; v[9] += (long long)cb * cc;
    }
  }
  for (int e = 0; e < 10; ++e) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
    if ((threadIdx.x & 31) == 0 && v[e]) atomicAdd(&sums[10 * p + e], (unsigned long long)v[e]);
  }
}

// Per particle: mass, centre of mass and inertia about it (the oracle's formulas and order);
// moves the body frame to the centre of mass (control points c_i - c_m in binary32, state
// origin + c_m)
__global__ void dem_mass_finish_kernel(DemArgs a, const unsigned long long* sums, const double* density,
                                       double* mass, double* Ib, double* props, float4* cbody) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.P) return;
  long long S[10];
  for (int e = 0; e < 10; ++e) S[e] = (long long)sums[10 * p + e];
  const double dn = (double)S[0];
  const double rho = density[p];
  double* out = props + 10 * p;
  out[0] = rho * (dn * 0.015625);
  double cm[3];
  for (int e = 0; e < 3; ++e) { cm[e] = ((double)S[1 + e] * 0.125) / dn; out[1 + e] = cm[e]; }
  const int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};
  double J[6];
  const double w = rho * 0.015625;
  for (int m = 0; m < 6; ++m) J[m] = ((double)S[4 + m] * 0.015625 - (dn * cm[ia[m]]) * cm[ib[m]]) * w;
  out[4] = J[1] + J[2];
  out[5] = J[0] + J[2];
  out[6] = J[0] + J[1];
  out[7] = -J[3];
  out[8] = -J[4];
  out[9] = -J[5];
  mass[p] = out[0];
  for (int m = 0; m < 6; ++m) Ib[6 * p + m] = out[4 + m];
  for (int q = a.desc[p].c0; q < a.desc[p].c1; ++q) {
    float4 c = cbody[q];
    c.x = (float)((double)c.x - cm[0]);
    c.y = (float)((double)c.y - cm[1]);
    c.z = (float)((double)c.z - cm[2]);
    cbody[q] = c;
  }
  for (int e = 0; e < 3; ++e) a.st[13 * p + e] = a.st[13 * p + e] + cm[e];
}

}  // namespace

void launch_dem_mass(const DemArgs& a, unsigned long long* sums, const double* density, double* mass, double* Ib,
                     double* props, float4* cbody, cudaStream_t st) {
  if (a.P <= 0) return;
  dem_mass_sums_kernel<<<(unsigned)a.P, 256, 0, st>>>(a, sums);
  dem_mass_finish_kernel<<<(unsigned)((a.P + 127) / 128), 128, 0, st>>>(a, sums, density, mass, Ib, props, cbody);
}

void launch_dem_init(const DemArgs& a, cudaStream_t st) {
  if (a.P > 0) dem_init_kernel<<<(unsigned)((a.P + 127) / 128), 128, 0, st>>>(a);
}

int launch_dem(const DemArgs& a, int substeps, cudaStream_t st) {
  if (a.P <= 0) return 0;
  const int npairs = a.P * (a.P - 1) / 2;
  if (a.P <= DEM_FUSED_MAX_P) {   // one cluster takes every step
    dem_cluster_kernel<<<DEM_CLUSTER, DEM_THREADS, 0, st>>>(a, substeps);
    return 1;
  }
  const int slots = npairs + 6 * a.P;
  const unsigned cblocks = (unsigned)((slots + 63) / 64), iblocks = (unsigned)((a.P + 127) / 128);
  for (int s = 0; s < substeps; ++s) {
    dem_contacts_kernel<<<cblocks, 64, 0, st>>>(a, npairs);
    dem_integrate_kernel<<<iblocks, 128, 0, st>>>(a);
  }
  return 2 * substeps;
}

}  // namespace rwmi
