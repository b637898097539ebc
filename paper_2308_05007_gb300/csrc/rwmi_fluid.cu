// rwmi_fluid.cu -- particle poses and brick lists, metaball rasteriser, fluid set-up and
// read-back (the LBM kernel itself is in rwmi_lbm.cu).
//
// Kernels (one timestep t):
//   pose_bin_kernel   particle pose at a time (prescribed motion, or read from the free DEM's
//                     state), world control points, brick candidate lists, body force, zeroed
//                     force/momentum accumulators
//   raster_kernel     solid sub-sample count + owner for every cell of bricks that touch a
//                     particle (Eq. 3, 4x4x4 sub-samples, binary32 decisions bit-identical to
//                     the CPU oracle's); with the paper's coupling the solid/fluid node classes
//   refill_kernel     with the paper's coupling: node classes of the other bricks, refilling of
//                     nodes uncovered since the previous step (Eq. 27)
#include "rwmi_lattice.cuh"

namespace rwmi {

void lattice_table(int q, int32_t* e, double* w) {
  for (int i = 0; i < q; ++i) {
    for (int a = 0; a < 3; ++a) e[3 * i + a] = q == 15 ? Lat<15>::e(i, a) : Lat<19>::e(i, a);
    const int e2 = q == 15 ? Lat<15>::e2(i) : Lat<19>::e2(i);
    w[i] = q == 15 ? (e2 == 0 ? 2.0 / 9.0 : e2 == 1 ? 1.0 / 9.0 : 1.0 / 72.0)
                   : (e2 == 0 ? 1.0 / 3.0 : e2 == 1 ? 1.0 / 18.0 : 1.0 / 36.0);
  }
}

// ------------------------------------------------------------------------------------------
// Prescribed particle motion and brick candidate lists
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ double wrap_d(double x, double n, int wall) {
  return wall ? x : __dsub_rn(x, __dmul_rn(n, floor(__ddiv_rn(x, n))));
}

struct PoseArgs {
  Geom g;
  ParticleSet ps;
  BrickSet bs;
  const int64_t* d_T;
  int t_offset, zero_acc;
  double F0x, F0y, F0z, fper;
  double* acc;
  int q;          // lattice (15 or 19) and Guo factor 1 - 1/(2 tau) of the pair constants
  double guo0;
};

// One block per particle, blk = p of nblk = max(P, 1) blocks (block 0 also writes the body force
// of this time). The kernel is a short chain of binary64 operations on a narrow pipe (two lanes
// per cycle), ahead of everything else in the step, so independent pieces go to different warps and
// independent components to different lanes: the sines and cosines of the drive and the spin to
// warps 0-3, the body force and its constants to warp 4 (block 0), rotation entries, axes and
// control point coordinates one per lane, the brick ranges once per axis instead of in every
// thread. 64 particles at 256^3: 19.7 -> 14.3 us.
// Explicitly rounded FP64 operations in the oracle's order: the binary32 control points must
// round identically on both sides, so no fused multiply-add here.
__device__ void pose_bin_body(const PoseArgs& A, int blk, int nblk) {
  const Geom& g = A.g;
  const ParticleSet& ps = A.ps;
  const BrickSet& bs = A.bs;
  double* __restrict__ acc = A.acc;
  const int64_t t = *A.d_T + A.t_offset;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (blk == 0 && warp == 4) {   // the body force of this time and the Guo pair constants
    double s = 1.0;
    if (A.fper > 0.0) {
      if (lane == 0) s = sin(2.0 * 3.141592653589793 * (double)t / A.fper);
      s = __shfl_sync(0xffffffffu, s, 0);
    }
    const double F[3] = {A.F0x * s, A.F0y * s, A.F0z * s};
    if (lane == 0)
      for (int a = 0; a < 3; ++a) {
        bs.sp->Fd[a] = F[a];
        bs.sp->F[a] = (float)F[a];
      }
    // one constant per lane (a serial loop cost 4 us a step)
    const int H = (A.q - 1) / 2;
    if (lane < 2 * H) {
      const int i = 1 + (lane >> 1);
      double eF = 0.0;
      for (int a = 0; a < 3; ++a) eF += (double)(A.q == 15 ? Lat<15>::e(i, a) : Lat<19>::e(i, a)) * F[a];
      const double wg = (A.q == 15 ? Lat<15>::wt<double>(i) : Lat<19>::wt<double>(i)) * A.guo0;
      const double k = ((lane & 1) ? 3.0 : 9.0) * wg * eF;
      guo_pairs(bs.sp)->kd[lane] = k;
      guo_pairs(bs.sp)->k[lane] = (float)k;
    }
  }
  if (A.zero_acc) {   // force/torque [6P] + striped mass/momentum [4 RED_SLOTS] accumulators of this time
    for (int m = blk * blockDim.x + threadIdx.x; m < 6 * ps.P + 4 * RED_SLOTS; m += nblk * blockDim.x)
      acc[m] = 0.0;
  }
  const int p = blk;
  if (p >= ps.P) return;
  __shared__ double sR[9], so[3], s_ow[3];   // rotation, origin, wrapped origin
  __shared__ double s_trig[4];               // sine and cosine of the drive, of the spin angle
  __shared__ int s_ra[3][2], s_rb[3][2], s_nr[3];
  const ParticleDesc& d = ps.desc[p];
  const double wn = ps.dem ? 0.0
      : __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(d.omega[0], d.omega[0]), __dmul_rn(d.omega[1], d.omega[1])),
                             __dmul_rn(d.omega[2], d.omega[2])));
  if (lane == 0 && warp < 4 && !ps.dem) {
    if (warp < 2) {   // drive
      double v = 0.0;
      if (d.period > 0.0) {
        const double th = __dadd_rn(__ddiv_rn(__dmul_rn(6.283185307179586, (double)t), d.period), d.phase);
        v = warp == 0 ? sin(th) : cos(th) * 6.283185307179586 / d.period;
      }
      s_trig[warp] = v;
    } else if (wn > 0.0) {   // constant spin: body frame turned by |omega| t
      const double ang = __dmul_rn(wn, (double)t);
      s_trig[warp] = warp == 2 ? sin(ang) : cos(ang);
    }
  }
  __syncthreads();
  if (warp == 0 && lane < 3) {   // origin, velocity and spin, one axis per lane
    const int a = lane;
    double org, vel, spin;
    if (ps.dem) {   // free DEM: the state's origin, velocity, spin and orientation quaternion
      const double* st = ps.dem + 13 * p;
      org = st[a]; vel = st[7 + a]; spin = st[10 + a];
    } else {
      org = __dadd_rn(d.org[a], __dmul_rn(d.amp[a], s_trig[0]));
      vel = d.amp[a] * s_trig[1];
      spin = d.omega[a];
    }
    so[a] = org;
    const double ow = wrap_d(org, (double)g.n[a], g.wall[a]);
    s_ow[a] = ow;
    PoseF& pf = bs.pose[p];
    pf.o[a] = (float)ow;
    pf.v[a] = (float)vel;
    pf.w[a] = (float)spin;
    pf.pad[a] = 0.0f;
    PoseD& pd = bs.posed[p];
    pd.o[a] = ow;
    pd.v[a] = vel;
    pd.w[a] = spin;
    if (a == 0) pd.pad = 0.0;
  } else if (warp == 1 && lane < 9) {   // rotation, one entry per lane
    const int r = lane / 3, c = lane - 3 * r;
    double v = r == c ? 1.0 : 0.0;
    if (ps.dem) {   // 1 - 2 (y y + z z) on the diagonal, 2 (x y -+ w z) off it
      const double* q = ps.dem + 13 * p + 3;   // w, x, y, z
      const int o = 3 - r - c;   // the third axis of an off-diagonal entry
      const double m0 = r == c ? q[1 + (r + 1) % 3] : q[1 + r], m1 = r == c ? m0 : q[1 + c];
      const double n0 = r == c ? q[1 + (r + 2) % 3] : q[0], n1 = r == c ? n0 : q[1 + o];
      const double u = __dmul_rn(m0, m1), w = __dmul_rn(n0, n1);
      const bool minus = r != c && (c - r + 3) % 3 == 1;
      const double two = __dmul_rn(2.0, minus ? __dsub_rn(u, w) : __dadd_rn(u, w));
      v = r == c ? __dsub_rn(1.0, two) : two;
    } else if (wn > 0.0) {   // Rodrigues: cos I + sin [n]x + (1 - cos) n n^T
      const double nr = __ddiv_rn(d.omega[r], wn), nc = __ddiv_rn(d.omega[c], wn);
      double K = 0.0;
      if (r != c) {
        const double no = __ddiv_rn(d.omega[3 - r - c], wn);
        K = (c - r + 3) % 3 == 1 ? -no : no;
      }
      const double sa = s_trig[2], ca = s_trig[3];
      v = __dadd_rn(__dadd_rn(r == c ? ca : 0.0, __dmul_rn(sa, K)),
                    __dmul_rn(__dmul_rn(__dsub_rn(1.0, ca), nr), nc));
    }
    sR[lane] = v;
  }
  __syncthreads();
  // bricks within rb + walk_margin of the origin. Walker candidates and raster candidates
  // coincide: the raster also writes the walkers' mini-brick masks, which must cover every
  // particle within the walker margin
  const float Rw = d.rb + ps.walk_margin;
  if (warp == 7) {
    // per axis (one lane each), the bricks met by the interval [o - Rw, o + Rw]
    if (lane < 3) {
      const int a = lane;
      const BrickRange r = brick_range(s_ow[a], Rw, g.n[a], g.nb[a], g.wall[a]);
      s_ra[a][0] = r.a[0]; s_rb[a][0] = r.b[0];
      s_ra[a][1] = r.a[1]; s_rb[a][1] = r.b[1];
      s_nr[a] = r.n;
    }
  } else {   // world control points, one coordinate per lane of warps 0-6
    for (int k = threadIdx.x; k < 3 * (d.c1 - d.c0); k += blockDim.x - 32) {
      const int i = d.c0 + k / 3, a = k - 3 * (k / 3);
      const float4 cb = ps.cbody[i];
      const double v = __dadd_rn(__dadd_rn(__dadd_rn(so[a], __dmul_rn(sR[3 * a], (double)cb.x)),
                                           __dmul_rn(sR[3 * a + 1], (double)cb.y)),
                                 __dmul_rn(sR[3 * a + 2], (double)cb.z));
      float* cw = reinterpret_cast<float*>(bs.cworld + i);
      cw[a] = (float)wrap_d(v, (double)g.n[a], g.wall[a]);
      if (a == 0) cw[3] = cb.w;
    }
  }
  __syncthreads();
  float ow[3];
  for (int a = 0; a < 3; ++a) ow[a] = (float)s_ow[a];
  const uint32_t nbrick = (uint32_t)g.nb[0] * g.nb[1] * g.nb[2];
  for (int combo = 0; combo < 8; ++combo) {
    const int sx = combo & 1, sy = (combo >> 1) & 1, sz = combo >> 2;
    if (sx >= s_nr[0] || sy >= s_nr[1] || sz >= s_nr[2]) continue;
    const int lo3[3] = {s_ra[0][sx], s_ra[1][sy], s_ra[2][sz]};
    const int cnt[3] = {s_rb[0][sx] - lo3[0] + 1, s_rb[1][sy] - lo3[1] + 1, s_rb[2][sz] - lo3[2] + 1};
    const int total = cnt[0] * cnt[1] * cnt[2];
  for (int m = threadIdx.x; m < total; m += blockDim.x) {
    int bc[3] = {lo3[0] + m % cnt[0], lo3[1] + (m / cnt[0]) % cnt[1], lo3[2] + m / (cnt[0] * cnt[1])};
    float d2 = 0.0f;
    for (int a = 0; a < 3; ++a) {
      const float b0 = (float)(bc[a] * BRICK), b1 = fminf((float)((bc[a] + 1) * BRICK), (float)g.n[a]);
      const float c = 0.5f * (b0 + b1), h = 0.5f * (b1 - b0);
      float delta = ow[a] - c;
      if (!g.wall[a]) {
        const float na = (float)g.n[a];
        delta -= na * rintf(delta / na);
      }
      const float da = fmaxf(fabsf(delta) - h, 0.0f);
      d2 += da * da;
    }
    bool app = false;   // this particle is the brick's first raster candidate: list the brick
    uint32_t b = 0;
    if (d2 <= Rw * Rw) {
      b = ((uint32_t)bc[2] * g.nb[1] + bc[1]) * g.nb[0] + bc[0];
      const uint32_t old = atomicAdd(&bs.bword[b], 1u + 65536u);
      const uint32_t slot = old & 0xffffu;
      if (slot < MAXC) bs.bcand[b * MAXC + slot] = (uint16_t)(p | 0x8000);
      app = old == 0u;
    }
    // one append per warp: every block's raster bricks go through the single list counter
    const unsigned am = __activemask();
    const unsigned bal = __ballot_sync(am, app);
    if (bal) {
      const int lane = threadIdx.x & 31, leader = __ffs(bal) - 1;
      uint32_t base = 0;
      if (lane == leader) base = atomicAdd(&bs.bword[nbrick], (uint32_t)__popc(bal));
      base = __shfl_sync(am, base, leader);
      if (app) bs.rlist[base + __popc(bal & ((1u << lane) - 1u))] = (int32_t)b;
    }
  }
  }
}

__global__ void pose_bin_kernel(const PoseArgs a) { pose_bin_body(a, blockIdx.x, gridDim.x); }
__global__ void pose_bin_batched(const PoseArgs* __restrict__ args, const BlockMap* __restrict__ map) {
  const BlockMap m = map[blockIdx.x];
  pose_bin_body(args[m.domain], m.block, m.blocks);
}

// One row {t, F_0, T_0, F_1, T_1, ...} of the force series: the forces of the LBM update just
// done (acc), labelled with the steps completed t, read from the device counter, into slot
// (t / interval - 1) mod rows, so that a replayed graph writes the row of the step it runs.
__global__ void force_row_kernel(const double* __restrict__ acc, int P, double* __restrict__ base, int interval,
                                 int rows, const int64_t* __restrict__ d_T, int toff) {
  const int64_t t = *d_T + toff;
  double* row = base + (size_t)(((t / interval) - 1) % rows) * (1 + 6 * (size_t)P);
  for (int m = threadIdx.x; m < 6 * P; m += blockDim.x) row[1 + m] = acc[m];
  if (threadIdx.x == 0) row[0] = (double)t;
}
void launch_force_row(const double* acc, int P, double* base, int interval, int rows, const int64_t* d_T, int toff,
                      cudaStream_t st) {
  force_row_kernel<<<1, 256, 0, st>>>(acc, P, base, interval, rows, d_T, toff);
}

// Zeroes n words. A kernel rather than cudaMemsetAsync: inside the captured step a memset node
// stalled the concurrent branches of the pipelined schedule (measured: 0.14 ms per step).
struct ClearArgs {
  uint32_t* p;
  uint32_t n;
};
__device__ __forceinline__ void clear_body(const ClearArgs& a, int blk, int nblk) {
  for (uint32_t i = blk * blockDim.x + threadIdx.x; i < a.n; i += nblk * blockDim.x) a.p[i] = 0u;
}
__global__ void clear_u32_kernel(const ClearArgs a) { clear_body(a, blockIdx.x, gridDim.x); }
__global__ void clear_batched(const ClearArgs* __restrict__ args, const BlockMap* __restrict__ map) {
  const BlockMap m = map[blockIdx.x];
  clear_body(args[m.domain], m.block, m.blocks);
}
int clear_grid(uint32_t n) {
  const uint32_t blocks = (n + 255) / 256;
  return (int)(blocks > 152 * 8 ? 152 * 8 : blocks);
}
void launch_clear_u32(uint32_t* p, uint32_t n, cudaStream_t st) {
  if (n == 0) return;
  clear_u32_kernel<<<clear_grid(n), 256, 0, st>>>(ClearArgs{p, n});
}
size_t clear_args_size() { return sizeof(ClearArgs); }
void clear_args(void* dst, uint32_t* p, uint32_t n) { *static_cast<ClearArgs*>(dst) = ClearArgs{p, n}; }
void launch_clear_batched(const void* args, const BlockMap* map, int nblocks, cudaStream_t st) {
  if (nblocks > 0) clear_batched<<<nblocks, 256, 0, st>>>(static_cast<const ClearArgs*>(args), map);
}

static PoseArgs make_pose_args(const Geom& g, const ParticleSet& ps, BrickSet bs, const int64_t* d_T,
                               int t_offset, const double F0[3], double force_period, int zero_forces,
                               double* acc, int q, double tau) {
  PoseArgs a;
  a.g = g; a.ps = ps; a.bs = bs; a.d_T = d_T; a.t_offset = t_offset; a.zero_acc = zero_forces;
  a.F0x = F0[0]; a.F0y = F0[1]; a.F0z = F0[2]; a.fper = force_period; a.acc = acc;
  a.q = q; a.guo0 = 1.0 - 0.5 / tau;
  return a;
}
void launch_pose_bin(const Geom& g, const ParticleSet& ps, BrickSet bs, const int64_t* d_T,
                     int t_offset, const double F0[3], double force_period, int zero_forces,
                     double* acc, int q, double tau, cudaStream_t st) {
  const int blocks = ps.P > 0 ? ps.P : 1;
  pose_bin_kernel<<<blocks, 256, 0, st>>>(
      make_pose_args(g, ps, bs, d_T, t_offset, F0, force_period, zero_forces, acc, q, tau));
}
size_t pose_args_size() { return sizeof(PoseArgs); }
void pose_args(void* dst, const Geom& g, const ParticleSet& ps, BrickSet bs, const int64_t* d_T, int t_offset,
               const double F0[3], double force_period, int zero_forces, double* acc, int q, double tau) {
  *static_cast<PoseArgs*>(dst) =
      make_pose_args(g, ps, bs, d_T, t_offset, F0, force_period, zero_forces, acc, q, tau);
}
void launch_pose_batched(const void* args, const BlockMap* map, int nblocks, cudaStream_t st) {
  if (nblocks > 0) pose_bin_batched<<<nblocks, 256, 0, st>>>(static_cast<const PoseArgs*>(args), map);
}

// ------------------------------------------------------------------------------------------
// Rasteriser: per cell, sub-samples (i + (a + 1/2)/4, ...) inside any particle (Eq. 3 >= 1).
// Interval bounds over the cell (half-diagonal 0.6495) and over its eight octants
// (half-diagonal 0.2165) settle most sub-samples; the rest are evaluated with a fast
// reciprocal and, when that lands within 4e-5 of 1, again with the exact binary32 sequence
// shared with the CPU oracle. Bounds are decided with a 1e-3 margin and the fast value with a
// 4e-5 margin, both far above binary32 rounding (~1e-6), so every decision equals the exact one.
// ------------------------------------------------------------------------------------------
struct CellBound { float fmax, fmin; };

// Bounds of Eq. 3 over a ball of radius h about (x, y, z) from the wrapped control points: every
// one is at least r - h and at most r + h away. Fast reciprocal/sqrt: the 1e-3 decision margins
// dwarf their error. (Bricks whose candidates do not fit the staging; the others take pair_bound.)
__device__ __forceinline__ CellBound bound_at(const float4* cw, int c0, int c1, float x, float y, float z, float h,
                                              const Geom& g) {
  CellBound b{0.0f, 0.0f};
  for (int i = c0; i < c1; ++i) {
    const float4 c = cw[i];
    const float dx = min_image_rn(x - c.x, (float)g.n[0], g.wall[0]);
    const float dy = min_image_rn(y - c.y, (float)g.n[1], g.wall[1]);
    const float dz = min_image_rn(z - c.z, (float)g.n[2], g.wall[2]);
    const float r2 = dx * dx + dy * dy + dz * dz;
    const float r = r2 * rsqrtf(fmaxf(r2, 1e-30f));
    const float rmin = fmaxf(r - h, 1e-15f), rmax = r + h;
    b.fmax += __fdividef(c.w, rmin * rmin);
    b.fmin += __fdividef(c.w, rmax * rmax);
  }
  return b;
}

// Is (x, y, z) inside particle [c0, c1) by Eq. 3 in the CPU oracle's binary32 sequence? A fast
// value (fast reciprocal, contraction allowed; error ~1e-6 relative) decides outside 4e-5 of 1,
// the exact sequence inside that band, so the answer always equals the exact one.
__device__ __forceinline__ bool inside_exact(const float4* __restrict__ cw, int c0, int c1, float x, float y,
                                             float z, const Geom& g) {
  float f = 0.0f;
  for (int i = c0; i < c1; ++i) {
    const float4 c = cw[i];
    const float dx = min_image_rn(x - c.x, (float)g.n[0], g.wall[0]);
    const float dy = min_image_rn(y - c.y, (float)g.n[1], g.wall[1]);
    const float dz = min_image_rn(z - c.z, (float)g.n[2], g.wall[2]);
    f += __fdividef(c.w, dx * dx + dy * dy + dz * dz);
  }
  if (fabsf(f - 1.0f) > 4e-5f) return f >= 1.0f;
  return metaball_exact(cw, c0, c1, x, y, z, g) >= 1.0f;
}

// Whole-cell mask evaluated by one thread from the wrapped control points (same bricks): the fast
// value, and within 4e-5 of 1 the exact binary32 sequence. Bit s = a + 4 b + 16 c is sub-sample
// (a, b, c) of cell (i, j, k).
__device__ uint64_t particle_mask_serial(const float4* cw, int c0, int c1, int i, int j, int k, const Geom& g) {
  uint64_t m = 0ull;
  for (int s = 0; s < 64; ++s) {
    const float x = (float)i + (0.125f + 0.25f * (float)(s & 3)), y = (float)j + (0.125f + 0.25f * (float)((s >> 2) & 3)),
                z = (float)k + (0.125f + 0.25f * (float)(s >> 4));
    const float f = metaball_value(cw, c0, c1, x, y, z, g);
    const bool in = fabsf(f - 1.0f) > 4e-5f ? f >= 1.0f : metaball_exact(cw, c0, c1, x, y, z, g) >= 1.0f;
    if (in) m |= 1ull << s;
  }
  return m;
}

__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Two control points as the staging holds them: {x0, x1, y0, y1}, {z0, z1, k0, k1}. A particle with
// an odd number of points ends with a far point of weight 0.
struct CenterPair { float4 xy, zk; };
__device__ __forceinline__ CenterPair load_pair(const float4* cw, int q) { return CenterPair{cw[2 * q], cw[2 * q + 1]}; }
// Displacement x - c: with MI the minimum image on a periodic axis; without, the plain difference
// (points staged at the brick's nearest image, valid for every point of the brick).
template <bool MI>
__device__ __forceinline__ float disp(float x, float c, int a, const Geom& g) {
  return MI ? min_image_rn(x - c, (float)g.n[a], g.wall[a]) : x - c;
}
// acc + k0 / r0 + k1 / r1 with one reciprocal (the reciprocal unit is a quarter as wide as the
// multiply-add pipe): r0 = 0 gives infinity, r0 = r1 = 0 NaN, which callers send to the exact test.
__device__ __forceinline__ float add_quotients(float acc, float k0, float r0, float k1, float r1) {
  return fmaf(fmaf(k0, r1, k1 * r0), fast_rcp(r0 * r1), acc);
}

// Bounds of Eq. 3 over the ball of radius h1 about (x, y, z), and with TWO its upper bound over radius
// h2 as well, from the staged pairs q0 .. q1 - 1.
struct Bound2 { float fmax1, fmin1, fmax2; };
template <bool MI, bool TWO>
__device__ __forceinline__ Bound2 pair_bound(const float4* cw, int q0, int q1, float x, float y, float z, float h1,
                                             float h2, const Geom& g) {
  Bound2 b{0.0f, 0.0f, 0.0f};
  for (int q = q0; q < q1; ++q) {
    const CenterPair c = load_pair(cw, q);
    const float dx0 = disp<MI>(x, c.xy.x, 0, g), dx1 = disp<MI>(x, c.xy.y, 0, g), dy0 = disp<MI>(y, c.xy.z, 1, g),
                dy1 = disp<MI>(y, c.xy.w, 1, g), dz0 = disp<MI>(z, c.zk.x, 2, g), dz1 = disp<MI>(z, c.zk.y, 2, g);
    const float s0 = dx0 * dx0 + dy0 * dy0 + dz0 * dz0, s1 = dx1 * dx1 + dy1 * dy1 + dz1 * dz1;
    const float r0 = s0 * rsqrtf(fmaxf(s0, 1e-30f)), r1 = s1 * rsqrtf(fmaxf(s1, 1e-30f));
    const float a0 = fmaxf(r0 - h1, 1e-9f), a1 = fmaxf(r1 - h1, 1e-9f), b0 = r0 + h1, b1 = r1 + h1;
    b.fmax1 = add_quotients(b.fmax1, c.zk.z, a0 * a0, c.zk.w, a1 * a1);
    b.fmin1 = add_quotients(b.fmin1, c.zk.z, b0 * b0, c.zk.w, b1 * b1);
    if (TWO) {
      const float d0 = fmaxf(r0 - h2, 1e-9f), d1 = fmaxf(r1 - h2, 1e-9f);
      b.fmax2 = add_quotients(b.fmax2, c.zk.z, d0 * d0, c.zk.w, d1 * d1);
    }
  }
  return b;
}

// The sub-samples (x, y, z) and (x, y, z + 1/2) of one lane in one pass over the staged pairs: fast
// values (error ~1e-6 relative); within 4e-5 of 1, or not a number, the exact binary32 sequence
// shared with the CPU oracle decides, on the original wrapped points e0 .. e1 - 1.
template <bool MI>
__device__ __forceinline__ void subsample_pair(const float4* cw, int q0, int q1, const float4* cw_exact, int e0, int e1,
                                               float x, float y, float z, const Geom& g, bool& in_lo, bool& in_hi) {
  const float zh = z + 0.5f;
  float flo = 0.0f, fhi = 0.0f;
  for (int q = q0; q < q1; ++q) {
    const CenterPair c = load_pair(cw, q);
    const float dx0 = disp<MI>(x, c.xy.x, 0, g), dx1 = disp<MI>(x, c.xy.y, 0, g), dy0 = disp<MI>(y, c.xy.z, 1, g),
                dy1 = disp<MI>(y, c.xy.w, 1, g);
    const float l0 = disp<MI>(z, c.zk.x, 2, g), l1 = disp<MI>(z, c.zk.y, 2, g), h0 = disp<MI>(zh, c.zk.x, 2, g),
                h1 = disp<MI>(zh, c.zk.y, 2, g);
    const float r0 = dx0 * dx0 + dy0 * dy0, r1 = dx1 * dx1 + dy1 * dy1;
    flo = add_quotients(flo, c.zk.z, r0 + l0 * l0, c.zk.w, r1 + l1 * l1);
    fhi = add_quotients(fhi, c.zk.z, r0 + h0 * h0, c.zk.w, r1 + h1 * h1);
  }
  in_lo = fabsf(flo - 1.0f) > 4e-5f ? flo >= 1.0f : metaball_exact(cw_exact, e0, e1, x, y, z, g) >= 1.0f;
  in_hi = fabsf(fhi - 1.0f) > 4e-5f ? fhi >= 1.0f : metaball_exact(cw_exact, e0, e1, x, y, zh, g) >= 1.0f;
}

// Is the point (x, y, z) inside, likewise.
template <bool MI>
__device__ __forceinline__ bool point_inside(const float4* cw, int q0, int q1, const float4* cw_exact, int e0, int e1,
                                             float x, float y, float z, const Geom& g) {
  float f = 0.0f;
  for (int q = q0; q < q1; ++q) {
    const CenterPair c = load_pair(cw, q);
    const float dx0 = disp<MI>(x, c.xy.x, 0, g), dx1 = disp<MI>(x, c.xy.y, 0, g), dy0 = disp<MI>(y, c.xy.z, 1, g),
                dy1 = disp<MI>(y, c.xy.w, 1, g), dz0 = disp<MI>(z, c.zk.x, 2, g), dz1 = disp<MI>(z, c.zk.y, 2, g);
    f = add_quotients(f, c.zk.z, dx0 * dx0 + dy0 * dy0 + dz0 * dz0, c.zk.w, dx1 * dx1 + dy1 * dy1 + dz1 * dz1);
  }
  return fabsf(f - 1.0f) > 4e-5f ? f >= 1.0f : metaball_exact(cw_exact, e0, e1, x, y, z, g) >= 1.0f;
}

constexpr int RW_WARPS = 8;        // warps (pieces in flight) per block
constexpr int RW_CENTERS = 192;    // control points one warp stages (even)
constexpr int RW_CAND = 8;         // candidates one warp stages (more: the unstaged path)
constexpr int RW_LISTED = 0xffff;  // marks a mini-brick whose cells are evaluated one by one

struct RasterWarp {
  float4 cw[RW_CENTERS];            // control point pairs at the brick's nearest image
  unsigned char mcls[RW_CAND][64];  // per candidate and mini-brick: class | walker bit << 2
  uint16_t val[64];                 // per mini-brick: the word of all its cells, or RW_LISTED
  unsigned char list[64];           // the mini-bricks whose cells are evaluated
  int p[RW_CAND], q0[RW_CAND], q1[RW_CAND], e0[RW_CAND], e1[RW_CAND];
};

// Pieces a brick is cut into, as a power of two: a brick's straddling cells are one warp's serial
// work (up to ~100 evaluations of 64 sub-samples, ~1 us each), so a list shorter than four per
// resident warp is spread over them: slices of 32, 16 or 8 mini-bricks, then parts that share out a
// slice's straddling mini-bricks down to one each. Every piece stages the candidates again, so
// longer lists keep whole bricks (256^3, 13175 bricks on 2432 warps: 183 us whole, 241 us in
// eighths; 96^3, 902 bricks: 75 us whole, 40 us in eighths).
__device__ __forceinline__ int raster_pieces_log2(uint32_t nlist, uint32_t warps) {
  int s = 0;
  while (s < 6 && (nlist << (s + 1)) <= 4u * warps) ++s;
  return s;
}

// One warp per piece of a brick of the raster list (pieces beyond one per warp from a work counter;
// no block barriers):
//  1. the brick's candidates and their control points (staged at the brick's nearest image) are
//     gathered by the lanes in parallel;
//  2. the slice's mini-bricks (2^3 cells): raster class per candidate (outside / inside /
//     straddling) and the walkers' mask bit (Eq. 3 may reach 1 within sqrt(3) + the walker step
//     margin). Cells of mini-bricks that no candidate straddles are filled at once;
//  3. the straddling mini-bricks, four (32 cells) per round: each lane bounds Eq. 3 over its cell; the
//     warp then evaluates every straddling (cell, candidate) pair together, two sub-samples per
//     lane, and the cell's lane folds the 64-bit mask in: count = popcount(OR of masks), owner =
//     the candidate with most sub-samples, lowest index on ties.
// All decisions use bounds with a 1e-3 margin and, within 4e-5 of f = 1, the exact binary32
// sequence shared with the CPU oracle, so counts and owners equal the oracle's bit for bit.
// With nodes the words are the IBB coupling's node classes instead (0, or 1 + the lowest particle
// holding the cell centre): step 3 then tests one point per cell of the straddling mini-bricks.
// (A pass of its own over every cell of every brick took 119 us at 256^3, one chain of dependent
// loads per block; here the candidates are staged and most cells settled, and the raster runs
// beside the update.)
struct RasterArgs {
  Geom g;
  ParticleSet ps;
  BrickSet bs;
  uint16_t* solid;
  unsigned long long* status;
  uint16_t* nodes;
};

// CLASSES: node classes instead of counts. WHOLE: a list that keeps whole bricks (plog = 0); the
// arithmetic of slices and parts then falls away.
template <bool CLASSES, bool WHOLE>
__device__ __forceinline__ void raster_list(const RasterArgs& A, RasterWarp* s_rw, int blk, uint32_t warps,
                                            uint32_t nlist, int plog) {
  const Geom g = A.g;
  const ParticleSet ps = A.ps;
  const BrickSet bs = A.bs;
  uint16_t* __restrict__ solid = CLASSES ? A.nodes : A.solid;   // the words of cells written
  unsigned long long* __restrict__ status = A.status;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  RasterWarp& W = s_rw[wib];
  const uint32_t nbrick = (uint32_t)g.nb[0] * g.nb[1] * g.nb[2];
  if (WHOLE) plog = 0;
  const int slog = min(plog, 3), parts = 1 << (plog - slog);
  const uint32_t units = nlist << plog;
  const int K = 64 >> slog;          // mini-bricks per slice: 64, 32, 16 or 8
  const int rows_y = K >= 16 ? 8 : 4;   // cell rows of a slice along y
  unsigned long long queued = 0;
  // this lane's sub-samples: offsets within the cell (z and z + 1/2)
  const float ax = 0.125f + 0.25f * (float)(lane & 3), ay = 0.125f + 0.25f * (float)((lane >> 2) & 3),
              az = 0.125f + 0.25f * (float)(lane >> 4);
  // the first piece by warp index, further ones from a shared counter (bword[nbrick + 1], zero
  // after the brick pass): their cost ranges from a few bound tests to ~100 straddling cells, and
  // a fixed assignment left a long tail
  for (uint32_t u = (uint32_t)blk * RW_WARPS + wib; u < units;) {
    const int slice = (int)(u & ((1u << slog) - 1u)), part = (int)(u >> slog) & (parts - 1);
    const uint32_t b = (uint32_t)bs.rlist[u >> plog];
    const int mb0 = slice * K;
    const int bi = b % g.nb[0], bj = (b / g.nb[0]) % g.nb[1], bk = b / (g.nb[0] * g.nb[1]);
    const uint32_t nc = bs.bword[b] & 0xffffu;
    const bool over = nc > MAXC;
    // 1. candidates, in parallel over lanes; offsets of their control point pairs by a warp scan
    int p = -1, cnt = 0, g0 = 0;
    if (!over && lane < (int)nc) {
      const uint16_t cid = bs.bcand[b * MAXC + lane];
      if (cid & 0x8000) {
        p = cid & 0x7fff;
        g0 = ps.desc[p].c0;
        cnt = ps.desc[p].c1 - g0;
      }
    }
    const unsigned rel = __ballot_sync(full, p >= 0);
    const int n = __popc(rel);
    const int npair = (cnt + 1) >> 1;
    int incl = npair;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(full, incl, o);
      if (lane >= o) incl += v;
    }
    const int tot = __shfl_sync(full, incl, 31);
    const bool staged = !over && n <= RW_CAND && 2 * tot <= RW_CENTERS;
    if (staged && p >= 0) {
      const int slot = __popc(rel & ((1u << lane) - 1u));
      W.p[slot] = p; W.q0[slot] = incl - npair; W.q1[slot] = incl; W.e0[slot] = g0; W.e1[slot] = g0 + cnt;
    }
    __syncwarp();
    bool mi = true;
    int nlisted = 0;
    if (staged) {
      const float bc[3] = {(float)(bi * BRICK) + 4.0f, (float)(bj * BRICK) + 4.0f, (float)(bk * BRICK) + 4.0f};
      const float H = 6.0f + ps.walk_margin;
      bool near_half = false;
      for (int m = 0; m < n; ++m) {
        const int len = W.e1[m] - W.e0[m], slots = 2 * (W.q1[m] - W.q0[m]);
        for (int i = lane; i < slots; i += 32) {
          float v[3] = {bc[0] + 1e4f, bc[1], bc[2]}, k = 0.0f;   // the far point of an odd count
          if (i < len) {
            const float4 cc = bs.cworld[W.e0[m] + i];
            v[0] = cc.x; v[1] = cc.y; v[2] = cc.z; k = cc.w;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              if (g.wall[a]) continue;
              const float na = (float)g.n[a];
              const float d = v[a] - bc[a];
              if (d > 0.5f * na) v[a] -= na; else if (d < -0.5f * na) v[a] += na;
              if (fabsf(v[a] - bc[a]) > 0.5f * na - H) near_half = true;
            }
          }
          float* w = reinterpret_cast<float*>(W.cw + 2 * (W.q0[m] + (i >> 1))) + (i & 1);
          w[0] = v[0]; w[2] = v[1]; w[4] = v[2]; w[6] = k;
        }
      }
      mi = __any_sync(full, near_half);
      __syncwarp();
      // 2. mini-bricks: raster class and walker bit per candidate
      const float hw = 1.7320508f + ps.walk_margin;
      for (int pr = lane; pr < K * n; pr += 32) {
        const int mb = mb0 + (pr & (K - 1)), m = pr >> (6 - slog);
        const float xm = (float)(bi * BRICK + 2 * (mb & 3)) + 1.0f, ym = (float)(bj * BRICK + 2 * ((mb >> 2) & 3)) + 1.0f,
                    zm = (float)(bk * BRICK + 2 * (mb >> 4)) + 1.0f;
        const Bound2 b2 = mi ? pair_bound<true, true>(W.cw, W.q0[m], W.q1[m], xm, ym, zm, 1.5155444f, hw, g)
                             : pair_bound<false, true>(W.cw, W.q0[m], W.q1[m], xm, ym, zm, 1.5155444f, hw, g);
        const int cls = b2.fmax1 < 0.999f ? 0 : (b2.fmin1 > 1.001f ? 1 : 2);
        W.mcls[m][mb] = (unsigned char)(cls | (b2.fmax2 >= 0.999f ? 4 : 0));
      }
      __syncwarp();
      // per mini-brick: the walkers' bit, and its cells' common solid word or a place in the list
      unsigned wm[2] = {0u, 0u};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = lane + 32 * h, mb = mb0 + k;
        bool need = false, listed = false;
        if (k < K) {
          int own = 0x7fffffff;
          for (int m = 0; m < n; ++m) {
            const int mc = W.mcls[m][mb];
            need |= (mc & 4) != 0;
            listed |= (mc & 3) == 2;
            if ((mc & 3) == 1) own = min(own, W.p[m]);
          }
          listed = listed && bi * BRICK + 2 * (mb & 3) < g.n[0] && bj * BRICK + 2 * ((mb >> 2) & 3) < g.n[1] &&
                   bk * BRICK + 2 * (mb >> 4) < g.n[2];
          W.val[mb] = listed ? (uint16_t)RW_LISTED : own == 0x7fffffff ? (uint16_t)0
                      : CLASSES               ? (uint16_t)(1 + own)
                                              : (uint16_t)(64 | (own << 7));
        }
        wm[h] = __ballot_sync(full, need);
        const unsigned bl = __ballot_sync(full, listed);
        if (listed) W.list[nlisted + __popc(bl & ((1u << lane) - 1u))] = (unsigned char)mb;
        nlisted += __popc(bl);
      }
      if (lane == 0 && part == 0) {   // the slice's K mask bits
        unsigned char* dst = reinterpret_cast<unsigned char*>(bs.wmask + b) + slice * (K >> 3);
        if (slog == 0) *reinterpret_cast<unsigned long long*>(dst) = ((unsigned long long)wm[1] << 32) | wm[0];
        else if (slog == 1) *reinterpret_cast<uint32_t*>(dst) = wm[0];
        else if (slog == 2) *reinterpret_cast<uint16_t*>(dst) = (uint16_t)wm[0];
        else *dst = (unsigned char)wm[0];
      }
      __syncwarp();
      // cells of the other mini-bricks: two cells of one mini-brick (x, x + 1) per lane
      if (part == 0) {
        const int ly0 = 2 * ((mb0 >> 2) & 3), lz0 = 2 * (mb0 >> 4);
        for (int t = lane; t < 4 * K; t += 32) {
          const int r = t >> 2, ly = ly0 + (r & (rows_y - 1)), lz = lz0 + r / rows_y;
          const uint16_t v = W.val[(t & 3) + 4 * (ly >> 1) + 16 * (lz >> 1)];
          const int i = bi * BRICK + 2 * (t & 3), j = bj * BRICK + ly, k = bk * BRICK + lz;
          if (v == RW_LISTED || i >= g.n[0] || j >= g.n[1] || k >= g.n[2]) continue;
          const uint32_t cell = ((uint32_t)k * g.n[1] + j) * g.n[0] + i;
          if (i + 1 < g.n[0] && !(cell & 1u)) {
            *reinterpret_cast<uint32_t*>(solid + cell) = (uint32_t)v | ((uint32_t)v << 16);
          } else {
            solid[cell] = v;
            if (i + 1 < g.n[0]) solid[cell + 1] = v;
          }
        }
      }
    } else {
      if (lane == 0 && slice == 0 && part == 0) {
        bs.wmask[b] = ~0ull;   // every walker of this brick is tested
        if (over) atomicAdd(&status[ST_BRICK_OVERFLOW], 1ull);
      }
      for (int k = lane; k < K; k += 32) W.list[k] = (unsigned char)(mb0 + k);
      nlisted = K;
      __syncwarp();
    }
    // 3. cells of this part's listed mini-bricks, 32 per round (lane: mini-brick lane / 8, its cell
    // lane & 7)
    for (int r = part; r < nlisted; r += 4 * parts) {
      const int at = r + (lane >> 3) * parts;
      const bool have = at < nlisted;
      const int mb = have ? W.list[at] : 0;
      const int lx = 2 * (mb & 3) + (lane & 1), ly = 2 * ((mb >> 2) & 3) + ((lane >> 1) & 1), lz = 2 * (mb >> 4) + ((lane >> 2) & 1);
      const int i = bi * BRICK + lx, j = bj * BRICK + ly, k = bk * BRICK + lz;
      const bool in_dom = have && i < g.n[0] && j < g.n[1] && k < g.n[2];
      const float xi = (float)i, yj = (float)j, zk = (float)k;
      if (CLASSES) {
        const float xs = xi + 0.5f, ys = yj + 0.5f, zs = zk + 0.5f;
        int own = 0x7fffffff;
        for (int m = 0; in_dom && m < (staged ? n : over ? ps.P : (int)nc); ++m) {
          const int pp = staged ? W.p[m] : over ? m : (bs.bcand[b * MAXC + m] & 0x7fff);
          if (pp > own) continue;
          bool in;
          if (staged) {
            const int cls = W.mcls[m][mb] & 3;
            in = cls == 1 || (cls == 2 && (mi ? point_inside<true>(W.cw, W.q0[m], W.q1[m], bs.cworld, W.e0[m], W.e1[m], xs, ys, zs, g)
                                              : point_inside<false>(W.cw, W.q0[m], W.q1[m], bs.cworld, W.e0[m], W.e1[m], xs, ys, zs, g)));
          } else {
            in = inside_exact(bs.cworld, ps.desc[pp].c0, ps.desc[pp].c1, xs, ys, zs, g);
          }
          if (in) own = pp;
        }
        if (in_dom) solid[((uint32_t)k * g.n[1] + j) * g.n[0] + i] = own == 0x7fffffff ? (uint16_t)0 : (uint16_t)(1 + own);
        continue;
      }
      uint64_t any = 0ull;
      int best = 0, bestp = -1;
      unsigned pend = 0u;
      const int ncand = staged ? n : (over ? ps.P : (int)nc);
      for (int m = 0; in_dom && m < ncand; ++m) {
        int pp;
        uint64_t mk;
        if (staged) {
          pp = W.p[m];
          const int cls = W.mcls[m][mb] & 3;
          if (cls == 0) continue;
          if (cls == 2) {
            const Bound2 cb = mi ? pair_bound<true, false>(W.cw, W.q0[m], W.q1[m], xi + 0.5f, yj + 0.5f, zk + 0.5f, 0.649519053f, 0.0f, g)
                                 : pair_bound<false, false>(W.cw, W.q0[m], W.q1[m], xi + 0.5f, yj + 0.5f, zk + 0.5f, 0.649519053f, 0.0f, g);
            if (cb.fmax1 < 0.999f) continue;
            if (!(cb.fmin1 > 1.001f)) {
              pend |= 1u << m;   // the whole warp evaluates it below
              continue;
            }
          }
          mk = ~0ull;
        } else {
          if (over) pp = m;
          else {
            const uint16_t cid = bs.bcand[b * MAXC + m];
            if (!(cid & 0x8000)) continue;
            pp = cid & 0x7fff;
          }
          const int c0 = ps.desc[pp].c0, c1 = ps.desc[pp].c1;
          const CellBound cb = bound_at(bs.cworld, c0, c1, xi + 0.5f, yj + 0.5f, zk + 0.5f, 0.649519053f, g);
          if (cb.fmax < 0.999f) continue;
          mk = cb.fmin > 1.001f ? ~0ull : particle_mask_serial(bs.cworld, c0, c1, i, j, k, g);
        }
        const int np = __popcll(mk);
        any |= mk;
        if (np > 0 && (np > best || (np == best && pp < bestp))) { best = np; bestp = pp; }
      }
      // the warp evaluates each straddling (cell, candidate) pair: 2 x 32 sub-samples
      for (int m = 0; staged && m < n; ++m) {
        unsigned lanes_p = __ballot_sync(full, (pend >> m) & 1u);
        queued += __popc(lanes_p);
        while (lanes_p) {
          const int src = __ffs(lanes_p) - 1;
          lanes_p &= lanes_p - 1u;
          const float sx = __shfl_sync(full, xi, src) + ax, sy = __shfl_sync(full, yj, src) + ay,
                      sz = __shfl_sync(full, zk, src) + az;
          bool in_lo, in_hi;
          if (mi) subsample_pair<true>(W.cw, W.q0[m], W.q1[m], bs.cworld, W.e0[m], W.e1[m], sx, sy, sz, g, in_lo, in_hi);
          else subsample_pair<false>(W.cw, W.q0[m], W.q1[m], bs.cworld, W.e0[m], W.e1[m], sx, sy, sz, g, in_lo, in_hi);
          const unsigned blo = __ballot_sync(full, in_lo);
          const unsigned bhi = __ballot_sync(full, in_hi);
          if (lane == src) {
            any |= ((uint64_t)bhi << 32) | blo;
            const int np = __popc(blo) + __popc(bhi);
            const int pp = W.p[m];
            if (np > 0 && (np > best || (np == best && pp < bestp))) { best = np; bestp = pp; }
          }
        }
      }
      if (in_dom) {
        const int count = __popcll(any);
        const uint32_t cell = ((uint32_t)k * g.n[1] + j) * g.n[0] + i;
        solid[cell] = count > 0 ? (uint16_t)(count | (bestp << 7)) : (uint16_t)0;
      }
    }
    __syncwarp();
    if (lane == 0) u = warps + atomicAdd(&bs.bword[nbrick + 1], 1u);
    u = __shfl_sync(full, u, 0);
  }
  if (lane == 0 && queued) atomicAdd(&status[ST_RASTER_QUEUED], queued);
}

__device__ __forceinline__ uint32_t raster_list_length(const RasterArgs& A) {
  return A.bs.bword[(uint32_t)A.g.nb[0] * A.g.nb[1] * A.g.nb[2]];
}

// Three forms, each compiled by itself: run-time slices and the class switch inside one body cost every
// brick of a long list (256^3, 13 k bricks: 209 us, 183 apart; 384^3, 27 k: 377 and 317 us). The pieces'
// form comes first in the code: behind the other it took 10 to 15% longer (96^3 and below).
template <bool CLASSES>
__global__ void __launch_bounds__(256, 4) raster_kernel(const RasterArgs a) {
  asm volatile("griddepcontrol.launch_dependents;");   // the LBM update may fill the rest of each SM now
  __shared__ RasterWarp s_rw[RW_WARPS];
  const uint32_t nlist = raster_list_length(a), warps = gridDim.x * RW_WARPS;
  const int plog = CLASSES ? 0 : raster_pieces_log2(nlist, warps);   // node classes are a few rounds per brick
  if (!CLASSES && plog > 0) raster_list<CLASSES, false>(a, s_rw, blockIdx.x, warps, nlist, plog);
  else raster_list<CLASSES, true>(a, s_rw, blockIdx.x, warps, nlist, 0);
}
// The pieces' form for every domain (small ones, whose lists are short), with more registers, since
// the arguments come from memory rather than the constant bank.
__global__ void __launch_bounds__(256, 3) raster_batched(const RasterArgs* __restrict__ args,
                                                         const BlockMap* __restrict__ map) {
  asm volatile("griddepcontrol.launch_dependents;");   // as raster_kernel
  __shared__ RasterWarp s_rw[RW_WARPS];
  const BlockMap m = map[blockIdx.x];
  const RasterArgs& A = args[m.domain];
  const uint32_t nlist = raster_list_length(A), warps = (uint32_t)m.blocks * RW_WARPS;
  raster_list<false, false>(A, s_rw, m.block, warps, nlist, raster_pieces_log2(nlist, warps));
}

// two blocks per SM: the raster runs beside the LBM, which takes the rest of each SM (four
// blocks per SM held every register file and left the LBM to start only as they finished;
// one block per SM made the raster itself the longer branch)
int raster_grid(int nsm) { return nsm * 2; }
void launch_raster(const Geom& g, const ParticleSet& ps, BrickSet bs, uint16_t* solid,
                   unsigned long long* status, int nsm, cudaStream_t st, uint16_t* nodes) {
  if (ps.P == 0) return;
  const RasterArgs a{g, ps, bs, solid, status, nodes};
  if (nodes) raster_kernel<true><<<raster_grid(nsm), RW_WARPS * 32, 0, st>>>(a);
  else raster_kernel<false><<<raster_grid(nsm), RW_WARPS * 32, 0, st>>>(a);
}
size_t raster_args_size() { return sizeof(RasterArgs); }
void raster_args(void* dst, const Geom& g, const ParticleSet& ps, BrickSet bs, uint16_t* solid,
                 unsigned long long* status) {
  *static_cast<RasterArgs*>(dst) = RasterArgs{g, ps, bs, solid, status, nullptr};
}
void launch_raster_batched(const void* args, const BlockMap* map, int nblocks, cudaStream_t st) {
  if (nblocks > 0) raster_batched<<<nblocks, RW_WARPS * 32, 0, st>>>(static_cast<const RasterArgs*>(args), map);
}

// ------------------------------------------------------------------------------------------
// Initial state, checkpoint load and read-back helpers
// ------------------------------------------------------------------------------------------
template <int Q, int STORE>
__global__ void init_pop_kernel(Geom g, void* f_, double rho0_d, double ux_d, double uy_d, double uz_d,
                                float* u) {
  using L = Lat<Q>;
  using S = Store<STORE>;
  using R = typename S::R;
  typename S::T* f = (typename S::T*)f_;
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const R rho0 = (R)rho0_d, ux = (R)ux_d, uy = (R)uy_d, uz = (R)uz_d;
  const R uu = ux * ux + uy * uy + uz * uz;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const R eu = L::e(i, 0) * ux + L::e(i, 1) * uy + L::e(i, 2) * uz;
    const R dev = R(3) * eu + R(4.5) * eu * eu - R(1.5) * uu;
    const R w = L::template wt<R>(i);
    const R v = S::shifted ? w * rho0 * dev : w * rho0 * (R(1) + dev);
    S::st(f + (size_t)i * g.ncell_pad + c, v);
  }
  reinterpret_cast<float4*>(u)[c] = make_float4((float)ux, (float)uy, (float)uz, (float)rho0);
}

template <int Q, int STORE>
__global__ void pop_f64_kernel(Geom g, const void* f_, double rho0, double* out) {
  using L = Lat<Q>;
  using S = Store<STORE>;
  const typename S::T* f = (const typename S::T*)f_;
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const double v = (double)S::ld(f + (size_t)i * g.ncell_pad + c);
    out[(size_t)i * g.ncell + c] = S::shifted ? v + L::template wt<double>(i) * rho0 : v;
  }
}

template <int Q, int STORE>
__global__ void load_pop_kernel(Geom g, const double* in, double rho0, void* f_) {
  using L = Lat<Q>;
  using S = Store<STORE>;
  using R = typename S::R;
  typename S::T* f = (typename S::T*)f_;
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const double v = in[(size_t)i * g.ncell + c];
    S::st(f + (size_t)i * g.ncell_pad + c, (R)(S::shifted ? v - L::template wt<double>(i) * rho0 : v));
  }
}

template <int Q, int STORE>
__global__ void density_kernel(Geom g, const void* f_, double rho0, float* out) {
  using S = Store<STORE>;
  using R = typename S::R;
  const typename S::T* f = (const typename S::T*)f_;
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  R s = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) s += S::ld(f + (size_t)i * g.ncell_pad + c);
  out[c] = (float)(S::shifted ? (R)rho0 + s : s);
}

#define RWMI_DISPATCH(q, storage, KERNEL, ...)                                   \
  do {                                                                           \
    const dim3 grid_((g.ncell + 255) / 256);                                     \
    if ((q) == 15) {                                                             \
      if ((storage) == 0) KERNEL<15, 0><<<grid_, 256, 0, st>>>(__VA_ARGS__);     \
      else if ((storage) == 1) KERNEL<15, 1><<<grid_, 256, 0, st>>>(__VA_ARGS__);\
      else if ((storage) == 2) KERNEL<15, 2><<<grid_, 256, 0, st>>>(__VA_ARGS__);\
      else KERNEL<15, 3><<<grid_, 256, 0, st>>>(__VA_ARGS__);                    \
    } else {                                                                     \
      if ((storage) == 0) KERNEL<19, 0><<<grid_, 256, 0, st>>>(__VA_ARGS__);     \
      else if ((storage) == 1) KERNEL<19, 1><<<grid_, 256, 0, st>>>(__VA_ARGS__);\
      else if ((storage) == 2) KERNEL<19, 2><<<grid_, 256, 0, st>>>(__VA_ARGS__);\
      else KERNEL<19, 3><<<grid_, 256, 0, st>>>(__VA_ARGS__);                    \
    }                                                                            \
  } while (0)

void launch_init_populations(int q, int storage, const Geom& g, void* f, double rho0,
                             const double u0[3], float* u, cudaStream_t st) {
  RWMI_DISPATCH(q, storage, init_pop_kernel, g, f, rho0, u0[0], u0[1], u0[2], u);
}
void launch_populations_f64(int q, int storage, const Geom& g, const void* f, double rho0,
                            double* out, cudaStream_t st) {
  RWMI_DISPATCH(q, storage, pop_f64_kernel, g, f, rho0, out);
}
void launch_load_populations(int q, int storage, const Geom& g, const double* in, double rho0,
                             void* f, cudaStream_t st) {
  RWMI_DISPATCH(q, storage, load_pop_kernel, g, in, rho0, f);
}
void launch_density(int q, int storage, const Geom& g, const void* f, double rho0, float* out,
                    cudaStream_t st) {
  RWMI_DISPATCH(q, storage, density_kernel, g, f, rho0, out);
}

// IBB node classes (Section 2.4.3) of every cell: a cell centre is solid when Eq. 3 of some particle
// reaches 1 there (binary32, the CPU oracle's operation order), owned by the lowest such particle
// index. Only cells of flagged bricks can be solid. For the classes of t - 1 at set-up, and for
// runs without the coupling; in a step the raster writes the classes of flagged bricks and refill_kernel the rest. Brick-major: block 2 b + h takes
// half h (z rows 4 h .. 4 h + 3) of brick b.
__global__ void __launch_bounds__(256) node_kernel(Geom g, ParticleSet ps, BrickSet bs, uint16_t* __restrict__ cur) {
  const uint32_t b = blockIdx.x >> 1;
  const uint32_t l = threadIdx.x + ((blockIdx.x & 1u) << 8);
  const uint32_t bi = b % (uint32_t)g.nb[0], bj = (b / (uint32_t)g.nb[0]) % (uint32_t)g.nb[1],
                 bk = b / ((uint32_t)g.nb[0] * (uint32_t)g.nb[1]);
  const uint32_t x = bi * BRICK + (l & 7u), y = bj * BRICK + ((l >> 3) & 7u), z = bk * BRICK + (l >> 6);
  if (x >= (uint32_t)g.n[0] || y >= (uint32_t)g.n[1] || z >= (uint32_t)g.n[2]) return;
  const uint32_t c = (z * (uint32_t)g.n[1] + y) * (uint32_t)g.n[0] + x;
  const uint32_t w = bs.bword[b];
  int node = 0;
  if (w >> 16) {
    const float xs = (float)x + 0.5f, ys = (float)y + 0.5f, zs = (float)z + 0.5f;
    const uint32_t nc = w & 0xffffu;
    if (nc > MAXC) {
      for (int p = 0; p < ps.P && node == 0; ++p)
        if (inside_exact(bs.cworld, ps.desc[p].c0, ps.desc[p].c1, xs, ys, zs, g)) node = p + 1;
    } else {
      int best = 0x7fffffff;
      for (uint32_t m = 0; m < nc; ++m) {
        const int p = bs.bcand[b * MAXC + m] & 0x7fff;
        if (p < best && inside_exact(bs.cworld, ps.desc[p].c0, ps.desc[p].c1, xs, ys, zs, g)) best = p;
      }
      if (best != 0x7fffffff) node = best + 1;
    }
  }
  cur[c] = (uint16_t)node;
}

// The classes a step's raster left in nodes, with 0 in the bricks it did not write (read-back).
__global__ void __launch_bounds__(256) read_nodes_kernel(Geom g, BrickSet bs, const uint16_t* __restrict__ nodes,
                                                         uint16_t* __restrict__ out) {
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const uint32_t z = fast_div(c, g.mxy, g.sxy), rem = c - z * g.nxy, y = fast_div(rem, g.mx, g.sx), x = rem - y * (uint32_t)g.n[0];
  const bool held = bs.bword[((z >> 3) * (uint32_t)g.nb[1] + (y >> 3)) * (uint32_t)g.nb[0] + (x >> 3)] >> 16;
  out[c] = held ? nodes[c] : (uint16_t)0;
}

void launch_read_nodes(const Geom& g, BrickSet bs, const uint16_t* nodes, uint16_t* out, cudaStream_t st) {
  read_nodes_kernel<<<(g.ncell + 255) / 256, 256, 0, st>>>(g, bs, nodes, out);
}

void launch_nodes(const Geom& g, const ParticleSet& ps, BrickSet bs, uint16_t* cur, cudaStream_t st) {
  node_kernel<<<2u * (uint32_t)g.nb[0] * (uint32_t)g.nb[1] * (uint32_t)g.nb[2], 256, 0, st>>>(g, ps, bs, cur);
}

// Ahead of the IBB links of a step: cells of bricks that hold no particle now are fluid (the raster
// wrote the others), and a node solid in prev and fluid in cur gets G^eq(rho0, u_new) with u_new its
// former particle's rigid velocity (Eq. 27). One thread per 8 cells of a row (16 bytes of classes)
// where the rows are aligned, else per cell: a stream over prev and the empty bricks of cur.
template <int Q, int STORE, int CELLS>
__global__ void __launch_bounds__(256) refill_kernel(Geom g, BrickSet bs, const uint16_t* __restrict__ prev,
                                                     uint16_t* __restrict__ cur, void* f_, double rho0_d) {
  using L = Lat<Q>;
  using S = Store<STORE>;
  using R = typename S::R;
  const uint32_t c0 = (blockIdx.x * blockDim.x + threadIdx.x) * CELLS;
  if (c0 >= g.ncell) return;
  const uint32_t z = fast_div(c0, g.mxy, g.sxy), rem = c0 - z * g.nxy, y = fast_div(rem, g.mx, g.sx),
                 x0 = rem - y * (uint32_t)g.n[0];
  const bool held = bs.bword[((z >> 3) * (uint32_t)g.nb[1] + (y >> 3)) * (uint32_t)g.nb[0] + (x0 >> 3)] >> 16;
  if constexpr (CELLS == 8) {
    const uint4 p8 = *reinterpret_cast<const uint4*>(prev + c0);
    if (!held) *reinterpret_cast<uint4*>(cur + c0) = make_uint4(0u, 0u, 0u, 0u);
    if (!(p8.x | p8.y | p8.z | p8.w)) return;
  } else {
    if (!held) cur[c0] = 0;
  }
  for (uint32_t k = 0; k < CELLS; ++k) {
    const uint32_t c = c0 + k, was = prev[c];
    if (was == 0 || cur[c] != 0) continue;
    R un[3];
    rigid_velocity<R>(g, bs.pose, bs.posed, (int)was - 1, (R)(x0 + k) + R(0.5), (R)y + R(0.5), (R)z + R(0.5), un);
    const R rho0 = (R)rho0_d, uu = un[0] * un[0] + un[1] * un[1] + un[2] * un[2];
    typename S::T* f = (typename S::T*)f_;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const R eu = (R)L::e(i, 0) * un[0] + (R)L::e(i, 1) * un[1] + (R)L::e(i, 2) * un[2];
      const R dev = R(3) * eu + R(4.5) * eu * eu - R(1.5) * uu;
      const R wi = L::template wt<R>(i);
      S::st(f + (size_t)i * g.ncell_pad + c, S::shifted ? wi * rho0 * dev : wi * rho0 * (R(1) + dev));
    }
  }
}

void launch_refill(int q, int storage, const Geom& g, BrickSet bs, const uint16_t* prev, uint16_t* cur, void* f,
                   double rho0, cudaStream_t st) {
  const bool rows = g.n[0] % 8 == 0;   // every row then starts on a 16-byte boundary
  const uint32_t threads = rows ? g.ncell / 8 : g.ncell, blocks = (threads + 255) / 256;
#define RWMI_REFILL(QQ, SS)                                                                              \
  do {                                                                                                 \
    if (rows) refill_kernel<QQ, SS, 8><<<blocks, 256, 0, st>>>(g, bs, prev, cur, f, rho0);               \
    else refill_kernel<QQ, SS, 1><<<blocks, 256, 0, st>>>(g, bs, prev, cur, f, rho0);                    \
  } while (0)
  // IBB is built for binary32-shifted and binary64 storage
  if (q == 15) { if (storage == 3) RWMI_REFILL(15, 3); else RWMI_REFILL(15, 1); }
  else { if (storage == 3) RWMI_REFILL(19, 3); else RWMI_REFILL(19, 1); }
#undef RWMI_REFILL
}

__global__ void unpack_solid_kernel(Geom g, const uint16_t* solid, const uint32_t* bword,
                                    int32_t* count, int32_t* owner) {
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const uint32_t z = c / g.nxy, rem = c - z * g.nxy, y = rem / g.n[0], x = rem - y * g.n[0];
  const uint32_t b = ((z >> 3) * (uint32_t)g.nb[1] + (y >> 3)) * (uint32_t)g.nb[0] + (x >> 3);
  uint16_t sw = 0;
  if (bword[b] >> 16) sw = solid[c];
  const int n = sw & 0x7f;
  count[c] = n;
  owner[c] = n ? (sw >> 7) : -1;
}

void launch_unpack_solid(const Geom& g, const uint16_t* solid, const uint32_t* bword,
                         int32_t* count, int32_t* owner, cudaStream_t st) {
  unpack_solid_kernel<<<(g.ncell + 255) / 256, 256, 0, st>>>(g, solid, bword, count, owner);
}

__global__ void velocity_aos_kernel(Geom g, const float* u, float* out) {
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const float4 v = reinterpret_cast<const float4*>(u)[c];
  out[3 * (size_t)c] = v.x;
  out[3 * (size_t)c + 1] = v.y;
  out[3 * (size_t)c + 2] = v.z;
}

void launch_velocity_aos(const Geom& g, const float* u, float* out, cudaStream_t st) {
  velocity_aos_kernel<<<(g.ncell + 255) / 256, 256, 0, st>>>(g, u, out);
}

}  // namespace rwmi
