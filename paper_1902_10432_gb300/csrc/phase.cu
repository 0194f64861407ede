// Solid-body kernels of the capillary-bridge step (Sec. 3.1 and 3.3 of arXiv:1902.10432).
//
// Each body's phase field lives in a tile (a box of the periodic lattice that follows the body);
// phi is zero outside it. All phase-field arithmetic, reductions and the rigid-body update are FP64.
//  k_rasterize    : initial profile 1/2 - 1/2 sin(pi d / eta) of the signed distance d (Sec. 3.1).
//  k_flags        : clamp to [0,1], renormalise the solid sum, obstacle flag (fluid phase below the
//                   threshold, Sec. 3.2.2), owner = argmax, cover events.
//  k_body_props   : mass, centre of mass and inertia from phi.
//  k_repulsion    : solid-solid repulsion between body points (Eqs. soild_solid_potential and
//                   solid_solid_force, Sec. 3.1.2).
//  k_bodies       : force/torque totals and the rigid-body update (Sec. 3.1.1), tile recentring,
//                   overlap lists, fluid-mass total.
//  k_sweep        : one conservative MUSCL sweep with the monotonized-central limiter of
//                   d(phi)/dt = -u_B . grad(phi) (Eq. phase_advection, Sec. 3.3), x, y, z in turn.
//  k_kinetics     : Eq. sim_proc_phase_field_dynamics with the volume-restoring Delta g (Sec. 3.3).
#include <climits>
#include "tile.cuh"

namespace cbl {

constexpr double PI = 3.14159265358979323846;
constexpr int MAXOFF = 512;
// (in global memory: lanes read different entries)
__device__ int c_off[3 * MAXOFF];
__device__ double c_offf[3 * MAXOFF];  // force on the first point of a pair at offset d: f(d)
__device__ int c_noff;

// Offsets d with 0 < |d| < r_c and the pair force e0 (n / r_c) |(|d| - r_c) / r_c|^(n-1) (-d/|d|)
// (Eq. solid_solid_force) that a point feels from a point at x + d.
void set_repulsion_offsets(double rc, double e0, int nrep, cudaStream_t s) {
  int off[3 * MAXOFF];
  double ff[3 * MAXOFF];
  int n = 0;
  int R = (int)ceil(rc);
  for (int dz = -R; dz <= R; ++dz)
    for (int dy = -R; dy <= R; ++dy)
      for (int dx = -R; dx <= R; ++dx) {
        int d2 = dx * dx + dy * dy + dz * dz;
        if (d2 > 0 && (double)d2 < rc * rc && n < MAXOFF) {
          off[3 * n] = dx;
          off[3 * n + 1] = dy;
          off[3 * n + 2] = dz;
          const double d = sqrt((double)d2);
          const double mag = e0 * nrep / rc * pow(fabs((d - rc) / rc), (double)(nrep - 1));
          ff[3 * n] = -dx / d * mag;
          ff[3 * n + 1] = -dy / d * mag;
          ff[3 * n + 2] = -dz / d * mag;
          n++;
        }
      }
  cudaMemcpyToSymbolAsync(c_off, off, sizeof(int) * 3 * n, 0, cudaMemcpyHostToDevice, s);
  cudaMemcpyToSymbolAsync(c_offf, ff, sizeof(double) * 3 * n, 0, cudaMemcpyHostToDevice, s);
  cudaMemcpyToSymbolAsync(c_noff, &n, sizeof(int), 0, cudaMemcpyHostToDevice, s);
}

__device__ __forceinline__ void quat_R(const double q[4], double R[9]) {
  double w = q[0], x = q[1], y = q[2], z = q[3];
  R[0] = 1 - 2 * (y * y + z * z); R[1] = 2 * (x * y - w * z);     R[2] = 2 * (x * z + w * y);
  R[3] = 2 * (x * y + w * z);     R[4] = 1 - 2 * (x * x + z * z); R[5] = 2 * (y * z - w * x);
  R[6] = 2 * (x * z - w * y);     R[7] = 2 * (y * z + w * x);     R[8] = 1 - 2 * (x * x + y * y);
}

__device__ __forceinline__ void xcross(const double a[3], const double b[3], double r[3]) {
  r[0] = a[1] * b[2] - a[2] * b[1];
  r[1] = a[2] * b[0] - a[0] * b[2];
  r[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ double dwarp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---- initial profile ---------------------------------------------------------------------------
__device__ double body_sdf(const BodyDev& b, const double r[3]) {
  if (b.shape == 0) return sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]) - b.radius;
  double R[9];
  quat_R(b.q0, R);
  double o = 0, m = -1e300;
  for (int a = 0; a < 3; ++a) {
    double l = R[0 + a] * r[0] + R[3 + a] * r[1] + R[6 + a] * r[2];
    double q = fabs(l) - b.half[a];
    double v = q > 0 ? q : 0;
    o += v * v;
    m = q > m ? q : m;
  }
  return sqrt(o) + (m < 0 ? m : 0.0);
}

__global__ void k_rasterize(BodyDev* bodies, double* arena, Lat lat, double eta) {
  const BodyDev& b = bodies[blockIdx.y];
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= b.sz) return;
  TileCell c = tile_cell(b, t, lat);
  double r[3] = {mimg(c.gx - b.c0[0], lat.nx), mimg(c.gy - b.c0[1], lat.ny), mimg(c.gz - b.c0[2], lat.nz)};
  double d = body_sdf(b, r);
  double v = d <= -0.5 * eta ? 1.0 : (d >= 0.5 * eta ? 0.0 : 0.5 - 0.5 * sin(PI * d / eta));
  double* buf = arena + b.off;
  buf[t] = __longlong_as_double(phi_clamp(dbits(v)));
  buf[b.sz + t] = 0.0;
  buf[2 * b.sz + t] = 0.0;
}

// ---- overlap lists -----------------------------------------------------------------------------
__device__ bool tiles_overlap(const BodyDev& a, const BodyDev& b, const Lat& lat) {
  const int n[3] = {lat.nx, lat.ny, lat.nz};
  for (int d = 0; d < 3; ++d) {
    bool ov = wrapi_near(b.o[d] - a.o[d], n[d]) < a.L[d] || wrapi_near(a.o[d] - b.o[d], n[d]) < b.L[d];
    if (!ov) return false;
  }
  return true;
}

__device__ void build_lists(BodyDev* bodies, int nb, const Lat& lat, StepState* st) {
  for (int a = threadIdx.x; a < nb; a += blockDim.x) {
    int cnt = 0;
    for (int b = 0; b < nb; ++b) {
      if (b == a || !tiles_overlap(bodies[a], bodies[b], lat)) continue;
      if (cnt < MAXNB) bodies[a].nbl[cnt++] = b;
      else atomicOr(&st->err, E_NBLIST);
    }
    bodies[a].nnb = cnt;
  }
}

__global__ void k_neighbour_lists(BodyDev* bodies, int nb, Lat lat, StepState* st) {
  build_lists(bodies, nb, lat, st);
}

// ---- flags --------------------------------------------------------------------------------------

// A cell's obstacle flag changed: a covered cell hands over its populations (near_refill), and the moment
// pass has to pull the cell's surroundings again from the populations (k_mom_close), which needs those
// within 3 cells of a covered, 2 of an uncovered cell stored; where the bricks do not say so, all of them
// are written first (k_mom_fill).
__device__ __noinline__ void flag_event(const TileSet& S, const TileCell& c, long long n, int reach) {
  S.events[atomicAdd(&S.cs->nevent, 1u)] = (int)n;
  if (!S.mom) return;
  const MomDev& md = S.md;
  int b[3][BRICK_SPAN], nbk[3];
  nbk[0] = brick_span(c.gx, reach, S.lat.nx, b[0]);
  nbk[1] = brick_span(c.gy, reach, S.lat.ny, b[1]);
  nbk[2] = brick_span(c.gz, reach, S.lat.nz, b[2]);
  const unsigned char* map = md.map(S.st->parity);
  bool all = true;
  for (int iz = 0; iz < nbk[2]; ++iz)
    for (int iy = 0; iy < nbk[1]; ++iy)
      for (int ix = 0; ix < nbk[0]; ++ix) all &= map[md.brick(b[0][ix], b[1][iy], b[2][iz])] != 0;
  if (!all) S.cs->full = 1;
}

// New obstacle flag of a cell; the near-solid bit is rebuilt by the pass that follows (the exchange keeps the
// solid cell's word whole while another block clears that bit). The cover bit stays until the body update of
// the next step clears it (its users come after this pass).
__device__ __forceinline__ void set_flag(const TileSet& S, const TileCell& c, bool solid, int owner, int init) {
  const long long n = lat_index(c, S.lat);
  uint16_t old = S.flags[n];
  if (solid && !init && !(old & F_SOLID)) {
    const uint16_t nf = F_SOLID | F_COVER | (uint16_t)owner;
    for (int k = 0; k < 4; ++k) {  // again only if the near-solid bit was cleared in between
      const uint16_t seen = atomicCAS(S.flags + n, old, nf);
      if (seen == old) {
        atomicAdd(&S.st->ncover, 1u);
        flag_event(S, c, n, 3);
        return;
      }
      if (seen & F_SOLID) return;
      old = seen;
    }
    return;
  }
  const uint16_t nf = solid ? (uint16_t)(F_SOLID | (uint16_t)owner | (old & F_COVER)) : (uint16_t)0;
  if (!init && !solid && (old & F_SOLID)) flag_event(S, c, n, 2);
  if ((uint16_t)(old & ~F_NEAR) != nf) S.flags[n] = nf;
}

// Clamp to [0, 1], renormalise the solid sum, obstacle flag (fluid phase below the threshold, Sec. 3.2.2) and
// owner (the largest phase, ties to the lower id), cover events. A cell is written by one body: the one
// whose phase field is not zero there, the lowest of them where several are not. All bodies' blocks run at
// once and look at each other's fields, so this kernel makes no value zero: what the clamp sets to 0 counts
// as 0 here and is set by the pass that follows (k_near_refill), each body's own. (What is rescaled to a
// sum of 1 stays above 1e-14.) A cell whose field has gone to zero under its owner in this step (a body
// moving by cells) is written by the owner, or by any body whose tile holds it if the owner's has left it,
// by all alike. The cells with phi >= the membership threshold make up the body's member record (tile-coordinate
// box and largest squared distance from X, a bound: the fields may still be rescaled) for the repulsion of
// the next step. The blocks also clear the near-solid bits of the old boundary list (atomically: a
// neighbouring half word may be written meanwhile).
template <bool B, int Z>
__global__ void __launch_bounds__(TILE_T) k_flags(const __grid_constant__ TileSet one, const TileSet* __restrict__ sets,
                                                  const int2* __restrict__ items, int init) {
  int self;
  const TileSet& S = tile_set<B>(one, sets, items, self);
  const Lat& lat = S.lat;
  __shared__ TileList list;
  __shared__ int sbox[7];
  if (threadIdx.x == 0) list.n = 0;
  if (threadIdx.x < 7) sbox[threadIdx.x] = threadIdx.x < 3 ? INT_MAX : (threadIdx.x < 6 ? INT_MIN : 0);
  if (!init) {
    const unsigned count = S.st->nbnd, per = gridDim.x * gridDim.y * TILE_T;
    for (unsigned k = ((unsigned)self * gridDim.y + blockIdx.y) * gridDim.x * TILE_T + blockIdx.x * TILE_T + threadIdx.x;
         k < count; k += per * (unsigned)S.nb) {
      const unsigned n = (unsigned)S.blist[k];
      atomicAnd(reinterpret_cast<unsigned*>(S.flags) + (n >> 1), ~((unsigned)F_NEAR << ((n & 1u) * 16u)));
    }
  }
  __syncthreads();
  const BodyDev& b = S.bodies[self];
  const int L0 = b.L[0], L1 = b.L[1], L2 = b.L[2], z0 = blockIdx.y * Z;
  const unsigned p = blockIdx.x * TILE_T + threadIdx.x, plane = (unsigned)L0 * L1;
  if (z0 >= L2) return;
  const int i1 = (int)(p / (unsigned)L0), i0 = (int)(p - (unsigned)i1 * L0);
  double* const phi = S.arena + b.off;
  const double thr = S.solid_thr;  // (above 1 every cell of a tile is solid)
  const bool low = thr <= 0.5;
#pragma unroll
  for (int q = 0; q < Z; ++q) {
    const bool in = p < plane && z0 + q < L2;
    const long long vb = in ? dbits(phi[p + (size_t)plane * (z0 + q)]) : 0;
    tile_append(list, in && (vb != 0 || thr > 1.0), q * TILE_T + threadIdx.x);
    if (!in || vb != 0 || init) continue;
    const TileCell c = tile_at(b, i0, i1, z0 + q, lat);
    const uint16_t old = S.flags[lat_index(c, lat)];
    if (!(old & F_SOLID)) continue;
    const int o = old & F_OWNER;
    if (o != self && (o >= S.nb || tile_index(S.bodies[o].o, S.bodies[o].L, c.gx, c.gy, c.gz, lat) >= 0)) continue;
    bool others = false;
    for (int k = 0; k < b.nnb && !others; ++k) {
      const BodyDev& ob = S.bodies[b.nbl[k]];
      const long long j = tile_index(ob.o, ob.L, c.gx, c.gy, c.gz, lat);
      others = j >= 0 && dbits(S.arena[ob.off + j]) != 0;
    }
    if (!others) set_flag(S, c, false, 0, init);
  }
  __syncthreads();
  const long long mthr = dbits(S.member_thr);
  int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {INT_MIN, INT_MIN, INT_MIN};
  float r2 = 0.0f;
  for (int e = threadIdx.x; e < list.n; e += TILE_T) {
    const int id = list.id[e];
    const unsigned pc = blockIdx.x * TILE_T + (id & (TILE_T - 1));
    const int z = z0 + id / TILE_T, c1 = (int)(pc / (unsigned)L0), c0 = (int)(pc - (unsigned)c1 * L0);
    const TileCell c = tile_at(b, c0, c1, z, lat);
    double* const p0 = phi + pc + (size_t)plane * z;
    const long long own = dbits(*p0);
    if (own >= mthr || (own > dbits(1.0 - PHI_EPS) && mthr <= dbits(1.0))) {
      // in float from the float mirror of X (FP64 is 1/64 rate here and this is a bound with slack);
      // tile cells lie within half a lattice length of X along each axis, so one wrap suffices
      float d2 = 0.0f;
      const int g[3] = {c.gx, c.gy, c.gz}, l[3] = {c0, c1, z}, nn[3] = {lat.nx, lat.ny, lat.nz};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        float d = (float)g[a] - b.Xf[a];
        const float h = 0.5f * (float)nn[a];
        if (d >= h) d -= (float)nn[a];
        else if (d < -h) d += (float)nn[a];
        d2 += d * d;
        lo[a] = min(lo[a], l[a]);
        hi[a] = max(hi[a], l[a]);
      }
      r2 = fmaxf(r2, d2);
    }
    // bodies whose field is not zero at this cell, ascending id
    double* ptr[MAXNB + 1];
    int ids[MAXNB + 1];
    int m = 0, me = -1;
    bool first = true;
    for (int k = 0; k <= b.nnb; ++k) {
      if (me < 0 && (k == b.nnb || b.nbl[k] > self)) {
        me = m;
        ptr[m] = p0;
        ids[m++] = self;
      }
      if (k == b.nnb) break;
      const BodyDev& o = S.bodies[b.nbl[k]];
      const long long j = tile_index(o.o, o.L, c.gx, c.gy, c.gz, lat);
      if (j < 0) continue;
      double* const po = S.arena + o.off + j;
      if (dbits(*po) == 0) continue;
      if (b.nbl[k] < self) {  // that body writes this cell
        first = false;
        break;
      }
      ptr[m] = po;
      ids[m++] = b.nbl[k];
    }
    if (!first) continue;
    if (thr > 1.0 && dbits(*p0) == 0 && (m > 1 || covered_by_lower_body(S.bodies, b, self, c.gx, c.gy, c.gz, lat))) continue;
    double S1 = 0.0;
    for (int k = 0; k < m; ++k) {
      const long long old = dbits(*ptr[k]), vb = phi_clamp(old);
      const double v = __longlong_as_double(vb);
      if (vb != old && vb != 0) *ptr[k] = v;  // 1
      S1 = k ? S1 + v : v;
    }
    if (m > 1 && S1 > 1.0) {
      double S2 = 0.0;
      for (int k = 0; k < m; ++k) {
        const long long vb = phi_clamp(dbits(*ptr[k]));
        if (vb == 0) continue;
        const double v = __longlong_as_double(vb) / S1;
        *ptr[k] = v;
        S2 += v;
      }
      S1 = S2;
    }
    // 1 - S < thr; no FP64 where S is 1, or below 1/2 with a threshold of at most 1/2
    bool solid;
    if (dbits(S1) == dbits(1.0)) solid = thr > 0.0;
    else if (low && dbits(S1) < dbits(0.5)) solid = false;
    else solid = 1.0 - S1 < thr;
    int best = ids[0];
    if (solid && m > 1) {
      double bv = __longlong_as_double(phi_clamp(dbits(*ptr[0])));
      for (int k = 1; k < m; ++k)
        if (*ptr[k] > bv) {
          bv = *ptr[k];
          best = ids[k];
        }
    }
    set_flag(S, c, solid, best, init);
  }
  if (init) return;
  // the body's member record: warp, then block, then one set of global atomics per block
  if (__any_sync(0xffffffffu, hi[0] >= 0)) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int l = __reduce_min_sync(0xffffffffu, lo[a]), h = __reduce_max_sync(0xffffffffu, hi[a]);
      if ((threadIdx.x & 31) == 0) {
        atomicMin(sbox + a, l);
        atomicMax(sbox + 3 + a, h);
      }
    }
    // non-negative floats order like their bit patterns
    const unsigned rb = __reduce_max_sync(0xffffffffu, __float_as_uint(r2));
    if ((threadIdx.x & 31) == 0) atomicMax(sbox + 6, (int)rb);
  }
  __syncthreads();
  if (threadIdx.x < 7) {
    int* const box = S.mbox + MBOX_N * self;
    if (mthr <= 0) {  // every cell of the tile is a member (a threshold of 0 or below)
      const int L = threadIdx.x < 6 ? b.L[threadIdx.x % 3] : 0;
      const float far2 = (float)(L0 * L0 + L1 * L1 + L2 * L2);
      if (threadIdx.x < 3) atomicMin(box + threadIdx.x, 0);
      else atomicMax(box + threadIdx.x, threadIdx.x < 6 ? L - 1 : __float_as_int(far2));
    } else if (sbox[0] <= sbox[3]) {
      if (threadIdx.x < 3) atomicMin(box + threadIdx.x, sbox[threadIdx.x]);
      else atomicMax(box + threadIdx.x, sbox[threadIdx.x]);
    }
  }
}

// ---- body properties (initialisation) ---------------------------------------------------------
// pass 0: sum phi and sum r phi about the nominal centre; pass 1: inertia about X
__global__ void k_body_props(const BodyDev* bodies, const double* arena, double* scratch, Lat lat, int pass) {
  const int self = blockIdx.y;
  const BodyDev& b = bodies[self];
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  TileCell c;
  if (t < b.sz) {
    c = tile_cell(b, t, lat);
    v = arena[b.off + t];
  }
  double a[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  if (v != 0.0) {
    if (pass == 0) {
      a[0] = v;
      a[1] = v * mimg(c.gx - b.c0[0], lat.nx);
      a[2] = v * mimg(c.gy - b.c0[1], lat.ny);
      a[3] = v * mimg(c.gz - b.c0[2], lat.nz);
    } else {
      double r[3] = {mimg(c.gx - b.X[0], lat.nx), mimg(c.gy - b.X[1], lat.ny), mimg(c.gz - b.X[2], lat.nz)};
      double rr = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
      for (int p = 0; p < 3; ++p)
        for (int q = 0; q < 3; ++q) a[3 * p + q] = v * ((p == q ? rr : 0.0) - r[p] * r[q]);
    }
  }
  for (int k = 0; k < 9; ++k) {
    double s = dwarp_sum(a[k]);
    if ((threadIdx.x & 31) == 0 && s != 0.0) atomicAdd(scratch + self * 9 + k, s);
  }
}

__global__ void k_body_props_finish(BodyDev* bodies, int nb, const double* scratch, Lat lat, int pass) {
  int self = blockIdx.x * blockDim.x + threadIdx.x;
  if (self >= nb) return;
  BodyDev& b = bodies[self];
  const double* s = scratch + self * 9;
  const int n[3] = {lat.nx, lat.ny, lat.nz};
  if (pass == 0) {
    for (int a = 0; a < 3; ++a) {
      double X = b.c0[a] + s[1 + a] / s[0];
      X = fmod(X, (double)n[a]);
      if (X < 0) X += n[a];
      b.X[a] = X;
      b.Xprev[a] = X;
    }
    mirror_f(b);
    b.M = b.rho_s * s[0];
    b.vol_ref = s[0];
  } else {
    double R[9];
    quat_R(b.Q, R);
    const double rho_s = b.rho_s;
    for (int a = 0; a < 3; ++a)
      for (int c = 0; c < 3; ++c) {
        double acc = 0;
        for (int k = 0; k < 3; ++k)
          for (int l = 0; l < 3; ++l) acc += R[3 * k + a] * (rho_s * s[3 * k + l]) * R[3 * l + c];
        b.Ib[3 * a + c] = acc;
      }
    const double* I = b.Ib;
    const double det = I[0] * (I[4] * I[8] - I[5] * I[7]) - I[1] * (I[3] * I[8] - I[5] * I[6]) +
                       I[2] * (I[3] * I[7] - I[4] * I[6]);
    b.Ibinv[0] = (I[4] * I[8] - I[5] * I[7]) / det;
    b.Ibinv[1] = (I[2] * I[7] - I[1] * I[8]) / det;
    b.Ibinv[2] = (I[1] * I[5] - I[2] * I[4]) / det;
    b.Ibinv[3] = (I[5] * I[6] - I[3] * I[8]) / det;
    b.Ibinv[4] = (I[0] * I[8] - I[2] * I[6]) / det;
    b.Ibinv[5] = (I[2] * I[3] - I[0] * I[5]) / det;
    b.Ibinv[6] = (I[3] * I[7] - I[4] * I[6]) / det;
    b.Ibinv[7] = (I[1] * I[6] - I[0] * I[7]) / det;
    b.Ibinv[8] = (I[0] * I[4] - I[1] * I[3]) / det;
  }
}

// ---- solid-solid repulsion ---------------------------------------------------------------------
// For a point x of body A (phi_A >= the membership threshold) and every body B whose tile overlaps
// A's: sum the table forces f(d) over the points x + d of B; torque (x - X_A) x (sum f).
// The points in reach of a contact are few and close together: blocks take chunks of them, a warp a point, a
// lane a few of its offsets. Two touching spheres of R = 20: 51 us with a point per thread (its
// hundred offsets one after the other, all in a few blocks), 27 to 34 here; four at R = 24, 65 and 28. None in range: 4.
constexpr unsigned REP_T = 256;

template <bool B>
__global__ void __launch_bounds__(REP_T) k_repulsion(const __grid_constant__ TileSet one, const TileSet* __restrict__ sets,
                                                   const int2* __restrict__ items) {
  int self;
  const TileSet& S = tile_set<B>(one, sets, items, self);
  const BodyDev* const bodies = S.bodies;
  const BodyDev& a = bodies[self];
  if (a.nnb == 0 || !S.rep) return;  // block-uniform
  const Lat& lat = S.lat;
  const double* const arena = S.arena;
  double* const acc = S.acc;
  const int* const mbox = S.mbox;
  const int Rc = S.Rc;
  const double thr = S.member_thr, rc = S.rc;
  // Block-uniform cull, a neighbour per thread: every member point (phi >= the membership threshold) of a
  // body lies within its member radius of its centre X, so two bodies whose centres are farther apart
  // than the two member radii plus rc (and a cell of slack, which covers FP32 rounding) have no pair in
  // range; and every member point of A lies in A's member box, so if along some axis the two boxes are
  // more than Rc cells apart (periodic distance), no point of A passes the per-point box test below.
  // (One thread in FP64 took most of this kernel's 27 us where no pair is in range.)
  bool nearby = false;
  // hull, in A's tile, of A's member box cut with the boxes (grown by Rc) of the neighbours in range: only
  // these cells can have a partner
  __shared__ int hull[6];
  if (threadIdx.x < 6) hull[threadIdx.x] = threadIdx.x < 3 ? INT_MAX : INT_MIN;
  __syncthreads();
  if (threadIdx.x < a.nnb) {
    const int nn[3] = {lat.nx, lat.ny, lat.nz};
    const int* ba = mbox + MBOX_N * self;
    const BodyDev& b = bodies[a.nbl[threadIdx.x]];
    const int* bb = mbox + MBOX_N * a.nbl[threadIdx.x];
    float d2 = 0.0f;
    bool boxes = true;
    for (int d = 0; d < 3; ++d) {
      float dx = b.Xf[d] - a.Xf[d];
      dx -= (float)nn[d] * rintf(dx / (float)nn[d]);
      d2 += dx * dx;
      if (ba[d] > ba[3 + d] || bb[d] > bb[3 + d]) {  // an empty box: no members
        boxes = false;
        break;
      }
      // centres and half-lengths (in half cells) of the two boxes in lattice coordinates
      const int ca2 = 2 * a.o[d] + ba[d] + ba[3 + d], cb2 = 2 * b.o[d] + bb[d] + bb[3 + d];
      const int ha2 = ba[3 + d] - ba[d], hb2 = bb[3 + d] - bb[d];
      int sep2 = wrapi(cb2 - ca2, 2 * nn[d]);
      if (sep2 > nn[d]) sep2 = 2 * nn[d] - sep2;  // periodic distance of the centres
      if (sep2 - ha2 - hb2 > 2 * Rc) boxes = false;
    }
    const float lim = sqrtf(__int_as_float(ba[MBOX_R2])) + sqrtf(__int_as_float(bb[MBOX_R2])) + (float)rc + 1.0f;
    nearby = boxes && !(d2 > lim * lim);
    if (nearby)
      for (int d = 0; d < 3; ++d)
        for (int image = -2; image <= 2; ++image) {
          // (tile origins lie within half a lattice length of [0, n): two images either way cover all)
          const int at = b.o[d] - a.o[d] + image * nn[d];
          const int lo = max(at + bb[d] - Rc, ba[d]), hi = min(at + bb[3 + d] + Rc, ba[3 + d]);
          if (lo > hi) continue;
          atomicMin(hull + d, lo);
          atomicMax(hull + 3 + d, hi);
        }
  }
  if (!__syncthreads_or(nearby)) return;
  const int h0 = hull[0], h1 = hull[1], h2 = hull[2], w0 = hull[3] - h0 + 1, w1 = hull[4] - h1 + 1, w2 = hull[5] - h2 + 1;
  if (w0 <= 0 || w1 <= 0 || w2 <= 0) return;
  const unsigned cells = (unsigned)w0 * (unsigned)w1 * (unsigned)w2, w01 = (unsigned)w0 * (unsigned)w1;
  const long long tb = dbits(thr);
  // chunks of the hull, of 32 to 256 cells, so that few cells still reach many SMs
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned share = (cells + gridDim.x - 1) / gridDim.x, chunk = min(REP_T, (share + 31u) & ~31u);
  __shared__ unsigned list[REP_T], reached[REP_T];
  static_assert(MAXNB <= 32, "a bit per neighbour");
  __shared__ int n_list;
  double F[3] = {0, 0, 0}, T[3] = {0, 0, 0};
  bool has = false;
  for (unsigned base = blockIdx.x * chunk; base < cells; base += gridDim.x * chunk) {
    if (threadIdx.x == 0) n_list = 0;
    __syncthreads();
    const unsigned k = base + threadIdx.x;
    if (threadIdx.x < chunk && k < cells) {
      const int l2 = (int)(k / w01), r = (int)(k - (unsigned)l2 * w01), l1 = r / w0, l0 = r - l1 * w0;
      unsigned reach = 0;  // neighbours that the point may reach
      if (dbits(arena[a.off + h0 + l0 + (long long)a.L[0] * (h1 + l1 + (long long)a.L[1] * (h2 + l2))]) >= tb) {
        const TileCell c = tile_at(a, h0 + l0, h1 + l1, h2 + l2, lat);
        const int g[3] = {c.gx, c.gy, c.gz}, nn[3] = {lat.nx, lat.ny, lat.nz};
        for (int kb = 0; kb < a.nnb; ++kb) {
          // tile coordinates of the other body's member cells (phi >= thr) lie in its box mbox (built by the
          // flag pass); the offsets reach Rc cells per axis, so a point outside the box grown by Rc
          // (periodically) finds no partner
          const BodyDev& b = bodies[a.nbl[kb]];
          const int* bx = mbox + MBOX_N * a.nbl[kb];
          bool near = true;
          for (int d = 0; d < 3; ++d) {
            const int l = wrapi_near(g[d] - b.o[d], nn[d]), lo = bx[d] - Rc, hi = bx[3 + d] + Rc;
            const bool in = (l >= lo && l <= hi) || (l - nn[d] >= lo && l - nn[d] <= hi) ||
                            (l + nn[d] >= lo && l + nn[d] <= hi);
            if (bx[d] > bx[3 + d] || !in) near = false;  // an empty box has no members
          }
          if (!near) continue;
          // and within B's member radius (plus rc and a cell) of B's centre
          float dx = (float)c.gx - b.Xf[0], dy = (float)c.gy - b.Xf[1], dz = (float)c.gz - b.Xf[2];
          dx -= (float)lat.nx * rintf(dx / (float)lat.nx);
          dy -= (float)lat.ny * rintf(dy / (float)lat.ny);
          dz -= (float)lat.nz * rintf(dz / (float)lat.nz);
          const float lim = sqrtf(__int_as_float(bx[MBOX_R2])) + (float)rc + 1.0f;
          if (!(dx * dx + dy * dy + dz * dz > lim * lim)) reach |= 1u << kb;
        }
      }
      if (reach) {
        const int at = atomicAdd(&n_list, 1);
        list[at] = k;
        reached[at] = reach;
      }
    }
    __syncthreads();
    const int n = n_list;
    for (int e = warp; e < n; e += REP_T / 32) {
      const unsigned q0 = list[e];
      const int l2 = (int)(q0 / w01), r = (int)(q0 - (unsigned)l2 * w01), l1 = r / w0, l0 = r - l1 * w0;
      const TileCell c = tile_at(a, h0 + l0, h1 + l1, h2 + l2, lat);
      const int g[3] = {c.gx, c.gy, c.gz};
      const int nn[3] = {lat.nx, lat.ny, lat.nz};
      double f[3] = {0, 0, 0};
      bool hit = false;
      for (unsigned todo = reached[e]; todo; todo &= todo - 1) {
        const BodyDev& b = bodies[a.nbl[__ffs(todo) - 1]];
        int l[3];  // the point's coordinates in the other body's tile, wrapped to [0, n)
        for (int d = 0; d < 3; ++d) l[d] = wrapi_near(g[d] - b.o[d], nn[d]);
        const double* bb = arena + b.off;
        // a lane per offset; four loads are issued before any of them is tested
        for (int j0 = 0; j0 < c_noff; j0 += 128) {
          double v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = j0 + 32 * u + lane;
            long long q = -1;
            if (j < c_noff) {
              int m[3];
              bool in = true;
              for (int d = 0; d < 3; ++d) {
                m[d] = l[d] + c_off[3 * j + d];  // |offset| <= 6: at most two wraps on a 4-cell side
                while (m[d] < 0) m[d] += nn[d];
                while (m[d] >= nn[d]) m[d] -= nn[d];
                in &= m[d] < b.L[d];
              }
              if (in) q = (long long)m[0] + (long long)b.L[0] * ((long long)m[1] + (long long)b.L[1] * m[2]);
            }
            v[u] = q >= 0 ? __ldg(bb + q) : 0.0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = j0 + 32 * u + lane;
            if (j >= c_noff || dbits(v[u]) < tb) continue;
            f[0] += c_offf[3 * j];
            f[1] += c_offf[3 * j + 1];
            f[2] += c_offf[3 * j + 2];
            hit = true;
          }
        }
      }
      if (!__any_sync(0xffffffffu, hit)) continue;
      // the arm, an axis per lane
      const int ax = min(lane, 2);
      const double arm1 = mimg((double)g[ax] - a.X[ax], nn[ax]);
      const double arm[3] = {__shfl_sync(0xffffffffu, arm1, 0), __shfl_sync(0xffffffffu, arm1, 1),
                             __shfl_sync(0xffffffffu, arm1, 2)};
      if (hit) {
        double t[3];
        xcross(arm, f, t);
        for (int p = 0; p < 3; ++p) {
          F[p] += f[p];
          T[p] += t[p];
        }
        has = true;
      }
    }
    __syncthreads();  // the list is written again
  }
  // block totals, then one atomic per component
  if (!__syncthreads_or(has)) return;
  __shared__ double sum[REP_T / 32][6];
  for (int p = 0; p < 3; ++p) {
    const double sf = dwarp_sum(F[p]), st = dwarp_sum(T[p]);
    if (lane == 0) {
      sum[warp][p] = sf;
      sum[warp][3 + p] = st;
    }
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double t = 0.0;
    for (int w = 0; w < REP_T / 32; ++w) t += sum[w][threadIdx.x];
    const int slot = threadIdx.x < 3 ? ACC_REP_F + threadIdx.x : ACC_REP_T + threadIdx.x - 3;
    if (t != 0.0) atomicAdd(acc + (size_t)self * ACC_N + slot, t);
  }
}

// ---- rigid bodies ------------------------------------------------------------------------------
// Semi-implicit Euler with dt = 1: V += F/M, X += V, omega += I_w^-1 T with I_w = R I_body R^T,
// q <- normalize(exp(omega/2) q); fixed bodies keep V = omega = 0.
// A body whose update is not finite, or moves it by a lattice length or more in one step (a run
// that has blown up), is held at its last pose from then on and E_UNSTABLE is raised: every later
// kernel that derives a tile origin or a wrap from X gets finite, in-range values.
//
// One block per body, its record in shared memory, translation and rotation on two warps with a
// component per lane: the update is a chain of dependent FP64 operations (64 times slower than FP32 on
// GB300), on the critical path of small lattices. One thread per body and global memory in the chain took
// 17 to 22 us for 2 to 4 bodies and 90 for 60; this 11. The orientation, which no kernel of the
// step needs, follows beside the first advection sweep (turn_body).
constexpr int BODY_T = 128;

__device__ __forceinline__ void turn_body(BodyDev& b) {
  if (b.fixed) return;
  const double w2 = b.W[0] * b.W[0] + b.W[1] * b.W[1] + b.W[2] * b.W[2];
  if (!(w2 > 0)) return;
  const double iw = rsqrt(w2), wn = w2 * iw;
  double sn, cs;
  sincos(0.5 * wn, &sn, &cs);
  const double s = sn * iw;
  const double dq[4] = {cs, b.W[0] * s, b.W[1] * s, b.W[2] * s};
  const double q[4] = {b.Q[0], b.Q[1], b.Q[2], b.Q[3]};
  const double nq[4] = {dq[0] * q[0] - dq[1] * q[1] - dq[2] * q[2] - dq[3] * q[3],
                        dq[0] * q[1] + dq[1] * q[0] + dq[2] * q[3] - dq[3] * q[2],
                        dq[0] * q[2] - dq[1] * q[3] + dq[2] * q[0] + dq[3] * q[1],
                        dq[0] * q[3] + dq[1] * q[2] - dq[2] * q[1] + dq[3] * q[0]};
  const double iq = rsqrt(nq[0] * nq[0] + nq[1] * nq[1] + nq[2] * nq[2] + nq[3] * nq[3]);
  for (int a = 0; a < 4; ++a) b.Q[a] = nq[a] * iq;
}

template <bool B>
__global__ void __launch_bounds__(BODY_T) k_bodies(const __grid_constant__ TileSet one, const TileSet* __restrict__ sets,
                                                   const int2* __restrict__ items) {
  int i;
  const TileSet& S = tile_set<B>(one, sets, items, i);
  const Lat& lat = S.lat;
  const int n[3] = {lat.nx, lat.ny, lat.nz}, tid = threadIdx.x, lane = tid & 31;
  static_assert(sizeof(BodyDev) % 8 == 0, "copied in 8-byte words");
  __shared__ __align__(8) unsigned char raw[sizeof(BodyDev)];
  __shared__ double a[ACC_N];
  __shared__ int s_bad;
  BodyDev& b = *reinterpret_cast<BodyDev*>(raw);
  unsigned long long* const rec = reinterpret_cast<unsigned long long*>(S.bodies + i);
  for (int k = tid; k < (int)(sizeof(BodyDev) / 8); k += BODY_T) reinterpret_cast<unsigned long long*>(raw)[k] = rec[k];
  if (tid < ACC_N) a[tid] = S.acc[(size_t)i * ACC_N + tid];
  if (tid == 0) s_bad = 0;
  __syncthreads();
  const int c = lane < 3 ? lane : 0;
  if (tid < 32) {
    // lane c: component c of the translation
    const double F = a[ACC_MOM_F + c] + a[ACC_ADH_F + c] + a[ACC_REP_F + c];
    const double X = b.X[c];
    if (lane < 3) {
      S.fsum[6 * i + c] += F;  // running sums (mean forces over many steps without host reads)
      b.Xprev[c] = X;
      if (!b.fixed) {
        const double V = b.V[c] + F * (1.0 / b.M);
        // periodic wrap in closed form (a move of less than a lattice side: the value of fmod)
        const double Xn = wrapd(X + V, n[c]);
        b.V[c] = V;
        b.X[c] = Xn;
        // finite and shorter than the lattice side (NaN fails the comparison)
        if (!(fabs(V) < (double)n[c]) || !isfinite(Xn)) s_bad = 1;
      } else {
        b.V[c] = 0;
      }
    }
  } else if (tid < 64) {
    // lane c: component c of the rotation, R (I_body^-1 (R^T T)) instead of forming the world-frame inverse
    const double T = a[ACC_MOM_T + c] + a[ACC_ADH_T + c] + a[ACC_REP_T + c];
    if (lane < 3) S.fsum[6 * i + 3 + c] += T;
    if (!b.fixed) {
      double R[9];
      quat_R(b.Q, R);
      const double T0 = __shfl_sync(0xffffffffu, T, 0), T1 = __shfl_sync(0xffffffffu, T, 1), T2 = __shfl_sync(0xffffffffu, T, 2);
      const double rc0 = c == 0 ? R[0] : (c == 1 ? R[1] : R[2]), rc1 = c == 0 ? R[3] : (c == 1 ? R[4] : R[5]),
                   rc2 = c == 0 ? R[6] : (c == 1 ? R[7] : R[8]);
      const double t1 = rc0 * T0 + rc1 * T1 + rc2 * T2;  // (R^T T)_c
      const double u0 = __shfl_sync(0xffffffffu, t1, 0), u1 = __shfl_sync(0xffffffffu, t1, 1), u2 = __shfl_sync(0xffffffffu, t1, 2);
      const double t2 = b.Ibinv[3 * c] * u0 + b.Ibinv[3 * c + 1] * u1 + b.Ibinv[3 * c + 2] * u2;
      const double v0 = __shfl_sync(0xffffffffu, t2, 0), v1 = __shfl_sync(0xffffffffu, t2, 1), v2 = __shfl_sync(0xffffffffu, t2, 2);
      const double rr0 = c == 0 ? R[0] : (c == 1 ? R[3] : R[6]), rr1 = c == 0 ? R[1] : (c == 1 ? R[4] : R[7]),
                   rr2 = c == 0 ? R[2] : (c == 1 ? R[5] : R[8]);
      double W = b.W[c] + (rr0 * v0 + rr1 * v1 + rr2 * v2);
      if (b.rot_lock >> c & 1) W = 0.0;
      // (a square that overflows would make the orientation not finite)
      if (lane < 3) {
        if (!isfinite(W * W) || !isfinite(b.Q[0] + b.Q[1] + b.Q[2] + b.Q[3])) s_bad = 1;
        b.W[c] = W;
      }
    } else if (lane < 3) {
      b.W[c] = 0;
    }
  } else if (tid < 64 + ACC_N) {
    S.last[(size_t)i * ACC_N + tid - 64] = a[tid - 64];
    S.acc[(size_t)i * ACC_N + tid - 64] = 0.0;
  } else if (tid >= 96 && tid < 98) {
    S.volacc[2 * i + tid - 96] = 0.0;
  } else if (tid >= 98 && tid < 98 + MBOX_R2 + 1) {  // member record: rebuilt by this step's flag pass
    const int e = tid - 98;
    S.mbox[MBOX_N * i + e] = e < 3 ? INT_MAX : (e < 6 ? INT_MIN : 0);
  }
  if (i == 0) {
    // the cover bits of the last flag update have been used
    const unsigned cov = S.cs->nprev;
    for (unsigned k = tid; k < cov; k += BODY_T) {
      const unsigned e = (unsigned)S.events[k];
      atomicAnd(reinterpret_cast<unsigned*>(S.flags) + (e >> 1), ~((unsigned)F_COVER << ((e & 1u) * 16u)));
    }
    if (tid == 0) S.st->ncover = 0;  // counted by the flag pass
  }
  __syncthreads();
  if (tid < 3) {
    if (s_bad) {
      b.X[tid] = b.Xprev[tid];
      b.V[tid] = 0.0;
      b.W[tid] = 0.0;
      if (tid == 0) {
        b.fixed = 1;
        atomicOr(&S.st->err, E_UNSTABLE);
      }
    }
    b.Xf[tid] = (float)b.X[tid];
    b.Vf[tid] = (float)b.V[tid];
    b.Wf[tid] = (float)b.W[tid];
    b.o_prev[tid] = b.o[tid];
    if (b.L[tid] < n[tid]) b.o[tid] = (int)floor(b.X[tid] + 0.5) - b.L[tid] / 2;
  }
  __syncthreads();
  for (int k = tid; k < (int)(sizeof(BodyDev) / 8); k += BODY_T) rec[k] = reinterpret_cast<unsigned long long*>(raw)[k];
  // per axis, the minimum-image offset of every tile coordinate from the pre-update centre (the advection's
  // face velocities need it; the table saves each cell the FP64 wrap)
  for (int ax = 0; ax < 3; ++ax)
    for (int l = tid; l < b.L[ax]; l += BODY_T)
      S.rtab[((size_t)3 * i + ax) * S.Lmax + l] = mimg(wrapi_near(b.o[ax] + l, n[ax]) - b.Xprev[ax], n[ax]);
}

__global__ void __launch_bounds__(256) k_finish(double* mass_part, unsigned n_mass_part, StepState* st,
                                                ChainState* cs) {
  finish_step<256>(mass_part, n_mass_part, st, cs);
}

// outside a step: the boundary list that the refill built becomes the current one
__global__ void k_commit(StepState* st, ChainState* cs) {
  st->nbnd = cs->nnew;
  cs->nnew = 0;
  cs->nprev = cs->nevent;
  cs->nevent = 0;
}

// ---- advection ---------------------------------------------------------------------------------
// Monotonized-central slope: 0 unless dm and dp have the same sign, else
// sign(dm) min(2|dm|, |dm + dp| / 2, 2|dp|). Evaluated on bit patterns, with the same result as the
// plain FP64 form: doubling and halving a normal double add to or subtract from its exponent field,
// and non-negative doubles order like their bit patterns. Only dm + dp is an FP64 operation (GB300
// issues FP64 at 1/64 of the FP32 rate). The differences of phase-field values that reach this
// function are 0 or far above the subnormal range, so no product underflows and no half is
// subnormal.
__device__ __forceinline__ double mc_slope(double dm, double dp) {
  const long long bm = dbits(dm), bp = dbits(dp);
  const long long mag = 0x7FFFFFFFFFFFFFFFLL, one_exp = 1LL << 52;
  const long long am = bm & mag, ap = bp & mag;
  if (((bm ^ bp) < 0) || am == 0 || ap == 0) return 0.0;
  const long long two_am = am + one_exp, two_ap = ap + one_exp;
  const long long half_s = (dbits(dm + dp) & mag) - one_exp;
  long long m = two_am < half_s ? two_am : half_s;
  m = m < two_ap ? m : two_ap;
  return __longlong_as_double(m | (bm & (long long)0x8000000000000000ULL));
}

// one sweep along axis D: out (origin b.o) <- in (origin o_in). The x-sweep reads with the previous
// origin, so the recentring shift (at most one cell per axis and step) is folded into it. Stencil
// values are addressed in tile-local coordinates; a periodic axis (tile as long as the lattice)
// wraps, any other axis reads zero outside the tile.
__device__ __forceinline__ int in_local(int i, int shift, int L, int n) {
  int l = i + shift;
  if (L == n) l = l < 0 ? l + n : (l >= n ? l - n : l);
  return l;
}

// Where the five stencil values along axis D of a tile cell lie in the input field: a value's offset, or -1
// for zero (outside the tile). li: the cell's coordinates in the input tile.
template <int D>
struct Stencil {
  long long at[5];
  __device__ Stencil(const BodyDev& b, const int sh[3], const int nn[3], int i0, int i1, int i2) {
    const int i[3] = {i0, i1, i2};
    int li[3];
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      li[a] = D == 0 ? in_local(i[a], sh[a], b.L[a], nn[a]) : i[a];
      if (D == 0 && a != D && (li[a] < 0 || li[a] >= b.L[a])) ok = false;
    }
    const long long sd = D == 0 ? 1 : (D == 1 ? b.L[0] : (long long)b.L[0] * b.L[1]);
    const long long base = li[0] + (long long)b.L[0] * (li[1] + (long long)b.L[1] * li[2]) - (long long)li[D] * sd;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const int l = in_local(li[D], k - 2, b.L[D], b.L[D] == nn[D] ? nn[D] : -1);
      at[k] = (ok && l >= 0 && l < b.L[D]) ? base + l * sd : -1;
    }
  }
  __device__ void load(const double* __restrict__ in, double p[5]) const {
#pragma unroll
    for (int k = 0; k < 5; ++k) p[k] = at[k] >= 0 ? in[at[k]] : 0.0;
  }
};

// phi as a multiple of 2^-62 (truncated): sums of phases on the integer pipe. False outside (-1, 1).
__device__ __forceinline__ bool phi_fixed(long long bits, long long& out) {
  const int e = (int)((unsigned long long)bits >> 52) & 0x7FF;  // value = 1.m x 2^(e - 1023)
  if (e >= 1023) return false;
  const unsigned long long m = ((unsigned long long)bits & 0xFFFFFFFFFFFFFULL) | (e ? 1ULL << 52 : 0ULL);
  const int up = e - 1023 + 10;  // m x 2^(e - 1023 - 52 + 62)
  const unsigned long long v = up >= 0 ? m << up : (up > -64 ? m >> -up : 0ULL);
  out = bits < 0 ? -(long long)v : (long long)v;
  return true;
}

// the body's list of bodies with overlapping tiles, ascending, by one warp
__device__ void build_list(BodyDev* bodies, int self, int nb, const Lat& lat, StepState* st) {
  const int lane = threadIdx.x & 31;
  int cnt = 0;
  for (int k0 = 0; k0 < nb; k0 += 32) {
    const int k = k0 + lane;
    const bool ov = k < nb && k != self && tiles_overlap(bodies[self], bodies[k], lat);
    const unsigned m = __ballot_sync(0xffffffffu, ov);
    const int at = cnt + __popc(m & ((1u << lane) - 1u));
    if (ov && at < MAXNB) bodies[self].nbl[at] = k;
    cnt += __popc(m);
  }
  if (lane == 0) {
    if (cnt > MAXNB) atomicOr(&st->err, E_NBLIST);
    bodies[self].nnb = min(cnt, MAXNB);
  }
}

// A body at rest without kinetics has nothing to copy: the halo check alone (a move or a turn may have put the
// field there), on the halo's cells alone: Z planes from z0 on of column t of its tile. (Not inlined: rare.)
__device__ __noinline__ void resting_halo(const TileSet& S, const BodyDev& b, unsigned t, int z0, int Z) {
  const int nn[3] = {S.lat.nx, S.lat.ny, S.lat.nz}, L0 = b.L[0], i1 = (int)(t / (unsigned)L0), i0 = (int)(t - (unsigned)i1 * L0);
  if (i1 >= b.L[1]) return;
  const size_t plane = (size_t)L0 * b.L[1];
  const double* const phi = S.arena + b.off + t;
  bool halo = false;
  for (int z = z0; z < min(z0 + Z, b.L[2]); ++z)
    if (tile_halo(b, nn, i0, i1, z)) halo |= (dbits(phi[plane * z]) << 1) > (dbits(PHI_EPS) << 1);
  if (halo) atomicOr(&S.st->err, E_TILE);
}

// Cells with a flat stencil keep their value (both face fluxes are u p with the same u, so the update is
// exactly zero); the others, the interface shell, are collected and updated in full warps. A body at rest
// changes nothing: its sweeps end at once, but for one copy of the field to where the kinetics reads it.
// Bound by the FP64 pipe (15 operations per interface cell). Measured on the four-sphere cluster (1.1 M tile
// cells): 27 us per sweep with a flat cell index and both signs of the velocity evaluated, 24, 23 and 30 here (z
// shares its loads between planes, x steps from plane to plane: 60 spheres 352 -> 334 us for the three).
template <bool B, int Z, int D, bool LAST>
__global__ void __launch_bounds__(TILE_T) k_sweep(const __grid_constant__ TileSet one, const TileSet* __restrict__ sets,
                                                  const int2* __restrict__ items) {
  int self;
  const TileSet& S = tile_set<B>(one, sets, items, self);
  const Lat& lat = S.lat;
  // the overlap lists follow the new origins (used by the kernels after the sweeps)
  if (D == 0 && blockIdx.x == 0 && blockIdx.y == 0) {
    if (threadIdx.x < 32) build_list(S.bodies, self, S.nb, lat, S.st);
    else if (threadIdx.x == 32) turn_body(S.bodies[self]);
  }
  const BodyDev& b = S.bodies[self];
  const int nn[3] = {lat.nx, lat.ny, lat.nz};
  const int L0 = b.L[0], L1 = b.L[1], L2 = b.L[2], z0 = blockIdx.y * Z;
  const unsigned plane = (unsigned)L0 * L1;
  if (z0 >= L2 || blockIdx.x * TILE_T >= plane) return;
  int sh[3] = {0, 0, 0};
  bool still = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // origins are unwrapped integers: take the shift as the minimum image of their difference
    if (b.L[a] < nn[a]) {
      int s = wrapi_near(b.o[a] - b.o_prev[a], nn[a]);
      if (s > nn[a] / 2) s -= nn[a];
      sh[a] = s;
    }
    still &= sh[a] == 0 && (dbits(b.V[a]) << 1) == 0 && (dbits(b.W[a]) << 1) == 0;
  }
  if (still && D != 0) return;
  if (D == 0 && still && !S.mpf) {
    resting_halo(S, b, blockIdx.x * TILE_T + threadIdx.x, z0, Z);
    return;
  }
  __shared__ TileList list;
  if (threadIdx.x == 0) list.n = 0;
  __syncthreads();
  // buffer 0 is the field, 1 and 2 are between the sweeps; the kinetics reads 1
  const double* const in = S.arena + b.off + (long long)D * b.sz;
  double* const out = S.arena + b.off + (long long)(LAST ? (S.mpf ? 1 : 0) : D + 1) * b.sz;
  const unsigned p0 = blockIdx.x * TILE_T, pt = p0 + threadIdx.x;
  const int i1 = (int)(pt / (unsigned)L0), i0 = (int)(pt - (unsigned)i1 * L0);
  // volume (sum phi, in units of 2^-62 below 1) and interface cells (0 < phi < 1) of what this thread writes in
  // the last sweep; a block's sum has room: whole ones are counted apart
  double big = 0.0;
  long long frac = 0;
  int ones = 0, shell = 0;
  bool halo = false;
  auto tally = [&](double v, int c0, int c1, int c2) {
    const long long vb = dbits(v);
    if ((vb << 1) == 0) return;
    long long fx;
    if (vb == dbits(1.0)) {
      ++ones;
    } else if (phi_fixed(vb, fx)) {
      frac += fx;
      if (frac >= 1LL << 62) {
        frac -= 1LL << 62;
        ++ones;
      }
    } else {
      big += v;
    }
    if (vb > dbits(PHI_EPS) && vb < dbits(1.0 - PHI_EPS)) ++shell;
    // the outer two layers must stay empty (they are the stencil halo); a moving body's upwind
    // scheme leaves a geometrically decaying tail ahead of its front, and the tile drops what
    // reaches past it, so values of at most PHI_EPS there are tolerated
    if ((vb << 1) > (dbits(PHI_EPS) << 1))
      halo |= tile_halo(b, nn, c0, c1, c2);
  };
  if (still) {
#pragma unroll
    for (int q = 0; q < Z; ++q)
      if (pt < plane && z0 + q < L2) {
        const size_t t = pt + (size_t)plane * (z0 + q);
        const double v = in[t];
        out[t] = v;
        tally(v, i0, i1, z0 + q);
      }
  } else {
    const bool on0 = pt < plane;
    auto visit = [&](int q, const double p[5]) {
      const long long c = dbits(p[2]);
      const bool flat = dbits(p[0]) == c && dbits(p[1]) == c && dbits(p[3]) == c && dbits(p[4]) == c;
      if (flat) {
        out[pt + (size_t)plane * (z0 + q)] = p[2];
        if (LAST) tally(p[2], i0, i1, z0 + q);
      }
      return !flat;
    };
    if constexpr (D == 2) {
      // the Z cells of a thread share the planes of their stencils: Z + 4 loads
      double v[Z + 4];
#pragma unroll
      for (int k = 0; k < Z + 4; ++k) {
        int l = z0 - 2 + k;
        if (L2 == nn[2]) l += l < 0 ? L2 : (l >= L2 ? -L2 : 0);
        v[k] = on0 && l >= 0 && l < L2 ? in[pt + (size_t)plane * l] : 0.0;
      }
#pragma unroll
      for (int q = 0; q < Z; ++q) {
        bool moves = false;
        if (on0 && z0 + q < L2) moves = visit(q, v + q);
        tile_append(list, moves, q * TILE_T + threadIdx.x);
      }
    } else {
      Stencil<D> st(b, sh, nn, on0 ? i0 : 0, on0 ? i1 : 0, z0);
#pragma unroll
      for (int q = 0; q < Z; ++q) {
        bool moves = false;
        if (on0 && z0 + q < L2) {
          if (q) {
            // a plane further, unless a shift in z can leave the tile there
            if (D == 0 && sh[2] != 0) {
              st = Stencil<D>(b, sh, nn, i0, i1, z0 + q);
            } else {
#pragma unroll
              for (int k = 0; k < 5; ++k) st.at[k] += st.at[k] >= 0 ? (long long)plane : 0LL;
            }
          }
          double p[5];
          st.load(in, p);
          moves = visit(q, p);
        }
        tile_append(list, moves, q * TILE_T + threadIdx.x);
      }
    }
    __syncthreads();
    constexpr int D1 = (D + 1) % 3, D2 = (D + 2) % 3;
    const double* const rt = S.rtab + (size_t)self * 3 * S.Lmax;
    const double vd = b.V[D], w1 = b.W[D1], w2 = b.W[D2];
    for (int e = threadIdx.x; e < list.n; e += TILE_T) {
      const int id = list.id[e];
      const unsigned pc = p0 + (id & (TILE_T - 1));
      const int c1 = (int)(pc / (unsigned)L0), c0 = (int)(pc - (unsigned)c1 * L0), c2 = z0 + id / TILE_T;
      const int ii[3] = {c0, c1, c2};
      double q[5];
      Stencil<D>(b, sh, nn, c0, c1, c2).load(in, q);
      // the face velocity u_d (the d-component of V + omega x r, r about X_prev) depends only on the two other
      // coordinates, so both faces of the cell share it; r_a = mimg(wrap(o_a + i_a) - Xprev_a) from the
      // per-body table built by k_bodies
      const double u = vd + (w1 * rt[D2 * S.Lmax + ii[D2]] - w2 * rt[D1 * S.Lmax + ii[D1]]);
      // face values, upwind + (1 - |u|) / 2 slope: with u >= 0 the left face's from cells 0 1 2 and the right
      // face's from 1 2 3, with u < 0 one cell further with the other sign
      const bool fwd = dbits(u) >= 0 || (dbits(u) << 1) == 0;
      const double r0 = fwd ? q[0] : q[1], r1 = fwd ? q[1] : q[2], r2 = fwd ? q[2] : q[3], r3 = fwd ? q[3] : q[4];
      const double h = 0.5 * (1.0 - fabs(u)), cf = fwd ? h : -h;
      const double d0 = r1 - r0, d1 = r2 - r1, d2 = r3 - r2;
      const double Fl = u * (r1 + cf * mc_slope(d0, d1)), Fr = u * (r2 + cf * mc_slope(d1, d2));
      const double v = q[2] - (Fr - Fl);
      out[pc + (size_t)plane * c2] = v;
      if (LAST) tally(v, c0, c1, c2);
    }
  }
  if (!(LAST || still)) return;
  // one FP64 atomic per block and sum (per-warp atomics on the same two words would queue up)
  if (__syncthreads_or(halo) && threadIdx.x == 0) atomicOr(&S.st->err, E_TILE);
  __shared__ long long wf[TILE_T / 32];
  __shared__ double wv[TILE_T / 32];
  __shared__ int wo[TILE_T / 32], wc[TILE_T / 32];
  const bool odd = __any_sync(0xffffffffu, big != 0.0);
  const double sv = odd ? dwarp_sum(big) : 0.0;
  // a thread's fraction is below 1 (2^62): halves of 2^31 add up in 64 bits
  long long lo = frac & 0x7FFFFFFFLL, hi = frac >> 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo += __shfl_xor_sync(0xffffffffu, lo, o);
    hi += __shfl_xor_sync(0xffffffffu, hi, o);
  }
  hi += lo >> 31;
  const int so = __reduce_add_sync(0xffffffffu, ones) + (int)(hi >> 31), sc = __reduce_add_sync(0xffffffffu, shell);
  if ((threadIdx.x & 31) == 0) {
    wf[threadIdx.x >> 5] = ((hi & 0x7FFFFFFFLL) << 31) | (lo & 0x7FFFFFFFLL);
    wv[threadIdx.x >> 5] = sv;
    wo[threadIdx.x >> 5] = so;
    wc[threadIdx.x >> 5] = sc;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    long long f = 0;
    double bv = 0.0;
    int bo = 0, bc = 0;
    for (int w = 0; w < TILE_T / 32; ++w) {
      f += wf[w];
      if (f >= 1LL << 62) {
        f -= 1LL << 62;
        ++bo;
      }
      if (wv[w] != 0.0) bv += wv[w];
      bo += wo[w];
      bc += wc[w];
    }
    bv += (double)bo + (double)f * 0x1p-62;
    if (bv != 0.0) atomicAdd(S.volacc + 2 * self, bv);
    if (bc != 0) atomicAdd(S.volacc + 2 * self + 1, (double)bc);
  }
}

// ---- MPF kinetics ------------------------------------------------------------------------------
// For body a at cell g: active phases = solids with phi > PHI_EPS at g or a face neighbour, plus the
// fluid if 1 - sum phi > PHI_EPS there; N = their number; explicit Euler step of
// phi_a += sum_b (M/N) [ s_ab (I_a - I_b) + sum_c (s_bc - s_ac) I_c + (D_a - D_b if 0<phi_a<1) ]
// with I = lap(phi) + (pi/eta)^2 phi, D_B = (V_B(0) - sum phi_B) / #{0 < phi_B < 1}, D_fluid = 0.

// phi at a cell of a tile given in tile-local coordinates l and its 6 face neighbours (order: self,
// +x, -x, +y, -y, +z, -z); periodic tile axes wrap, other axes read zero outside the tile
__device__ __forceinline__ void tile_val7(const double* __restrict__ buf, const int L[3], const int l[3], const int nn[3],
                                          double out[7]) {
  const long long s1 = L[0], s2 = (long long)L[0] * L[1];
  const bool in0 = l[0] >= 0 && l[0] < L[0] && l[1] >= 0 && l[1] < L[1] && l[2] >= 0 && l[2] < L[2];
  const long long c = l[0] + s1 * l[1] + s2 * l[2];
  out[0] = in0 ? buf[c] : 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int sg = 0; sg < 2; ++sg) {
      const int dlt = sg == 0 ? 1 : -1;
      int q[3] = {l[0], l[1], l[2]};
      q[a] += dlt;
      if (L[a] == nn[a]) q[a] = q[a] < 0 ? q[a] + nn[a] : (q[a] >= nn[a] ? q[a] - nn[a] : q[a]);
      const bool ok = q[0] >= 0 && q[0] < L[0] && q[1] >= 0 && q[1] < L[1] && q[2] >= 0 && q[2] < L[2];
      out[1 + 2 * a + sg] = ok ? buf[q[0] + s1 * q[1] + s2 * q[2]] : 0.0;
    }
  }
}

// volume-restoring term D = (V(0) - sum phi) / #{0 < phi < 1} of a body, 0 without interface cells
__device__ __forceinline__ double volume_term(const TileSet& S, int id) {
  const double cnt = S.volacc[2 * id + 1];
  return cnt > 0.0 ? (S.bodies[id].vol_ref - S.volacc[2 * id]) / cnt : 0.0;
}

// a listed body's tile coordinates of the cell at g; false if no cell of the 7-point stencil is in its tile
__device__ __forceinline__ bool near_tile(const BodyDev& o, const int g[3], const int nn[3], int lo[3]) {
  bool near = true;
  for (int a = 0; a < 3; ++a) {
    lo[a] = wrapi_near(g[a] - o.o[a], nn[a]);
    if (o.L[a] < nn[a]) {
      if (lo[a] > nn[a] - 2) lo[a] -= nn[a];  // just below the tile: keep the +1 neighbour reachable
      if (lo[a] < -1 || lo[a] > o.L[a]) near = false;
    }
  }
  return near;
}

// the general form, where another body is present in the cell's stencil (rare: a function of its own, so
// that its arrays do not cost the common form its registers)
__device__ __noinline__ double kinetics_shared(const TileSet& S, int self, const double pa[7], const int g[3],
                                               const int nn[3]) {
  const BodyDev* const bodies = S.bodies;
  const BodyDev& b = bodies[self];
  const double* const arena = S.arena;
  const KinParams& kp = S.kin;
  const long long eb = dbits(PHI_EPS);
  // active solids in ascending id order, with their 7-point values
  double vals[MAXACT][7];
  int dslot[MAXACT];  // body of each active phase
  int na = 0;
  int pos_self = -1;
  double sum[7] = {0, 0, 0, 0, 0, 0, 0};
  int k_nb = 0;
  for (int step = 0; step <= b.nnb; ++step) {
    int id;
    if (pos_self < 0 && (k_nb >= b.nnb || b.nbl[k_nb] > self)) id = self;
    else id = b.nbl[k_nb++];
    if (id == self) {
      pos_self = na;
      for (int k = 0; k < 7; ++k) {
        vals[na][k] = pa[k];
        sum[k] += pa[k];
      }
      dslot[na] = self;
      ++na;
      continue;
    }
    const BodyDev& o = bodies[id];
    int lo[3];
    if (!near_tile(o, g, nn, lo)) continue;
    double v7[7];
    tile_val7(arena + o.off + o.sz, o.L, lo, nn, v7);
    bool on = false;
    for (int k = 0; k < 7; ++k) on |= dbits(v7[k]) > eb;
    if (!on) continue;
    if (na < MAXACT - (pos_self < 0 ? 1 : 0)) {  // always keep a slot for self
      for (int k = 0; k < 7; ++k) {
        vals[na][k] = v7[k];
        sum[k] += v7[k];
      }
      dslot[na] = id;
      ++na;
    }
  }
  // sum >= 0, so the signed bit patterns order like the values
  const long long one_eb = dbits(1.0 - PHI_EPS);
  bool fl = false;
  for (int k = 0; k < 7; ++k) fl |= dbits(sum[k]) < one_eb;
  const int N = na + (fl ? 1 : 0);
  if (N <= 1) return pa[0];
  const double k2 = kp.k2;
  double I[MAXACT + 1], D[MAXACT + 1];
  for (int j = 0; j < na; ++j) {
    double lap = 0.0;
    for (int k = 1; k < 7; ++k) lap += vals[j][k];
    lap -= 6.0 * vals[j][0];
    I[j] = lap + k2 * vals[j][0];
    D[j] = volume_term(S, dslot[j]);
  }
  if (fl) {
    double lap = 0.0;
    for (int k = 1; k < 7; ++k) lap += 1.0 - sum[k];
    lap -= 6.0 * (1.0 - sum[0]);
    I[na] = lap + k2 * (1.0 - sum[0]);
    D[na] = 0.0;
  }
  const double s_sf = kp.s_sf, s_ss = kp.s_ss;
  auto sig = [&](int p, int q) { return (p == na || q == na) ? s_sf : s_ss; };
  const int a = pos_self;
  const bool in_if = dbits(pa[0]) > eb && dbits(pa[0]) < one_eb;
  double rate = 0.0;
  for (int bq = 0; bq < N; ++bq) {
    if (bq == a) continue;
    double term = sig(a, bq) * (I[a] - I[bq]);
    for (int gg = 0; gg < N; ++gg) {
      if (gg == a || gg == bq) continue;
      term += (sig(bq, gg) - sig(a, gg)) * I[gg];
    }
    if (in_if) term += D[a] - D[bq];
    rate += kp.mobN[N] * term;
  }
  return pa[0] + rate;
}

// One pass over the tile writes the cells that keep their value (0 with nothing around, 1 inside a body that
// no other tile touches) and collects the rest. Four-sphere cluster: 54 us with one cell per thread and a flat
// index (74 registers, 3 blocks per SM), 39 us here.
template <bool B, int Z>
__global__ void __launch_bounds__(TILE_T) k_kinetics(const __grid_constant__ TileSet one, const TileSet* __restrict__ sets,
                                                     const int2* __restrict__ items) {
  int self;
  const TileSet& S = tile_set<B>(one, sets, items, self);
  if (!S.mpf) return;
  const BodyDev& b = S.bodies[self];
  const Lat& lat = S.lat;
  const int nn[3] = {lat.nx, lat.ny, lat.nz};
  const int L0 = b.L[0], L1 = b.L[1], L2 = b.L[2], z0 = blockIdx.y * Z;
  const unsigned plane = (unsigned)L0 * L1, p0 = blockIdx.x * TILE_T, pt = p0 + threadIdx.x;
  if (z0 >= L2 || p0 >= plane) return;
  __shared__ TileList list;
  __shared__ double sD;
  if (threadIdx.x == 0) {
    list.n = 0;
    sD = volume_term(S, self);
  }
  __syncthreads();
  const double* const in = S.arena + b.off + b.sz;  // buffer 1: advected field
  double* const out = S.arena + b.off;              // buffer 0: new field
  const int nnb = b.nnb;
  const int i1 = (int)(pt / (unsigned)L0), i0 = (int)(pt - (unsigned)i1 * L0);
  // lateral neighbours: their offset from the cell, or none (outside the tile: zero); the column's own values
  // are kept as the planes go by
  const bool col = pt < plane;
  const double* const pc0 = in + pt;
  int side[4];
  bool has[4];
  {
    const bool px = L0 == nn[0], py = L1 == nn[1];
    has[0] = i0 + 1 < L0 || px;
    has[1] = i0 > 0 || px;
    has[2] = i1 + 1 < L1 || py;
    has[3] = i1 > 0 || py;
    side[0] = i0 + 1 < L0 ? 1 : 1 - L0;
    side[1] = i0 > 0 ? -1 : L0 - 1;
    side[2] = i1 + 1 < L1 ? L0 : L0 * (1 - L1);
    side[3] = i1 > 0 ? -L0 : L0 * (L1 - 1);
  }
  auto at = [&](int z) -> double {
    if (L2 == nn[2]) z = z < 0 ? z + L2 : (z >= L2 ? z - L2 : z);
    return col && z >= 0 && z < L2 ? pc0[(size_t)plane * z] : 0.0;
  };
  double below = at(z0 - 1), here = at(z0);
#pragma unroll
  for (int q = 0; q < Z; ++q) {
    const bool on = col && z0 + q < L2;
    const double above = at(z0 + q + 1);
    bool want = false;
    if (on) {
      const long long c = dbits(here);
      bool flat = dbits(below) == c && dbits(above) == c;
      const double* const h = pc0 + (size_t)plane * (z0 + q);
#pragma unroll
      for (int k = 0; k < 4; ++k) flat &= dbits(has[k] ? h[side[k]] : 0.0) == c;
      want = !(flat && (c == 0 || (c == dbits(1.0) && nnb == 0)));
      if (!want) out[pt + (size_t)plane * (z0 + q)] = here;
    }
    tile_append(list, want, q * TILE_T + threadIdx.x);
    below = here;
    here = above;
  }
  __syncthreads();
  const KinParams& kp = S.kin;
  const long long eb = dbits(PHI_EPS), one_eb = dbits(1.0 - PHI_EPS), neg0 = (long long)0x8000000000000000ULL;
  for (int e = threadIdx.x; e < list.n; e += TILE_T) {
    const int id = list.id[e];
    const unsigned pc = p0 + (id & (TILE_T - 1));
    const int c1 = (int)(pc / (unsigned)L0), c0 = (int)(pc - (unsigned)c1 * L0), c2 = z0 + id / TILE_T;
    const size_t t = pc + (size_t)plane * c2;
    const int l[3] = {c0, c1, c2};
    double pa[7];
    tile_val7(in, b.L, l, nn, pa);
    bool act_a = false;
#pragma unroll
    for (int k = 0; k < 7; ++k) act_a |= dbits(pa[k]) > eb;
    if (!act_a) {
      out[t] = pa[0];
      continue;
    }
    const int g[3] = {wrapi_near(b.o[0] + c0, nn[0]), wrapi_near(b.o[1] + c1, nn[1]), wrapi_near(b.o[2] + c2, nn[2])};
    // is any other body present in this cell's 7-point stencil?
    bool others = false;
    for (int k = 0; k < nnb && !others; ++k) {
      const BodyDev& o = S.bodies[b.nbl[k]];
      int lo[3];
      if (!near_tile(o, g, nn, lo)) continue;
      double v7[7];
      tile_val7(S.arena + o.off + o.sz, o.L, lo, nn, v7);
#pragma unroll
      for (int k2 = 0; k2 < 7; ++k2) others |= dbits(v7[k2]) > eb;
    }
    if (others) {
      out[t] = kinetics_shared(S, self, pa, g, nn);
      continue;
    }
    // one solid phase a and the fluid f = 1 - phi: N = 2 where the fluid is present at the cell or a
    // face neighbour, and then the rate is (M/2) [sigma_sf (I_a - I_f) + D_a (interface cells)]. With
    // lap = the 7-point Laplacian of phi, I_a = lap + k2 phi and I_f = -lap + k2 (1 - phi), so
    // I_a - I_f = 2 lap + k2 (2 phi - 1) (the same quantity as the general form, up to rounding). Presence of
    // the fluid (1 - phi > PHI_EPS) is tested on bit patterns.
    bool fl = false;
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      const long long bk = dbits(pa[k]);
      fl |= (bk == neg0 ? 0LL : bk) < one_eb;
    }
    if (!fl) {  // N = 1: no kinetics
      out[t] = pa[0];
      continue;
    }
    double lap = 0.0;
#pragma unroll
    for (int k = 1; k < 7; ++k) lap += pa[k];
    lap -= 6.0 * pa[0];
    double term = kp.s_sf * (2.0 * lap + kp.k2 * (2.0 * pa[0] - 1.0));
    if (dbits(pa[0]) > eb && dbits(pa[0]) < one_eb) term += sD;
    out[t] = pa[0] + kp.mobN[2] * term;
  }
}


// ---- dense read-out ----------------------------------------------------------------------------
__global__ void k_fill(double* out, long long N, double v) {
  long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n < N) out[n] = v;
}

// body >= 0: scatter that body's field; body < 0: 1 - sum of all bodies (fluid phase)
__global__ void k_phi_scatter(const BodyDev* bodies, const double* arena, double* out, Lat lat, int body) {
  const int self = body >= 0 ? body : blockIdx.y;
  const BodyDev& b = bodies[self];
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= b.sz) return;
  TileCell c = tile_cell(b, t, lat);
  const long long n = c.gx + (long long)lat.nx * (c.gy + (long long)lat.ny * c.gz);
  if (body >= 0) {
    out[n] = arena[b.off + t];
    return;
  }
  if (b.nnb && covered_by_lower_body(bodies, b, self, c.gx, c.gy, c.gz, lat)) return;
  double S = arena[b.off + t];
  for (int k = 0; k < b.nnb; ++k) {
    const BodyDev& o = bodies[b.nbl[k]];
    if (b.nbl[k] < self) continue;
    long long j = tile_index(o.o, o.L, c.gx, c.gy, c.gz, lat);
    if (j >= 0) S += arena[o.off + j];
  }
  out[n] = 1.0 - S;
}

// before the bodies are moved: every cell of their current tiles loses its flags, except that a
// solid cell keeps the solid bit under the owner id F_STALE, so the next flag pass does not count
// it as covered again
__global__ void k_clear_tile_flags(const BodyDev* bodies, uint16_t* flags, Lat lat) {
  const BodyDev& b = bodies[blockIdx.y];
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= b.sz) return;
  const TileCell c = tile_cell(b, t, lat);
  uint16_t& f = flags[c.gx + (long long)lat.nx * (c.gy + (long long)lat.ny * c.gz)];
  f = (f & F_SOLID) ? (uint16_t)(F_SOLID | F_STALE) : (uint16_t)0;
}

// after the flag pass at the new poses: cells still marked stale lie outside every new tile and
// are uncovered (their populations were zeroed while they were solid)
__global__ void k_clear_stale(uint16_t* flags, long long N) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n < N && flags[n] == (uint16_t)(F_SOLID | F_STALE)) flags[n] = 0;
}

__global__ void k_clear_cover(uint16_t* flags, long long N) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n < N && (flags[n] & F_COVER)) flags[n] &= (uint16_t)~F_COVER;
}

// ---- launchers ---------------------------------------------------------------------------------
static dim3 tile_grid(int max_tile, int nb) { return dim3((unsigned)((max_tile + 255) / 256), (unsigned)nb); }

void launch_rasterize(const Lat& lat, BodyDev* bodies, int nb, int max_tile, double* arena, double eta,
                      cudaStream_t s) {
  if (nb) k_rasterize<<<tile_grid(max_tile, nb), 256, 0, s>>>(bodies, arena, lat, eta);
}
void launch_neighbour_lists(BodyDev* bodies, int nb, const Lat& lat, StepState* st, cudaStream_t s) {
  if (nb) k_neighbour_lists<<<1, 256, 0, s>>>(bodies, nb, lat, st);
}
// launch a tile kernel template <bool B, ...> over a context's bodies or a batch's
static int sm_count() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}
static dim3 tile_blocks(const ChainLaunch& c, int z) {
  return dim3((unsigned)((c.max_xy + TILE_T - 1) / TILE_T), (unsigned)((c.max_z + z - 1) / z), (unsigned)c.bodies);
}
template <bool B, int Z>
static void flags_t(const ChainLaunch& c, int init, cudaStream_t s) {
  k_flags<B, Z><<<tile_blocks(c, Z), TILE_T, 0, s>>>(c.one, c.sets, c.items, init);
}
// the form of a tile launch: one context or a batch, planes per block
#define CBL_TILE_LAUNCH(fn, c, ...)                                                                 \
  do {                                                                                              \
    const bool four = tile_planes(c, sm_count()) == TILE_Z;                                         \
    if ((c).sets) {                                                                                 \
      if (four) fn<true, TILE_Z>(c, __VA_ARGS__);                                                   \
      else fn<true, 1>(c, __VA_ARGS__);                                                             \
    } else {                                                                                        \
      if (four) fn<false, TILE_Z>(c, __VA_ARGS__);                                                  \
      else fn<false, 1>(c, __VA_ARGS__);                                                            \
    }                                                                                               \
  } while (0)
void launch_flags(const ChainLaunch& c, int init, cudaStream_t s) {
  if (!c.bodies) return;
  CBL_TILE_LAUNCH(flags_t, c, init, s);
}
void launch_commit(StepState* st, ChainState* cs, cudaStream_t s) { k_commit<<<1, 1, 0, s>>>(st, cs); }
void launch_body_props(const Lat& lat, BodyDev* bodies, int nb, int max_tile, double* arena, double* scratch,
                       cudaStream_t s) {
  if (!nb) return;
  cudaMemsetAsync(scratch, 0, sizeof(double) * 9 * nb, s);
  k_body_props<<<tile_grid(max_tile, nb), 256, 0, s>>>(bodies, arena, scratch, lat, 0);
  k_body_props_finish<<<(nb + 127) / 128, 128, 0, s>>>(bodies, nb, scratch, lat, 0);
  cudaMemsetAsync(scratch, 0, sizeof(double) * 9 * nb, s);
  k_body_props<<<tile_grid(max_tile, nb), 256, 0, s>>>(bodies, arena, scratch, lat, 1);
  k_body_props_finish<<<(nb + 127) / 128, 128, 0, s>>>(bodies, nb, scratch, lat, 1);
}
void launch_repulsion(const ChainLaunch& c, cudaStream_t s) {
  if (!c.bodies) return;
  const int nsm = sm_count();
  const unsigned tile = (unsigned)(((long long)c.max_xy * c.max_z + 255) / 256);
  // a few waves in all. Only the points near a contact have work, and every block repeats the cull, so many
  // bodies get few blocks each (128 bodies of a batch: 140 us with a block for four chunks of the tile, 12 now)
  const dim3 g(std::min(tile, (unsigned)std::max(8, 4 * nsm / c.bodies)), 1, (unsigned)c.bodies);
  if (c.sets) k_repulsion<true><<<g, REP_T, 0, s>>>(c.one, c.sets, c.items);
  else k_repulsion<false><<<g, REP_T, 0, s>>>(c.one, nullptr, nullptr);
}
void launch_bodies(const ChainLaunch& c, cudaStream_t s) {
  if (!c.bodies) return;
  const dim3 g(1, 1, (unsigned)c.bodies);
  if (c.sets) k_bodies<true><<<g, BODY_T, 0, s>>>(c.one, c.sets, c.items);
  else k_bodies<false><<<g, BODY_T, 0, s>>>(c.one, nullptr, nullptr);
}
void launch_finish(double* mass_part, unsigned n_mass_part, StepState* st, ChainState* cs, cudaStream_t s) {
  k_finish<<<1, 256, 0, s>>>(mass_part, n_mass_part, st, cs);
}
template <bool B, int Z>
static void advect_t(const ChainLaunch& c, cudaStream_t s) {
  const dim3 g = tile_blocks(c, Z);
  k_sweep<B, Z, 0, false><<<g, TILE_T, 0, s>>>(c.one, c.sets, c.items);
  k_sweep<B, Z, 1, false><<<g, TILE_T, 0, s>>>(c.one, c.sets, c.items);
  k_sweep<B, Z, 2, true><<<g, TILE_T, 0, s>>>(c.one, c.sets, c.items);
}
void launch_advect(const ChainLaunch& c, cudaStream_t s) {
  if (!c.bodies) return;
  CBL_TILE_LAUNCH(advect_t, c, s);
}
KinParams kin_params(const PhysParams& pp) {
  KinParams kp;
  kp.k2 = PI * PI / (pp.eta * pp.eta);
  kp.s_sf = pp.sigma_sf;
  kp.s_ss = pp.sigma_ss;
  for (int k = 0; k < MAXACT + 2; ++k) kp.mobN[k] = k ? pp.mobility / k : 0.0;
  return kp;
}
template <bool B, int Z>
static void kinetics_t(const ChainLaunch& c, cudaStream_t s) {
  k_kinetics<B, Z><<<tile_blocks(c, Z), TILE_T, 0, s>>>(c.one, c.sets, c.items);
}
void launch_kinetics(const ChainLaunch& c, cudaStream_t s) {
  if (!c.bodies) return;
  CBL_TILE_LAUNCH(kinetics_t, c, s);
}
void launch_phi_dense(const Lat& lat, const BodyDev* bodies, int nb, int max_tile, const double* arena, int body,
                      double* out, cudaStream_t s) {
  k_fill<<<(unsigned)((lat.N + 255) / 256), 256, 0, s>>>(out, lat.N, body >= 0 ? 0.0 : 1.0);
  if (!nb) return;
  dim3 g = tile_grid(max_tile, body >= 0 ? 1 : nb);
  k_phi_scatter<<<g, 256, 0, s>>>(bodies, arena, out, lat, body);
}

void launch_clear_tile_flags(const Lat& lat, const BodyDev* bodies, int nb, int max_tile, uint16_t* flags,
                             cudaStream_t s) {
  if (nb) k_clear_tile_flags<<<tile_grid(max_tile, nb), 256, 0, s>>>(bodies, flags, lat);
}
__global__ void k_reset_member_boxes(int* mbox, int nb) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < MBOX_N * nb) {
    const int e = k % MBOX_N;
    mbox[k] = e < 3 ? INT_MAX : (e < 6 ? INT_MIN : 0);
  }
}
void launch_reset_member_boxes(int* mbox, int nb, cudaStream_t s) {
  if (nb) k_reset_member_boxes<<<(MBOX_N * nb + 255) / 256, 256, 0, s>>>(mbox, nb);
}
void launch_clear_cover(const Lat& lat, uint16_t* flags, cudaStream_t s) {
  k_clear_cover<<<(unsigned)((lat.N + 255) / 256), 256, 0, s>>>(flags, lat.N);
}
void launch_clear_stale(const Lat& lat, uint16_t* flags, cudaStream_t s) {
  k_clear_stale<<<(unsigned)((lat.N + 255) / 256), 256, 0, s>>>(flags, lat.N);
}

}  // namespace cbl
