// Moment pass of the bulk fluid (lbm_variant 3), included by lbm.cu in the namespace of a velocity set.
//
// At tau = 1 the relaxation drops the old population: f*_i = f_eq,i(rho, v) + S_i(v, F) is a function
// of the density, the momentum and the force alone (Eqs. lb_collision, distribution_eq, guo_forcing),
// and F a function of psi (Eq. benzi_force). A cell without a solid neighbour therefore needs no
// stored populations: this pass carries (rho, m = sum c_i f_i) and psi of the post-streaming state,
// forms f* in shared memory, streams it there, and stores the next (rho, m) and psi. That is 42 bytes
// per cell and step (16 + 4 read, 16 + 4 written, 2 flag) against the 234 of the split pass, which
// pulls 19 populations twice and stores them once.
//
// Where populations are still stored: the fluid cells next to a solid (F_NEAR: bounce-back, wall
// terms, collided by k_collide_near before this pass) and every cell of the bricks (4 x 4 x 4 cells)
// within 3 cells of one, which this pass stores beside the moments. k_mom_close pulls them at the end
// of the step: psi of the next step's near cells, and the moments around every cell whose obstacle
// flag changed (the refill rewrites populations there). A flag that changes where populations are
// not stored (a body moving by cells in one step) makes k_mom_fill write all of them first; the same
// kernel serves every reader of populations outside a step (cbl_read_populations, cbl_save,
// cbl_move_bodies, a batch).
//
// Index convention: within step t (parity q) the moments M[q] and psi[q] are those after streaming at t,
// f*_t is the buffer the step writes, map[q] names the bricks in which f*_t is stored.

// solid cells carry this density in M
constexpr float MOM_SOLID = -1e30f;

// Every operation below is rounded as written (no contraction is left to the compiler): the pass, the
// fill and each unrolled copy of the loop give the same bits for the same cell, so populations read or
// saved between steps are those the next step pulls.

// c . (x, y, z) for a direction with components -1, 0, 1
__device__ __forceinline__ float dir_dot(int i, float x, float y, float z) {
  float r = 0.0f;
  bool set = false;
  const int c[3] = {cx_of(i), cy_of(i), cz_of(i)};
  const float v[3] = {x, y, z};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (!c[a]) continue;
    const float t = c[a] > 0 ? v[a] : -v[a];
    r = set ? __fadd_rn(r, t) : t;
    set = true;
  }
  return r;
}

// force from opposite differences of psi: the weight of a class of directions (faces, edges, corners)
// multiplies the sum of its differences
template <typename PsiAt>
__device__ __forceinline__ void mom_force(const PsiAt& psi_at, const PhysParams& pp, float& Fx, float& Fy, float& Fz) {
  const float ps = psi_at(0);
  float f[3] = {0, 0, 0}, e[3] = {0, 0, 0}, k[3] = {0, 0, 0};
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const float d = __fsub_rn(psi_at(i), psi_at(i + 1));
    const int c[3] = {cx_of(i), cy_of(i), cz_of(i)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float& s = i <= 6 ? f[a] : (i <= 18 ? e[a] : k[a]);
      const bool first = i <= 6 || i == (a == 2 ? 11 : 7) || i == 19;  // of the class along this axis
      if (c[a] > 0) s = first ? d : __fadd_rn(s, d);
      if (c[a] < 0) s = first ? -d : __fsub_rn(s, d);
    }
  }
  const float w1 = (float)w_of(1), w2 = (float)w_of(7), w3 = (float)w_of(Q - 1);
  const float mG = __fmul_rn(-pp.G_f, ps);
  float F[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float s = __fmaf_rn(w1, f[a], __fmul_rn(w2, e[a]));
    if constexpr (Q == 27) s = __fmaf_rn(w3, k[a], s);
    F[a] = __fmaf_rn(mG, s, pp.ext_f[a]);
  }
  Fx = F[0];
  Fy = F[1];
  Fz = F[2];
}

// velocity with the half-force shift (Eq. fluid_velocity) and the post-collision values at tau = 1,
// f*_i = w_i [b + 4.5 (c.v)(c.(rho v + F)) + 3 c.(rho v + F / 2)], b = rho (1 - 1.5 v.v) - 1.5 v.F,
// handed to sink(i, f*_i) in direction order; opposite directions share the even part
template <typename Sink>
__device__ __forceinline__ void mom_values(const float4& m, float Fx, float Fy, float Fz, float& vx, float& vy,
                                           float& vz, const Sink& sink) {
  vx = vy = vz = 0.0f;
  if (m.x > 0.0f) {
    const float ir = 1.0f / m.x;
    vx = __fmul_rn(__fmaf_rn(0.5f, Fx, m.y), ir);
    vy = __fmul_rn(__fmaf_rn(0.5f, Fy, m.z), ir);
    vz = __fmul_rn(__fmaf_rn(0.5f, Fz, m.w), ir);
  }
  // rho v, from v as the population form of the collision has it (rho <= 0 leaves v = 0)
  const float qx = __fmul_rn(m.x, vx), qy = __fmul_rn(m.x, vy), qz = __fmul_rn(m.x, vz);
  const float gx = __fadd_rn(qx, Fx), gy = __fadd_rn(qy, Fy), gz = __fadd_rn(qz, Fz);
  const float px = __fmul_rn(3.0f, __fmaf_rn(0.5f, Fx, qx)), py = __fmul_rn(3.0f, __fmaf_rn(0.5f, Fy, qy)),
              pz = __fmul_rn(3.0f, __fmaf_rn(0.5f, Fz, qz));
  // b = rho - 1.5 v . (rho v + F)
  const float b = __fmaf_rn(-1.5f, __fmaf_rn(vx, gx, __fmaf_rn(vy, gy, __fmul_rn(vz, gz))), m.x);
  const float ux = __fmul_rn(4.5f, vx), uy = __fmul_rn(4.5f, vy), uz = __fmul_rn(4.5f, vz);
  sink(0, __fmul_rn(wgt<float>(0), b));
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const float cu = dir_dot(i, ux, uy, uz), cg = dir_dot(i, gx, gy, gz), cp = dir_dot(i, px, py, pz);
    const float w = wgt<float>(i);
    const float s = __fmul_rn(w, __fmaf_rn(cu, cg, b));
    sink(i, __fmaf_rn(w, cp, s));
    sink(i + 1, __fmaf_rn(-w, cp, s));
  }
}

// density and momentum of streamed populations (momentum over opposite pairs, as fluid_velocity)
__device__ __forceinline__ float4 moments_of(const float fi[Q]) {
  float rho = fi[0], m[3] = {0, 0, 0};
#pragma unroll
  for (int i = 1; i < Q; ++i) rho = __fadd_rn(rho, fi[i]);
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const float d = __fsub_rn(fi[i], fi[i + 1]);
    const int c[3] = {cx_of(i), cy_of(i), cz_of(i)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (c[a] > 0) m[a] = i <= 6 ? d : __fadd_rn(m[a], d);
      if (c[a] < 0) m[a] = __fsub_rn(m[a], d);
    }
  }
  return make_float4(rho, m[0], m[1], m[2]);
}

// psi = 1 - exp(-rho / rho0) (Eq. mean_field_potential); rho0 = 1, the paper's, needs no division
__device__ __forceinline__ float mom_psi(float rho, float rho0) {
  return 1.0f - expf(rho0 == 1.0f ? -rho : -rho / rho0);
}

__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Geometry of a block of the moment pass: a column of 32 x TY cells, its one-cell ring (the cells
// whose f* the column pulls) and the two-cell ring of psi that their force needs. One thread per cell
// of column and ring.
template <int TY>
struct MomTile {
  static constexpr int EX = 34, EY = TY + 2, NE = EX * EY;
  static constexpr int PX = 36, PY = TY + 4, NP = PX * PY;
  static constexpr int NT = 32 * TY + ((NE - 32 * TY + 31) / 32) * 32;
  static constexpr int FS = 4, PS = 4;  // planes of f* and of psi in shared memory
  static constexpr size_t smem = sizeof(float) * ((size_t)FS * (Q - 1) * NE + (size_t)PS * NP);
};

// A block marches its column through sz planes. For plane p it forms f* of column and ring from M and
// psi (both fetched one plane ahead: M into registers, psi by asynchronous copies into shared memory),
// passes the block's one barrier, and then completes plane p - 1: every cell pulls its 18 (26)
// sources from the three newest planes in shared memory, in the order of the population form, and
// stores (rho, m) and psi of the next step. The loop is unrolled over the four planes of the rings, so
// that every shared-memory address is a constant offset.
// Bound by instruction issue (ring cells are computed twice: x 1.375 in warps at TY = 8).
template <typename S>
struct MomArgs {
  S *fa, *fb;
  const uint16_t* flags;
  float *psi_a, *psi_b;
  MomDev md;
  double* mass_part;
  const StepState* st;
  double *diag_rho, *diag_vel;
};

// FETCH: f* of the cells next to a solid is fetched a plane ahead. Loaded where it is used, a plane that
// holds such a cell waits for memory once more; fetched, every plane pays for the look ahead. Spheres of
// R 5 to 24 in boxes of 64 to 128 cells (nearly every column meets one): 2600 -> 1812 us per step of 64. One
// 256^3 lattice with four of R = 24: 335 -> 347 us; 60 spheres in 224^3: 439 -> 424 of a step of 1240. A batch
// fetches, a single lattice does not.
template <typename S, int TY, bool FETCH>
__device__ __forceinline__ void mom_column(const MomArgs<S>& a, const Lat& lat, const PhysParams& pp, int x0, int y0,
                                           int zb, int sz, unsigned slot_id, float* __restrict__ smem) {
  using T = MomTile<TY>;
  float* const sf = smem;                                   // [FS][Q - 1][NE]
  float* const sp = smem + (size_t)T::FS * (Q - 1) * T::NE;  // [PS][NP]
  const MomDev& md = a.md;
  const uint16_t* __restrict__ flags = a.flags;
  double* __restrict__ diag_rho = a.diag_rho;
  double* __restrict__ diag_vel = a.diag_vel;
  const int parity = a.st->parity, diag = a.st->diag;
  S* const dst = parity ? a.fa : a.fb;
  const float* __restrict__ psi = parity ? a.psi_b : a.psi_a;
  float* __restrict__ psi_next = parity ? a.psi_a : a.psi_b;
  const float4* __restrict__ M = md.M(parity);
  float4* __restrict__ M_next = md.M(parity ^ 1);
  const unsigned char* __restrict__ map = md.map(parity);
  const size_t N = (size_t)lat.Ns;
  const int tid = threadIdx.x;
  const int planes = min(sz, lat.nz - zb);
  // this thread's cell of the column (tid < 32 TY) or of the ring
  int ex, ey;
  bool ext = true;
  if (tid < 32 * TY) {
    ex = (tid & 31) + 1;
    ey = (tid >> 5) + 1;
  } else {
    int r = tid - 32 * TY;
    if (r < 2 * T::EX) {
      ey = r < T::EX ? 0 : TY + 1;
      ex = r < T::EX ? r : r - T::EX;
    } else {
      r -= 2 * T::EX;
      ex = (r & 1) * (T::EX - 1);
      ey = 1 + (r >> 1);
      if (ey > TY) {
        ext = false;
        ex = ey = 0;
      }
    }
  }
  const bool own = tid < 32 * TY && x0 + ex - 1 < lat.nx && y0 + ey - 1 < lat.ny;
  const int x = wrapi(x0 - 1 + ex, lat.nx), y = wrapi(y0 - 1 + ey, lat.ny);
  const unsigned nxy = (unsigned)lat.nx * (unsigned)lat.ny, col = (unsigned)x + (unsigned)lat.nx * (unsigned)y;
  const int e = ey * T::EX + ex, pe = (ey + 1) * T::PX + ex + 1;
  const unsigned char* const mapc = map + md.brick(x >> BRICK_BITS, y >> BRICK_BITS, 0);
  const unsigned mapz = (unsigned)(md.nbx * md.nby);
  // psi columns this thread copies (at most two)
  unsigned pc[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int q = min(tid + k * T::NT, T::NP - 1);
    pc[k] = (unsigned)wrapi(x0 - 2 + q % T::PX, lat.nx) + (unsigned)lat.nx * (unsigned)wrapi(y0 - 2 + q / T::PX, lat.ny);
  }
  static_assert(T::NP <= 2 * T::NT, "two psi cells per thread");
  // first cell of plane z in [-2, nz + 1] (nz >= 4: one wrap)
  auto plane0 = [&](int z) { return nxy * (unsigned)(z < 0 ? z + lat.nz : (z >= lat.nz ? z - lat.nz : z)); };
  // psi plane k is z = zb - 2 + k, in slot k mod 4
  auto copy_psi = [&](int k, int slot) {
    if (k <= planes + 3) {
      const unsigned base = plane0(zb - 2 + k);
      if (tid < T::NP) cp_async4(sp + slot * T::NP + tid, psi + (base + pc[0]));
      if (tid + T::NT < T::NP) cp_async4(sp + slot * T::NP + tid + T::NT, psi + (base + pc[1]));
    }
    cp_async_commit();
  };
  copy_psi(0, 0);
  copy_psi(1, 1);
  copy_psi(2, 2);
  unsigned nq = col + plane0(zb - 1), nq1 = col + plane0(zb);  // cell of the plane being computed, of the next
  float4 m = M[nq];
  // flags of the plane being computed, of the one before and (FETCH) the one after
  uint16_t fl = flags[nq], fl_prev = 0, fl_next = FETCH ? flags[nq1] : (uint16_t)0;
  float f0 = 0.0f;
  bool brick = mapc[mapz * ((unsigned)zb >> BRICK_BITS)];  // populations are stored in the cell's brick
  MassAcc<float> mass;
  float* const fe = sf + e;
  const float* const pe0 = sp + pe;
  // f* of a cell next to a solid (k_collide_near stored it), fetched into its place in shared memory behind
  // the completion of the plane before. Halves arrive as the aligned word that holds them.
  auto fetch_near = [&](float* s, unsigned n) {
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const size_t k = (size_t)i * N + n;
      cp_async4(s + (i - 1) * T::NE, sizeof(S) == 2 ? dst + (k & ~(size_t)1) : dst + k);
    }
  };
  if (FETCH && ext && (fl & (F_SOLID | F_NEAR)) == F_NEAR) fetch_near(fe, nq);
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  // plane j is z = zb - 1 + j; planes 0 and planes + 1 are only pulled from. C = j mod 4.
  auto plane = [&](auto ic, const int j) {
    constexpr int C = decltype(ic)::value, SP = (C + 3) & 3, SU = (C + 2) & 3;  // slots of j, j - 1, j - 2
    copy_psi(j + 3, SP);
    const unsigned n = nq;
    const float4 mc = m;
    const uint16_t fc = fl;
    if (j <= planes) {
      if constexpr (FETCH) {
        nq = nq1;
        m = M[nq];
        fl = fl_next;
        nq1 = col + plane0(zb + min(j, planes - 1) + 1);
        fl_next = flags[nq1];
      } else {
        nq = col + plane0(zb + j);
        m = M[nq];
        fl = flags[nq];
      }
    }
    const float f0_prev = f0;
    const bool mine = own && j >= 1 && j <= planes;
    float* const s = fe + C * (Q - 1) * T::NE;
    if (fc & (F_SOLID | F_NEAR)) {
      if (fc & F_SOLID) {
        if (mine && diag) {
          diag_rho[n] = 0.0;
          diag_vel[3 * (size_t)n] = 0.0;
          diag_vel[3 * (size_t)n + 1] = 0.0;
          diag_vel[3 * (size_t)n + 2] = 0.0;
        }
      } else if (ext) {
        f0 = St<S>::ldv(dst, (size_t)n, 0);  // (used a plane later)
        if constexpr (!FETCH) {
#pragma unroll
          for (int i = 1; i < Q; ++i) s[(i - 1) * T::NE] = St<S>::ldv(dst, (size_t)i * N + n, i);
        } else if constexpr (sizeof(S) == 2) {
          cp_async_wait<0>();
#pragma unroll
          for (int i = 1; i < Q; ++i) {
            const unsigned w = __float_as_uint(s[(i - 1) * T::NE]);
            s[(i - 1) * T::NE] = St<S>::from_raw((unsigned short)(((size_t)i * N + n) & 1 ? w >> 16 : w), i);
          }
        }
      }
    } else if (ext) {
      auto psi_at = [&](int i) -> float {
        const int slot = cz_of(i) > 0 ? SU : (cz_of(i) < 0 ? C : (C + 1) & 3);
        return pe0[slot * T::NP + cy_of(i) * T::PX + cx_of(i)];
      };
      float Fx, Fy, Fz, vx, vy, vz;
      mom_force(psi_at, pp, Fx, Fy, Fz);
      mom_values(mc, Fx, Fy, Fz, vx, vy, vz, [&](int i, float v) {
        const float r = St<S>::rt(v, i);
        if (i == 0) f0 = r;
        else s[(i - 1) * T::NE] = r;
      });
      if (mine) {
        if (brick) {
          St<S>::st(dst, (size_t)n, 0, f0);
#pragma unroll
          for (int i = 1; i < Q; ++i) St<S>::st(dst, (size_t)i * N + n, i, s[(i - 1) * T::NE]);
        }
        mass.add(mc.x);
        if (diag) {
          diag_rho[n] = (double)mc.x;
          diag_vel[3 * (size_t)n] = (double)vx;
          diag_vel[3 * (size_t)n + 1] = (double)vy;
          diag_vel[3 * (size_t)n + 2] = (double)vz;
        }
      }
    }
    if (j >= 1 && ((zb + j) & ((1 << BRICK_BITS) - 1)) == 0 && j < planes) brick = mapc[mapz * ((unsigned)(zb + j) >> BRICK_BITS)];
    cp_async_wait<0>();
    // the one barrier per plane: f* of this plane and psi of the plane after next are in place. The planes
    // of f* that the slowest warp still pulls (j - 2 .. j) and the one the fastest writes next (j + 1)
    // are four different ones; psi that is overwritten next was read before this barrier.
    __syncthreads();
    // into the plane of f* that was last pulled from before this barrier
    if (FETCH && j <= planes && ext && (fl & (F_SOLID | F_NEAR)) == F_NEAR) fetch_near(fe + ((C + 1) & 3) * (Q - 1) * T::NE, nq);
    if (j >= 2 && own) {
      float fi[Q];
      fi[0] = f0_prev;
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const int slot = cz_of(i) > 0 ? SU : (cz_of(i) < 0 ? C : SP);
        fi[i] = fe[(slot * (Q - 1) + i - 1) * T::NE - cy_of(i) * T::EX - cx_of(i)];
      }
      float4 r = moments_of(fi);
      const unsigned t = col + nxy * (unsigned)(zb + j - 2);
      psi_next[t] = mom_psi(r.x, pp.rho0_f);
      if (fl_prev & F_SOLID) r = make_float4(MOM_SOLID, 0.0f, 0.0f, 0.0f);
      M_next[t] = r;
    }
    fl_prev = fc;
  };
  const int last = planes + 2;
  for (int j = 0; j < last; j += 4) {
    plane(std::integral_constant<int, 0>{}, j);
    if (j + 1 < last) plane(std::integral_constant<int, 1>{}, j + 1);
    if (j + 2 < last) plane(std::integral_constant<int, 2>{}, j + 2);
    if (j + 3 < last) plane(std::integral_constant<int, 3>{}, j + 3);
  }
  add_mass_slot(a.mass_part, mass, slot_id);
}

// at the start of a step: the next step's brick map is empty (it was last read in the step before). Share
// k of n threads.
__device__ __forceinline__ void mom_reset(const MomDev& md, int parity, unsigned k, unsigned n) {
  unsigned char* const map = md.map(parity ^ 1);
  const unsigned bricks = md.bricks();
  for (; k < bricks; k += n) map[k] = 0;
}

template <typename S, int TY, int MINB>
__global__ void __launch_bounds__(MomTile<TY>::NT, MINB) k_mom(const MomArgs<S> a, const Lat lat, const PhysParams pp, int sz) {
  extern __shared__ __align__(16) float mom_smem[];
  const unsigned blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  mom_reset(a.md, a.st->parity, blk * MomTile<TY>::NT + threadIdx.x, gridDim.x * gridDim.y * gridDim.z * MomTile<TY>::NT);
  mom_column<S, TY, false>(a, lat, pp, blockIdx.x * 32, blockIdx.y * TY, blockIdx.z * sz, sz, blk, mom_smem);
}

// The moment pass over a batch: one persistent launch (as k_batch_lbm: every block resident, work items
// from a device queue, one bounded grid barrier). Phase 0: the cells next to a solid of every instance,
// near_items each; phase 1: the columns, sz planes each. The instance's entry is copied to shared
// memory and phase 0 kept out of line: with the table read from global memory and both phases in one
// body, 50 words spilled. 64 pairs of spheres, 54 M cells on this pass: 1812 us (k_mom's rate on
// 256^3 would give 1000; the near cells, and box sides that are no multiple of 32, take the rest).
template <typename S>
__device__ __noinline__ float batch_near_item(const BatchInst& I, unsigned k, unsigned n) {
  mom_reset(I.md, I.st->parity, k, n);
  return near_cells<S, true>((S*)I.fa, (S*)I.fb, I.flags, (const float*)I.psi, (const float*)I.psi2, I.bodies, I.st,
                             I.diag_rho, I.diag_vel, I.blist, I.lat, I.pp, (RhoPsi<float>*)I.nbuf, k, n);
}
template <typename S, int TY, int MINB>
__global__ void __launch_bounds__(MomTile<TY>::NT, MINB)
    k_batch_mom(const BatchInst* __restrict__ tab, int ninst, long long items, BatchCtl* ctl, int sz) {
  constexpr int NT = MomTile<TY>::NT;
  extern __shared__ __align__(16) float mom_smem[];
  __shared__ BatchInst I;
  __shared__ long long s_item;
  __shared__ int s_inst;
  // enough for the few thousand cells next to a pair of spheres, more where there are blocks to spare
  const int near_items = min(max(8, (int)gridDim.x / ninst), 32);
  for (;;) {
    if (threadIdx.x == 0) s_item = (long long)atomicAdd(&ctl->queue[0], 1ull);
    __syncthreads();
    const long long item = s_item;
    __syncthreads();  // s_item is written again in the next round
    if (item >= (long long)ninst * near_items) break;
    const BatchInst& J = tab[item / near_items];
    const float m = batch_near_item<S>(J, (unsigned)(item % near_items) * NT + threadIdx.x, near_items * NT);
    add_mass_slot(J.mass_part, m, (unsigned)item);
  }
  if (!grid_barrier(ctl)) return;
  long long item0 = 0, item1 = 0;  // items of the instance in I
  for (;;) {
    if (threadIdx.x == 0) s_item = (long long)atomicAdd(&ctl->queue[1], 1ull);
    __syncthreads();
    const long long item = s_item;
    if (item >= items) return;
    if (item < item0 || item >= item1) {
      for (int k = threadIdx.x; k < ninst; k += NT)
        if (tab[k].item0 <= item && (k + 1 == ninst || tab[k + 1].item0 > item)) s_inst = k;
      __syncthreads();
      static_assert(sizeof(BatchInst) % sizeof(long long) == 0, "copied in words of eight bytes");
      for (int k = threadIdx.x; k < (int)(sizeof(BatchInst) / sizeof(long long)); k += NT)
        reinterpret_cast<long long*>(&I)[k] = reinterpret_cast<const long long*>(tab + s_inst)[k];
      __syncthreads();
      item0 = I.item0;
      item1 = item0 + (long long)I.tiles[0] * I.tiles[1] * I.tiles[2];
    }
    const int k = (int)(item - item0);
    const int tx = I.tiles[0], ty = I.tiles[1], bx = k % tx, by = (k / tx) % ty, bz = k / (tx * ty);
    const MomArgs<S> a{(S*)I.fa, (S*)I.fb, I.flags, (float*)I.psi, (float*)I.psi2, I.md, I.mass_part, I.st,
                       I.diag_rho, I.diag_vel};
    mom_column<S, TY, true>(a, I.lat, I.pp, bx * 32, by * TY, bz * sz, sz, (unsigned)k, mom_smem);
    __syncthreads();  // s_item, I and the planes in shared memory are written again
  }
}

// a solid cell's populations are zero in both buffers, from here or from the step that covered it on: a cell
// that is uncovered starts empty
template <typename S>
__device__ __forceinline__ void zero_populations(S* fa, S* fb, const Lat& lat, unsigned n) {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    St<S>::st(fa, (size_t)i * (size_t)lat.Ns + n, i, 0.0f);
    St<S>::st(fb, (size_t)i * (size_t)lat.Ns + n, i, 0.0f);
  }
}

// moments and psi of every cell from complete populations (after initialisation, a load, a move): the
// entry into the moment pass
template <typename S>
__global__ void __launch_bounds__(128) k_mom_enter(S* fa, S* fb, const StepState* __restrict__ st, const uint16_t* __restrict__ flags,
                                                   float* __restrict__ psi_a, float* __restrict__ psi_b, MomDev md,
                                                   Lat lat, float rho0_f) {
  const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 4 + (threadIdx.x >> 5), z = blockIdx.z;
  const int parity = st->parity;
  {
    // every population is stored; the bricks of the step to come are marked by k_mom_close
    const unsigned k = threadIdx.x + 128u * (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z));
    if (k < md.bricks()) {
      md.map(parity)[k] = 0;
      md.map(parity ^ 1)[k] = 1;
    }
  }
  if (x >= lat.nx || y >= lat.ny) return;
  const S* const f = parity ? fb : fa;
  const Cell c = make_cell(x, y, z, lat);
  const uint16_t fl = flags[c.n];
  if (fl & F_SOLID) {
    md.M(parity)[c.n] = make_float4(MOM_SOLID, 0.0f, 0.0f, 0.0f);
    zero_populations<S>(fa, fb, lat, c.n);
    return;
  }
  float fi[Q];
  unsigned sl;
  pull<S>(f, flags, lat, c, (long long)c.n, fi, sl, fl);
  const float4 m = moments_of(fi);
  md.M(parity)[c.n] = m;
  (parity ? psi_b : psi_a)[c.n] = mom_psi(m.x, rho0_f);
}

// Populations of every cell in whose brick they are not stored, from the moments and psi of the step
// that made them. next = 1: inside a step (the parity has not flipped), and then only if a flag
// changed outside the stored bricks; next = 0: between steps.
template <typename S>
__device__ __forceinline__ void mom_fill(S* __restrict__ fa, S* __restrict__ fb, const StepState* __restrict__ st,
                                         const float* __restrict__ psi_a, const float* __restrict__ psi_b,
                                         const MomDev& md, const ChainState* __restrict__ cs, const Lat& lat,
                                         const PhysParams& pp, int next) {
  if (next && !cs->full) return;
  const int t = next ? st->parity : st->parity ^ 1;
  S* __restrict__ f = t ? fa : fb;
  const float* __restrict__ psi = t ? psi_b : psi_a;
  const size_t N = (size_t)lat.Ns;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < lat.N; k += (long long)gridDim.x * blockDim.x) {
    const Cell c = cell_of(k, lat);
    if (md.map(t)[md.brick(c.x >> BRICK_BITS, c.y >> BRICK_BITS, c.z >> BRICK_BITS)]) continue;
    const float4 m = md.M(t)[c.n];
    if (m.x == MOM_SOLID) {
#pragma unroll
      for (int i = 0; i < Q; ++i) St<S>::st(f, (size_t)i * N + c.n, i, 0.0f);
      continue;
    }
    auto psi_at = [&](int i) -> float { return i ? psi[nbr(c, lat, i, +1)] : psi[c.n]; };
    float Fx, Fy, Fz, vx, vy, vz;
    mom_force(psi_at, pp, Fx, Fy, Fz);
    mom_values(m, Fx, Fy, Fz, vx, vy, vz, [&](int i, float v) { St<S>::st(f, (size_t)i * N + c.n, i, v); });
  }
}

// the bricks around a cell near the periodic seam
__device__ __noinline__ void mark_bricks_seam(const MomDev& md, int t, int x, int y, int z, const Lat& lat) {
  int b[3][BRICK_SPAN], nbk[3];
  nbk[0] = brick_span(x, BRICK_REACH, lat.nx, b[0]);
  nbk[1] = brick_span(y, BRICK_REACH, lat.ny, b[1]);
  nbk[2] = brick_span(z, BRICK_REACH, lat.nz, b[2]);
  for (int iz = 0; iz < nbk[2]; ++iz)
    for (int iy = 0; iy < nbk[1]; ++iy)
      for (int ix = 0; ix < nbk[0]; ++ix) md.map(t)[md.brick(b[0][ix], b[1][iy], b[2][iz])] = 1;
}

template <typename S>
__global__ void __launch_bounds__(256) k_mom_fill(S* fa, S* fb, const StepState* st, const float* psi_a,
                                                  const float* psi_b, const MomDev md, const ChainState* cs, const Lat lat,
                                                  const PhysParams pp, int next) {
  mom_fill<S>(fa, fb, st, psi_a, psi_b, md, cs, lat, pp, next);
}
template <typename S>
__global__ void __launch_bounds__(256) k_batch_fill(const BatchInst* __restrict__ tab) {
  const BatchInst& I = tab[blockIdx.y];
  mom_fill<S>((S*)I.fa, (S*)I.fb, I.st, (const float*)I.psi, (const float*)I.psi2, I.md, I.cs, I.lat, I.pp, 1);
}

// End of a step, after the refill: for the cells next to a solid, psi of the next step and the bricks
// around them in which the next step stores populations; and around every cell whose obstacle flag
// changed the moments and psi of the cells that are not: within 2 cells of a covered one (the receivers of
// its refill are next to it, and the cells that pull from those one further), within 1 of an uncovered one.
// The last block then ends the step, as k_finish does for the other passes.
template <typename S>
__device__ __forceinline__ void mom_close(S* fa, S* fb, StepState* __restrict__ st,
                                          const uint16_t* __restrict__ flags, float* __restrict__ psi_a,
                                          float* __restrict__ psi_b, const MomDev& md, const int* __restrict__ events,
                                          ChainState* __restrict__ cs, const int* __restrict__ blist, const Lat& lat,
                                          float rho0_f, int next, double* __restrict__ mass_part) {
  const int t = next ? st->parity ^ 1 : st->parity;  // the next step's parity
  const S* const f = t ? fb : fa;
  float* __restrict__ psi = t ? psi_b : psi_a;
  const unsigned near = next ? cs->nnew : st->nbnd, total = near + 125u * (next ? cs->nevent : 0u);
  for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += gridDim.x * blockDim.x) {
    float fi[Q];
    unsigned sl;
    if (k < near) {
      const Cell c = cell_of(blist[k], lat);
      pull<S>(f, flags, lat, c, (long long)c.n, fi, sl, F_NEAR);
      float rho = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) rho += fi[i];
      psi[c.n] = mom_psi(rho, rho0_f);
      if (c.x >= BRICK_REACH && c.y >= BRICK_REACH && c.z >= BRICK_REACH && c.x + BRICK_REACH < lat.nx &&
          c.y + BRICK_REACH < lat.ny && c.z + BRICK_REACH < lat.nz) {
        // seven cells in a row touch at most three bricks of four
#pragma unroll
        for (int q = 0; q < 27; ++q)
          md.map(t)[md.brick((c.x + (q % 3 - 1) * BRICK_REACH) >> BRICK_BITS, (c.y + (q / 3 % 3 - 1) * BRICK_REACH) >> BRICK_BITS,
                             (c.z + (q / 9 - 1) * BRICK_REACH) >> BRICK_BITS)] = 1;
      } else {
        mark_bricks_seam(md, t, c.x, c.y, c.z, lat);
      }
    } else {
      const unsigned r = k - near, ev = r / 125u, o = r - 125u * ev;
      const Cell a = cell_of(events[ev], lat);
      const int x = wrapi_near(a.x + (int)(o % 5u) - 2, lat.nx), y = wrapi_near(a.y + (int)((o / 5u) % 5u) - 2, lat.ny),
                z = wrapi_near(a.z + (int)(o / 25u) - 2, lat.nz);
      const Cell c = make_cell(x, y, z, lat);
      // an uncovered cell starts empty: it changes itself and those that pull from it, no further
      const bool inner = (unsigned)((int)(o % 5u) - 1) < 3u && (unsigned)((int)((o / 5u) % 5u) - 1) < 3u && o >= 25u && o < 100u;
      if (!inner && !(flags[a.n] & F_COVER)) continue;
      const uint16_t fl = flags[c.n];
      if (fl & F_NEAR) continue;
      if (fl & F_SOLID) {
        md.M(t)[c.n] = make_float4(MOM_SOLID, 0.0f, 0.0f, 0.0f);
        // (no fluid cell pulls from a solid one, so nothing reads what this overwrites)
        if (o == 62u && (fl & F_COVER)) zero_populations<S>(fa, fb, lat, c.n);
        continue;
      }
      pull<S>(f, flags, lat, c, (long long)c.n, fi, sl, 0);
      const float4 m = moments_of(fi);
      md.M(t)[c.n] = m;
      psi[c.n] = mom_psi(m.x, rho0_f);
    }
  }
  if (!next) return;
  // After a fill in this step every population of it is stored, and what the refill added and what was zeroed above
  // is in the populations alone: a fill between steps must leave them. (Nothing reads this map any more but
  // such a fill; the next step's start empties it.)
  if (cs->full) {
    unsigned char* const map = md.map(t ^ 1);
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < md.bricks(); k += gridDim.x * blockDim.x) map[k] = 1;
  }
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&cs->done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  if (threadIdx.x == 0) cs->done = 0;
  finish_step<128>(mass_part, MASS_SLOTS, st, cs);
}

template <typename S>
__global__ void __launch_bounds__(128) k_mom_close(S* fa, S* fb, StepState* st, const uint16_t* flags,
                                                   float* psi_a, float* psi_b, const MomDev md, const int* events,
                                                   ChainState* cs, const int* blist, const Lat lat, float rho0_f, int next,
                                                   double* mass_part) {
  mom_close<S>(fa, fb, st, flags, psi_a, psi_b, md, events, cs, blist, lat, rho0_f, next, mass_part);
}
template <typename S>
__global__ void __launch_bounds__(128) k_batch_close(const BatchInst* __restrict__ tab) {
  const BatchInst& I = tab[blockIdx.y];
  mom_close<S>((S*)I.fa, (S*)I.fb, I.st, I.flags, (float*)I.psi, (float*)I.psi2, I.md, I.events, I.cs, I.blist,
               I.lat, I.pp.rho0_f, 1, I.mass_part);
}
// the cells next to a solid of a batch's instances on the split pass
template <typename S>
__global__ void __launch_bounds__(128) k_batch_near(const BatchInst* __restrict__ tab) {
  using R = typename St<S>::R;
  const BatchInst& I = tab[blockIdx.y];
  const R mass = near_cells<S, false>((S*)I.fa, (S*)I.fb, I.flags, (const R*)I.psi, (const R*)nullptr, I.bodies, I.st,
                                      I.diag_rho, I.diag_vel, I.blist, I.lat, I.pp, (RhoPsi<R>*)I.nbuf,
                                      blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
  add_mass_slot(I.mass_part, mass, blockIdx.x * 7u + 3u);
}
// start of a batch's step: field record on or off, work queues and barrier arrivals cleared
__global__ void k_batch_begin(const BatchInst* __restrict__ tab, int ninst, BatchCtl* ctl, int diag) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < ninst) tab[k].st->diag = diag;
  if (k < 2) {
    ctl[k].queue[0] = ctl[k].queue[1] = 0;
    ctl[k].arrive = 0;
  }
}
