// Liquid tiles of the 3D step.  Away from the solid the phase field is
// pure liquid (phi_l = 1, every other phase 0) in a tile's whole reach, and
// Algorithm 1 reduces there to: phi^{n+1} = phi^n (only one phase is present
// in every 3x3x3 neighbourhood, so it has no rate), the chemical potential
// diffusing with M = D_liq / (2 A_l) and advected by U^n with h_l = 1 and
// chi = 1 / (2 A_l), and the lattice Boltzmann step with phi_l = 1 (no drag,
// the full buoyancy).  liquid_march advances such tiles with the same
// arithmetic, term for term, as the general path's liquid planes --
// the results are bit-identical -- but without the phase-field machinery,
// so it needs far fewer registers and instructions.
//
// Which tiles are liquid: a flag per tile of the step grid (x tile, y tile,
// z segment) says that every cell the tile owns is pure liquid.  A tile whose
// own flag and its 26 neighbours' flags are set reads only pure liquid (its
// reach is two cells and two planes), so the liquid path takes it;
// otherwise the general path does.  Both write the flags of the tile's new
// state, one per plane.
#pragma once

#include "gpflbm_kernels.cuh"
#include "step3d.cuh"

namespace gpflbm {

// Segments one CTA of the liquid path may march in one go.  A march repeats two
// planes, 8 for the 6 of one segment and 14 for 12.  With 16-bit populations
// the path is bound by instruction issue and marches two (FP16 dendrite 256^3:
// 603 us a step against 638); with FP32 ones by the traffic between L2 and the
// SMs, where the z-neighbours' planes are in L2 more often the sooner they are
// read again, and marches one (ternary eutectic: 1.65 ms against 1.73 with two,
// 1.83 with three).
template <class Store>
constexpr int kLiquidGroup = sizeof(Store) == 2 ? 2 : 1;

template <int NP, int NC, class Real, class Store, int QQ = 19, bool EXT = false>
struct Liquid3D {
  static constexpr int BX = Block3D<Real>::BX, BY = Block3D<Real>::BY, ZS = Block3D<Real>::ZS;
  static constexpr int NT = BX * BY;
  static constexpr int OX = BX - 2, OY = BY - 2;
  // mu and the y current of a plane, for the rows next to a thread's (its own
  // row is its warp, its own column its registers), in two slots: one barrier
  // a plane
  static constexpr size_t bytes = sizeof(Real) * 2 * 2 * NC * NT;
  // Two phases with FP32 populations: a plane's loads are issued before the
  // barrier of the plane below, from a pointer a population (dendrite 256^3:
  // 666 us a step against 673; not four phases, 1655 against 1651, nor 16-bit
  // populations, which then pay for packing them, 733 against 603, nor D3Q27,
  // 120^3: 206 against 191).
  static constexpr bool AHEAD = NP == 2 && QQ == 19 && sizeof(Store) == 4 && sizeof(Real) == 4;
};

// The liquid path for n planes from z0 of xy tile (bx, by) (z0 + n <= v_hi).
// Bound by the sectors that pass between L2 and the SMs and by instruction
// issue: a kernel that only loads and stores the 21 planes of the ternary
// eutectic in this pattern takes 1.26 ms for 256 x 256 x 512 cells (6.8 TB/s
// without halos and off-by-one rows: 0.85 ms), this path 1.24 ms.  x-faces pass
// between the lanes of a warp (a warp is a row of the tile), z-faces stay in a
// thread's registers, and each thread forms both its y-faces, so that shared
// memory holds mu and the y currents alone.  A cell mirrored at a wall hands
// out its currents with the sign turned, which makes the flux through the
// wall's face exactly zero without a test.
template <int NP, int NC, class Real, class Store, int QQ, bool EXT>
__device__ __forceinline__ void liquid_march(const DevParams<Real>& P, const Step3DIO& io, int bx, int by, int z0,
                                             int n, int gxt, int gyt) {
  using S = Liquid3D<NP, NC, Real, Store, QQ, EXT>;
  using Lat = Lattice<QQ>;
  constexpr int BX = S::BX, BY = S::BY, NT = S::NT, Q = QQ;
  constexpr int NS = PhiStore<NP>::NS;
  static_assert(BX == 32, "a row of the tile is a warp");
  extern __shared__ __align__(16) unsigned char smem[];
  // planes whose phi in the output buffer already is pure liquid (its flags,
  // from when it was last written): nothing to write there
  __shared__ unsigned char s_have[kLiquidGroup<Store> * S::ZS];

  const Real* __restrict__ mu_in = static_cast<const Real*>(io.mu_in);
  const Store* __restrict__ f_in = static_cast<const Store*>(io.f_in);
  Real* __restrict__ phi_out = static_cast<Real*>(io.phi_out);
  Real* __restrict__ mu_out = static_cast<Real*>(io.mu_out);
  Store* __restrict__ f_out = static_cast<Store*>(io.f_out);

  const int tid = threadIdx.x;
  const int tx = tid % BX, ty = tid / BX;
  const int nx = P.n[0], ny = P.n[1], nz = P.n[2], px = P.px;
  const int zst = px * ny;
  const int x0 = bx * S::OX, y0 = by * S::OY;
  const int gx = x0 - 1 + tx, gy = y0 - 1 + ty;
  // (tiles this far inside are the general path's: one condition for both)
  const bool inner_xy = x0 >= 2 && x0 - 2 + BX + 2 <= nx && y0 >= 2 && y0 - 2 + BY + 2 <= ny;
  const int fx = inner_xy ? gx : fold_axis(P, gx, 0);
  const int fy = inner_xy ? gy : fold_axis(P, gy, 1);
  const int gxy = fy * px + fx;
  const bool owner = tx >= 1 && tx <= BX - 2 && ty >= 1 && ty <= BY - 2 && gx < nx && gy < ny;
  if (tid < n) s_have[tid] = io.flags_out[liquid_flag_index(bx, by, z0 + tid, gxt, gyt)];
  const Real theta_base = theta_at(P, io.clock_in[0]);
  auto ceq_of = [&](int i, int v) -> Real {
    if constexpr (EXT)
      return fma_rn(P.dceq_dT[0][i], fma_rn(P.G, Real(v), theta_base), P.ceq[0][i]);
    else
      return P.ceq[0][i];
  };
  // planes z0 - 1 .. z0 + n, folded at the ends of the vertical axis
  const bool zin = z0 >= 1 && z0 + n < nz;
  auto vz = [&](int v) {
    if (zin) return v;
    const int f = fold_axis(P, v, 2);
    return f < P.v_lo - 2 ? P.v_lo - 2 : (f > P.v_hi + 1 ? P.v_hi + 1 : f);
  };
  auto zrow = [&](int fz) { return (fz - P.zbase) * zst; };
  // a cell mirrored at a wall in x, y
  const bool mirror_x = P.bc[0] == kWall && (gx < 0 || gx >= nx);
  const bool mirror_y = P.bc[1] == kWall && (gy < 0 || gy >= ny);
  const int up = ty < BY - 1 ? BX : 0, down = ty > 0 ? -BX : 0;

  Store fk[Q];
  Real mu_n[NC];
  auto load = [&](int v) {
    const int g = zrow(vz(v)) + gxy;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      if constexpr (S::AHEAD)
        fk[k] = static_cast<const Store*>(io.fi[k])[(unsigned)g];
      else
        fk[k] = at_bytes(f_in + g, P.f_at[k]);
    }
#pragma unroll
    for (int i = 0; i < NC; ++i) mu_n[i] = (mu_in + i * P.plane)[g];
  };
  if constexpr (S::AHEAD) load(z0 - 1);
  // of the plane below: mu and the z current of this column, the in-plane part
  // of the divergence, and the solute flux through its lower z-face
  Real mu_b[NC], wz_b[NC], div_b[NC], z_lo[NC];
#pragma unroll
  for (int i = 0; i < NC; ++i) mu_b[i] = wz_b[i] = div_b[i] = z_lo[i] = Real(0);
  for (int C = z0 - 1; C <= z0 + n; ++C) {
    const bool inside = C >= z0 && C < z0 + n;  // a plane this march advances
    const int fzc = vz(C), gi = zrow(fzc) + gxy;
    Real* const sl = reinterpret_cast<Real*>(smem) + (C & 1) * 2 * NC * NT + tid;
    Real mu[NC], wx[NC], wy[NC], wz[NC];
    {
      Real dk[Q];
      if constexpr (!S::AHEAD) load(C);
#pragma unroll
      for (int k = 0; k < Q; ++k) dk[k] = Codec<Store>::load(fk[k]);
#pragma unroll
      for (int i = 0; i < NC; ++i) mu[i] = mu_n[i];
      Real drho = Real(0), m3[3] = {Real(0), Real(0), Real(0)};
#pragma unroll
      for (int k = 0; k < Q; ++k) {
        drho += dk[k];
#pragma unroll
        for (int a = 0; a < 3; ++a)
          if (Lat::c(k, a) != 0) m3[a] += Real(Lat::c(k, a)) * dk[k];
      }
      const Real rho = Real(1) + drho;
      // force_velocity with phi_l = 1: no drag, the buoyancy alone
      const Real FB = mul_rn(rho, buoyancy_drive<NC, EXT>(P, fma_rn(P.G, Real(fzc), theta_base), mu));
      const Real inv = rcp_rn(rho);
      const Real u[3] = {mul_rn(m3[0], inv), mul_rn(m3[1], inv), mul_rn(fma_rn(Real(0.5), FB, m3[2]), inv)};
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        const Real c = ceq_of(i, fzc);
        wx[i] = liquid_adv(P, u[0], mu[i], c);
        wy[i] = liquid_adv(P, u[1], mu[i], c);
        wz[i] = liquid_adv(P, u[2], mu[i], c);
        if (mirror_x) wx[i] = -wx[i];
        if (mirror_y) wy[i] = -wy[i];
      }
      if (inside) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          sl[(2 * i) * NT] = mu[i];
          sl[(2 * i + 1) * NT] = wy[i];
        }
      }
      if (owner && inside) {
        const Real F[3] = {Real(0), Real(0), FB};
        if (inner_xy && C >= 1 && C + 1 < nz) {
          Store* const fo = f_out + gi;
          collide<Q, true>(P, dk, drho, rho, u, F,
                           [&](int k, Real val) {
                             if constexpr (S::AHEAD)
                               static_cast<Store*>(io.fo[k])[(unsigned)gi] = Codec<Store>::put(val);
                             else
                               at_bytes(fo, P.f_to[k]) = Codec<Store>::put(val);
                           });
        } else {
          const PushAxis X = push_axis(gx, nx, P.bc[0] == kWall, 1);
          const PushAxis Y = push_axis(gy, ny, P.bc[1] == kWall, px);
          const PushAxis Z = push_axis(C, nz, P.bc[2] == kWall, zst);
          collide<Q, true>(P, dk, drho, rho, u, F, [&](int k, Real val) {
            push_store<Lat>(f_out, P.plane, gi, k, Codec<Store>::put(val), X, Y, Z);
          });
        }
      }
    }
    if constexpr (S::AHEAD) {
      if (C < z0 + n) load(C + 1);
    }
    if (inside) __syncthreads();
    if (C >= z0) {
      // the z-face between this plane and the one below, whose update it ends
      const int M = C - 1;
      const bool closed = !zin && P.bc[2] == kWall && (C == 0 || C == nz);
      Real z_hi[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) z_hi[i] = closed ? Real(0) : liquid_flux(P, mu_b[i], mu[i], wz_b[i], wz[i]);
      if (M >= z0 && owner) {
        const int g = zrow(M) + gxy;
        if (!s_have[M - z0]) {
#pragma unroll
          for (int sidx = 0; sidx < NS; ++sidx)
            phi_out[sidx * P.plane + g] = (NP != 2 && sidx == 0) ? Real(1) : Real(0);
        }
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          const Real div = div_b[i] + sub_rn(z_hi[i], z_lo[i]);
          Real src = Real(0);
          if constexpr (EXT) {
#pragma unroll
            for (int a = 0; a < NP; ++a) src -= P.GV_r * P.dceq_dT[a][i] * (a == 0 ? Real(1) : Real(0));
          }
          mu_out[i * P.plane + g] = liquid_mu(P, mu_b[i], div, src);
        }
      }
#pragma unroll
      for (int i = 0; i < NC; ++i) z_lo[i] = z_hi[i];
    }
    if (inside) {
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        const Real* m = sl + (2 * i) * NT;
        const Real* w = sl + (2 * i + 1) * NT;
        const Real mr = __shfl_down_sync(0xffffffffu, mu[i], 1), wr = __shfl_down_sync(0xffffffffu, wx[i], 1);
        const Real jr = liquid_flux(P, mu[i], mr, wx[i], wr);
        const Real jl = __shfl_up_sync(0xffffffffu, jr, 1);
        const Real ju = liquid_flux(P, mu[i], m[up], wy[i], w[up]);
        const Real jd = liquid_flux(P, m[down], mu[i], w[down], wy[i]);
        div_b[i] = sub_rn(jr, jl) + sub_rn(ju, jd);
      }
    }
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      mu_b[i] = mu[i];
      wz_b[i] = wz[i];
    }
  }
  if (tid < n) io.flags_out[liquid_flag_index(bx, by, z0 + tid, gxt, gyt)] = 1;
}

// The liquid tiles of the group of segments starting at segment bz of xy tile
// (bx, by): each run of neighbouring liquid segments is one march.  Which
// segments are liquid is decided as the general pass decides it
// (liquid_reach).
template <int NP, int NC, class Real, class Store, int QQ, bool EXT>
__device__ __forceinline__ void liquid_tiles(const DevParams<Real>& P, const Step3DIO& io, int bx, int by, int bz,
                                             int gxt, int gyt) {
  using S = Liquid3D<NP, NC, Real, Store, QQ, EXT>;
  constexpr int ZS = S::ZS, G = kLiquidGroup<Store>;
  static_assert(9 * (G * ZS + 4) <= S::NT, "one flag a thread");
  __shared__ int s_bad[G];
  const int z0 = P.v_lo + bz * ZS, group = P.liq_group;
  const int tid = threadIdx.x;
  if (bx == 0 && by == 0 && bz == 0 && tid == 0) io.clock_out[0] = io.clock_in[0] + 1.0;
  if (tid < G) s_bad[tid] = 0;
  __syncthreads();
  if (tid < 9 * (group * ZS + 4)) {
    const int p = tid / 9;
    if (!liquid_flag_near(P, io.flags_in, bx, by, z0 - 2 + p, tid - 9 * p, gxt, gyt)) {
#pragma unroll
      for (int s = 0; s < G; ++s)
        if (s < group && p >= s * ZS && p < s * ZS + ZS + 4) s_bad[s] = 1;
    }
  }
  __syncthreads();
  for (int s = 0; s < group && z0 + s * ZS < P.v_hi;) {
    if (s_bad[s]) {
      ++s;
      continue;
    }
    int e = s + 1;
    while (e < group && z0 + e * ZS < P.v_hi && !s_bad[e]) ++e;
    const int zs = z0 + s * ZS, ze = min(z0 + e * ZS, P.v_hi);
    liquid_march<NP, NC, Real, Store, QQ, EXT>(P, io, bx, by, zs, ze - zs, gxt, gyt);
    __syncthreads();  // (s_have and the slots are reused)
    s = e;
  }
}

// The step kernels.  Where both paths fit 64 registers (FP32 arithmetic on
// D3Q19: two CTAs share an SM either way) and the general path is that of
// two phases (Step3D::ONE_LAUNCH), one launch takes every tile: its
// grid holds the tiling twice, z blocks 0 .. gzt-1 the general pass and those
// after them the liquid pass (a group of segments each), and a CTA returns
// unless its tile's flags pick its pass.  CTAs start in block order, so the general tiles, the slow
// ones, start first and the liquid tiles fill the SMs as they finish
// instead of waiting for the last general tile.  Elsewhere (FP64, D3Q27:
// the general path needs more registers than the liquid one, and one kernel
// would hold the liquid tiles to its occupancy; three or four phases: its
// shared memory, see ONE_LAUNCH) step3d_kernel takes the general tiles and
// step3d_liquid_kernel, launched after it, the others.
template <int NP, int NC, class Real, class Store, bool SHRINK = false, int QQ = 19, bool EXT = false, bool ANISO = false>
__global__ void __launch_bounds__(Step3D<NP, NC, Real, Store, QQ, SHRINK>::NT, Step3D<NP, NC, Real, Store, QQ>::MIN_CTAS)
    step3d_kernel(const DevParams<Real> P, const Step3DIO io) {
  using S = Step3D<NP, NC, Real, Store, QQ, SHRINK>;
  constexpr int ZS = S::ZS;
  const int gxt = gridDim.x, gyt = gridDim.y, gzt = (P.v_hi - P.v_lo + ZS - 1) / ZS;
  const int bx = blockIdx.x, by = blockIdx.y;
  const bool liquid_pass = S::ONE_LAUNCH && (int)blockIdx.z >= gzt;
  // (a shrinkage launch has no liquid pass; the kernel without its code is 3 %
  // slower all the same, 322 against 313 us on the dendrite 150 x 130 x 171)
  if constexpr (S::ONE_LAUNCH) {
    if (liquid_pass) {
      liquid_tiles<NP, NC, Real, Store, QQ, EXT>(P, io, bx, by, ((int)blockIdx.z - gzt) * P.liq_group, gxt, gyt);
      return;
    }
  }
  const int bz = blockIdx.z;
  if (P.liq_dispatch && liquid_reach<ZS>(P, io.flags_in, bx, by, P.v_lo + bz * ZS, gxt, gyt)) return;
  general_tile<NP, NC, Real, Store, SHRINK, QQ, EXT, ANISO>(P, io, bx, by, bz, gxt, gyt);
}

template <int NP, int NC, class Real, class Store, int QQ = 19, bool EXT = false>
__global__ void __launch_bounds__(Liquid3D<NP, NC, Real, Store, QQ, EXT>::NT, 2)
    step3d_liquid_kernel(const DevParams<Real> P, const Step3DIO io) {
  liquid_tiles<NP, NC, Real, Store, QQ, EXT>(P, io, blockIdx.x, blockIdx.y, blockIdx.z * P.liq_group, gridDim.x,
                                             gridDim.y);
}

// The liquid flags of a state (after a load or a frame shift): one CTA per
// xy tile and plane, the flag set when every cell the tile owns in the plane
// is pure liquid.
template <int NP, class Real>
__global__ void liquid_flags_kernel(const DevParams<Real> P, const Real* __restrict__ phi,
                                    unsigned char* __restrict__ flags) {
  constexpr int BX = Block3D<Real>::BX, BY = Block3D<Real>::BY;
  constexpr int OX = BX - 2, OY = BY - 2;
  const int x0 = blockIdx.x * OX, y0 = blockIdx.y * OY, z = P.v_lo + blockIdx.z;
  const int wx = min(OX, P.n[0] - x0), wy = min(OY, P.n[1] - y0);
  const int zst = P.px * P.n[1];
  bool liq = true;
  for (int c = threadIdx.x; c < wx * wy; c += blockDim.x) {
    const int x = x0 + c % wx, y = y0 + c / wx;
    Real v[NP];
    load_phases<NP>(phi, (long long)(z - P.zbase) * zst + (long long)y * P.px + x, P.plane, v);
    bool p = v[0] == Real(1);
#pragma unroll
    for (int a = 1; a < NP; ++a) p = p && v[a] == Real(0);
    liq = liq && p;
  }
  liq = __syncthreads_and(liq);
  if (threadIdx.x == 0) flags[liquid_flag_index(blockIdx.x, blockIdx.y, z, gridDim.x, gridDim.y)] = liq;
}

}  // namespace gpflbm
