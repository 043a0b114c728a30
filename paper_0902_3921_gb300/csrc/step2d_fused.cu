// step2d_fused.cu -- one LB step of a small 2D lattice in one launch (FP32
// deviations; FP16 storage keeps the separate kernels, because a step of
// another operation order rounds its stored populations differently, and over
// 64 steps phi then differs by as much as FP16 storage itself costs, 2e-5).
//
// On lattices up to about 512^2 the step is bound by latency: two launches, of
// which the FD block kernel's 128 x 80 regions put a 64^2 lattice on one or two
// SMs.  The launch here covers the FD update of step t - 1 and the collide of
// step t, which need nothing from other CTAs of the same launch: a CTA forms
// phi(t) on its tile plus a halo of 2 (all m <= 4 substeps, on a region with a
// halo of 3 m + 2), then mu, the force, the moments and the collision of the
// tile; the pulled populations arrive while mu is formed.  A run of n
// steps is n + 1 launches instead of 2 n: collide of the first step, n - 1
// fused launches, FD of the last one; the first and the last are the same
// kernel with one half left out, and every operation is explicitly rounded, so
// a run gives the same bits however it is cut into lbm_step calls.
// u* alternates between the handle's planes and a second pair in the staging
// buffer, because a CTA reads u*(t - 1) of its neighbours' tiles while they
// write u*(t).
//
// A region is 64 columns wide: a half-warp owns a row, a lane four columns
// (one float4), x neighbours by shuffles, y neighbours through one
// shared-memory plane per field (phi, phih, psi) with the own row in
// registers, so a phase is two shared loads, two shuffles and one store.
// Tiles of 16 rows keep a small lattice's critical path short; 32 rows halve
// the halo work once the tiles of 16 exceed the SMs (the autotuner times
// both, and both against the two separate kernels, whose 128 x 96 FD regions have
// half the halo: they win from 450^2 to 600^2 on, see its rule).
// Step on a GB300, two kernels -> this one: 64^2 14.1 -> 5.35 us, 256^2 15.1 -> 5.5,
// 384^2 15.1 -> 7.5, 432^2 16.3 -> 14.4, 509 x 251 in flux form 18.4 -> 8.8; the paper's
// fluid (m = 1), 64^2 7.7 -> 3.5 us.
#include "lbm_common.cuh"

namespace hlbm {

namespace {

constexpr int FS_RW = 64;  // region columns
constexpr unsigned FULL = 0xffffffffu;

enum { FS_FD = 1, FS_COLLIDE = 2 };  // halves of a launch

template <int SUB, int TY>
struct FStep {
  static constexpr int HY = 3 * SUB + 2, HX = (HY + 3) / 4 * 4;  // halo; columns in whole float4
  static constexpr int TX = FS_RW - 2 * HX, RY = TY + 2 * HY;
  static constexpr int NW_FD = RY / 2, NW = TY == 32 && NW_FD < 32 ? 32 : NW_FD, NT = 32 * NW;
  static constexpr int SITES = TX * TY, NS = (SITES + NT - 1) / NT;  // sites per thread of the collision
  static_assert(RY % 2 == 0 && NT <= 1024, "one row per half-warp");
  static constexpr size_t smem = sizeof(float) * 3 * RY * FS_RW;
};

__device__ __forceinline__ float fm(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fa(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fs(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float ff(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// left and right neighbours of a lane's quad (the outermost lanes of a row get
// their own values: those columns are never valid)
__device__ __forceinline__ void xn(const float4 &c, float &l, float &r) {
  l = __shfl_up_sync(FULL, c.w, 1, 16);
  r = __shfl_down_sync(FULL, c.x, 1, 16);
}

// 5-point Laplacian of a quad
__device__ __forceinline__ void lap5(const float4 &c, const float4 &up, const float4 &dn, float2 &lo, float2 &hi) {
  float l, r;
  xn(c, l, r);
  const float2 m4 = f2(-4.f, -4.f);
  lo = __ffma2_rn(m4, f2(c.x, c.y), __fadd2_rn(__fadd2_rn(f2(up.x, up.y), f2(dn.x, dn.y)), f2(fa(l, c.y), fa(c.x, c.z))));
  hi = __ffma2_rn(m4, f2(c.z, c.w), __fadd2_rn(__fadd2_rn(f2(up.z, up.w), f2(dn.z, dn.w)), f2(fa(c.y, c.w), fa(c.z, r))));
}

__device__ __forceinline__ float at4(const float4 &v, int j) { return j == 0 ? v.x : (j == 1 ? v.y : (j == 2 ? v.z : v.w)); }

template <int SUB, int TY, bool FLUX, int MODE>
__global__ void __launch_bounds__(FStep<SUB, TY>::NT, 1)
    step2d_kernel(const float *phi_in, const float *u_in, float *phi_out, const float *hin, float *hout, float *u_out,
                  KParams<float> p) {
  using G = FStep<SUB, TY>;
  constexpr int HX = G::HX, HY = G::HY, TX = G::TX, RY = G::RY, NS = G::NS;
  extern __shared__ __align__(16) float fs_smem[];
  float *sp = fs_smem, *sa = sp + RY * FS_RW, *sq = sa + RY * FS_RW;
  const int tid = threadIdx.x, lane = tid & 31, c = 4 * (lane & 15);
  const int row = 2 * (tid >> 5) + (lane >> 4);
  const bool fdw = row < RY;  // warp-uniform: warps beyond the region's rows only collide
  const int r = fdw ? row : RY - 1;
  const int Lx = p.Lx, Ly = p.Ly;
  const long long Sz = (long long)Lx * Ly;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const bool vec = (Lx & 3) == 0;  // TX and HX are multiples of 4: a quad never straddles the wrap
  int gx[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) gx[j] = wrapi(x0 - HX + c + j, Lx);
  auto rowof = [&](int rr) { return (long long)wrapi(y0 - HY + rr, Ly) * Lx; };
  auto ldq = [&](const float *f, long long ro) {
    if (vec) return *reinterpret_cast<const float4 *>(f + ro + gx[0]);
    return make_float4(f[ro + gx[0]], f[ro + gx[1]], f[ro + gx[2]], f[ro + gx[3]]);
  };
  auto sld = [&](const float *pl, int rr) { return *reinterpret_cast<const float4 *>(pl + rr * FS_RW + c); };
  auto sst = [&](float *pl, const float4 &v) {
    if (fdw) *reinterpret_cast<float4 *>(pl + r * FS_RW + c) = v;
  };
  const int rm = r > 0 ? r - 1 : 0, rp = r < RY - 1 ? r + 1 : r;  // rows 0 and RY - 1 are never valid
  const long long ro = rowof(r);

  // pulled populations f_i(r, t) = buf_i(r - e_i) of this thread's sites
  float h[NS][9];
  int sx[NS], sy[NS];
  bool ok[NS];
  auto load_pops = [&]() {
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const int s = tid + k * G::NT;
      sy[k] = s / TX;
      sx[k] = s - sy[k] * TX;
      ok[k] = s < G::SITES && x0 + sx[k] < Lx && y0 + sy[k] < Ly;
      const int x = ok[k] ? x0 + sx[k] : 0, y = ok[k] ? y0 + sy[k] : 0;
      const int xm = x == 0 ? Lx - 1 : x - 1, xp = x == Lx - 1 ? 0 : x + 1;
      const float *rc = hin + (long long)y * Lx, *rdn = hin + (long long)(y == 0 ? Ly - 1 : y - 1) * Lx,
              *rup = hin + (long long)(y == Ly - 1 ? 0 : y + 1) * Lx;
      h[k][0] = rc[x];
      h[k][1] = rc[Sz + xm];
      h[k][2] = rdn[2 * Sz + x];
      h[k][3] = rc[3 * Sz + xp];
      h[k][4] = rup[4 * Sz + x];
      h[k][5] = rdn[5 * Sz + xm];
      h[k][6] = rdn[6 * Sz + xp];
      h[k][7] = rup[7 * Sz + xp];
      h[k][8] = rup[8 * Sz + xm];
    }
  };

  // phi, u* and the populations come from the previous launch, which may still run
  // when this one starts: ordinary loads (no __ldg, no restrict, which would let the
  // compiler make them read-only ones), all after the wait
  pdl_wait();
  pdl_trigger();
  float4 ph = ldq(phi_in, ro);
  if constexpr ((MODE & FS_FD) != 0) {
    // advection coefficients of the row (Eqs. 32-35): printed form c0, dt u,
    // dt v; flux form the four face velocities
    const float4 uc = ldq(u_in, ro), vc = ldq(u_in + Sz, ro);
    const float4 vm = ldq(u_in + Sz, rowof(rm)), vp = ldq(u_in + Sz, rowof(rp));
    sst(sp, ph);
    float t0[4], t1[4], t2[4], t3[FLUX ? 4 : 1];
    {
      float ul, ur;
      xn(uc, ul, ur);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float uj = at4(uc, j), uL = j == 0 ? ul : at4(uc, j - 1), uR = j == 3 ? ur : at4(uc, j + 1);
        const float vj = at4(vc, j), vmj = at4(vm, j), vpj = at4(vp, j);
        if constexpr (!FLUX) {
          const float div = ff(0.5f, fa(fs(uR, uL), fs(vpj, vmj)), fa(fabsf(uj), fabsf(vj)));
          t0[j] = ff(-p.dt, div, 1.f);
          t1[j] = fm(p.dt, uj);
          t2[j] = fm(p.dt, vj);
        } else {
          t0[j] = fm(0.5f, fa(uj, uR));
          t1[j] = fm(0.5f, fa(uL, uj));
          t2[j] = fm(0.5f, fa(vj, vpj));
          t3[j] = fm(0.5f, fa(vmj, vj));
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < SUB; ++s) {
      // phih (Eqs. 32-35)
      const float4 pd = sld(sp, rm), pu = sld(sp, rp);
      float4 a4;
      {
        float pl, pr;
        xn(ph, pl, pr);
        float e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float pc = at4(ph, j), L = j == 0 ? pl : at4(ph, j - 1), R = j == 3 ? pr : at4(ph, j + 1);
          const float D = at4(pd, j), U = at4(pu, j);
          if constexpr (!FLUX) {
            const float upx = t1[j] > 0.f ? L : R, upy = t2[j] > 0.f ? D : U;  // u = 0 contributes nothing
            e[j] = ff(fabsf(t2[j]), upy, ff(fabsf(t1[j]), upx, fm(t0[j], pc)));
          } else {
            float t = fm(t0[j], t0[j] > 0.f ? pc : R);
            t = ff(-t1[j], t1[j] > 0.f ? L : pc, t);
            t = ff(t2[j], t2[j] > 0.f ? pc : U, t);
            t = ff(-t3[j], t3[j] > 0.f ? D : pc, t);
            e[j] = ff(-p.dt, t, pc);
          }
        }
        a4 = make_float4(e[0], e[1], e[2], e[3]);
      }
      sst(sa, a4);
      __syncthreads();
      // psi = a phih + b phi^3 - kappa lap phih (Eq. 36)
      float4 q4;
      {
        float2 L[2], o[2];
        lap5(a4, sld(sa, rp), sld(sa, rm), L[0], L[1]);
        const float4 cb = p.cubic_at_half ? a4 : ph;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float2 hk = k ? f2(a4.z, a4.w) : f2(a4.x, a4.y), ck = k ? f2(cb.z, cb.w) : f2(cb.x, cb.y);
          o[k] = __ffma2_rn(f2(p.a, p.a), hk,
                            __ffma2_rn(f2(p.b, p.b), __fmul2_rn(__fmul2_rn(ck, ck), ck),
                                       __fmul2_rn(f2(-p.kappa, -p.kappa), L[k])));
        }
        q4 = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
      }
      sst(sq, q4);
      __syncthreads();
      // phi^{n+1} = phih + dt Gamma lap psi
      {
        float2 L[2];
        lap5(q4, sld(sq, rp), sld(sq, rm), L[0], L[1]);
        const float2 g = f2(p.dtG, p.dtG), lo = __ffma2_rn(g, L[0], f2(a4.x, a4.y)), hi = __ffma2_rn(g, L[1], f2(a4.z, a4.w));
        ph = make_float4(lo.x, lo.y, hi.x, hi.y);
      }
      if (s + 1 < SUB || (MODE & FS_COLLIDE) != 0) {
        sst(sp, ph);
        __syncthreads();
        // the populations are in flight under mu (64^2 5.35 us a step; issued in the last
        // substep or earlier 5.45 to 5.6)
        if constexpr ((MODE & FS_COLLIDE) != 0)
          if (s == SUB - 1) load_pops();
      }
    }
    const int yt = r - HY, xt = c - HX;  // tile coordinates
    if (fdw && yt >= 0 && yt < TY && y0 + yt < Ly && xt >= 0 && xt < TX) {
      float *dst = phi_out + (long long)(y0 + yt) * Lx + x0 + xt;
      if (vec) {
        if (x0 + xt < Lx) *reinterpret_cast<float4 *>(dst) = ph;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (x0 + xt + j < Lx) dst[j] = at4(ph, j);
      }
    }
  } else {
    load_pops();
    sst(sp, ph);
    __syncthreads();
  }

  if constexpr ((MODE & FS_COLLIDE) != 0) {
    // mu = a phi + b phi^3 - kappa lap_D phi (Eqs. 5, 31) on the tile + 1
    {
      const float4 up = sld(sp, rp), dn = sld(sp, rm);
      float cl, cr, ul, ur, dl, dr;
      xn(ph, cl, cr);
      xn(up, ul, ur);
      xn(dn, dl, dr);
      float e[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float cc = at4(ph, j);
        const float W = j == 0 ? cl : at4(ph, j - 1), E = j == 3 ? cr : at4(ph, j + 1);
        const float NW_ = j == 0 ? ul : at4(up, j - 1), NE = j == 3 ? ur : at4(up, j + 1);
        const float SW = j == 0 ? dl : at4(dn, j - 1), SE = j == 3 ? dr : at4(dn, j + 1);
        // sums of differences from the centre, exact for close neighbours: sums
        // of the values themselves round at 4 |phi| (the error of mu is 2 to
        // 3 times that of the row-by-row order of the other kernels)
        const float faces = fa(fa(fs(at4(dn, j), cc), fs(at4(up, j), cc)), fa(fs(W, cc), fs(E, cc)));
        const float corners = fa(fa(fs(SW, cc), fs(SE, cc)), fa(fs(NW_, cc), fs(NE, cc)));
        const float lap = ff(p.Q, faces, fm(p.R, corners));
        e[j] = ff(ff(p.b, fm(cc, cc), p.a), cc, fm(-p.kappa, lap));
      }
      sst(sa, make_float4(e[0], e[1], e[2], e[3]));  // phih's plane
    }
    __syncthreads();
    // force (Eq. 28), moments (Eqs. 12, 18) and collision (Eqs. 15, 17, 29):
    // f_i = (1 - 1/tau) f_i + E + O, f_ib = (1 - 1/tau) f_ib + E - O of opposite
    // directions, O = q + r, q = 3 A n (e.u), r = 3 B (e.F), E = A base -
    // 3 B u.F + 1.5 (e.u)(q + 2 r), A = w / tau, B = w (1 - 1/2tau).
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      if (!ok[k]) continue;
      const float *m = sa + (sy[k] + HY) * FS_RW + sx[k] + HX;
      const float P = fs(m[FS_RW + 1], m[-FS_RW - 1]), D = fs(m[-FS_RW + 1], m[FS_RW - 1]);
      const float gmx = ff(p.M, fa(P, D), fm(p.N, fs(m[1], m[-1])));
      const float gmy = ff(p.M, fs(P, D), fm(p.N, fs(m[FS_RW], m[-FS_RW])));
      const float phc = sp[(sy[k] + HY) * FS_RW + sx[k] + HX];
      float Fx = fm(-phc, gmx), Fy = fm(-phc, gmy);
      const float *f = h[k];
      const float dens = fa(fa(f[0], fa(fa(f[1], f[3]), fa(f[2], f[4]))), fa(fa(f[5], f[7]), fa(f[6], f[8])));
      const float d5 = fs(f[5], f[7]), d6 = fs(f[6], f[8]);
      const float jx = fa(fs(f[1], f[3]), fs(d5, d6)), jy = fa(fs(f[2], f[4]), fa(d5, d6));
      const float n = fa(1.f, dens);
      Fx = ff(n, p.gx, Fx);
      Fy = ff(n, p.gy, Fy);
      const float inv_n = __frcp_rn(n);
      const float ux = fm(ff(0.5f, Fx, jx), inv_n), uy = fm(ff(0.5f, Fy, jy), inv_n);
      const float uF = ff(ux, Fx, fm(uy, Fy));
      const float om = p.tau_inv, keep = fs(1.f, om);
      const float base = ff(fm(-1.5f, n), ff(ux, ux, fm(uy, uy)), dens);
      const float iso = ff(om, base, fm(fm(-3.f, p.pref), uF));
      const float an3 = fm(fm(3.f, om), n), b3 = fm(3.f, p.pref);
      const float w0 = (float)q9_w(0), w1 = (float)q9_w(1), w2 = (float)q9_w(5);
      const long long s = (long long)(y0 + sy[k]) * Lx + x0 + sx[k];
      float *dst = hout + s;
      dst[0] = ff(keep, f[0], fm(w0, iso));
      auto pair = [&](int i, float iw, float q, float rr, float eu15) {
        const float O = fa(q, rr), E = ff(eu15, ff(2.f, rr, q), iw);
        dst[i * Sz] = fa(ff(keep, f[i], E), O);
        dst[(i + 2) * Sz] = fs(ff(keep, f[i + 2], E), O);
      };
      const float tx = fm(1.5f, ux), ty = fm(1.5f, uy);
      {
        const float A = fm(w1, an3), B = fm(w1, b3), iw = fm(w1, iso);
        pair(1, iw, fm(A, ux), fm(B, Fx), tx);
        pair(2, iw, fm(A, uy), fm(B, Fy), ty);
      }
      {
        const float A = fm(w2, an3), B = fm(w2, b3), iw = fm(w2, iso);
        const float qx = fm(A, ux), qy = fm(A, uy), rx = fm(B, Fx), ry = fm(B, Fy);
        pair(5, iw, fa(qx, qy), fa(rx, ry), fa(tx, ty));
        pair(6, iw, fs(qy, qx), fs(ry, rx), fs(ty, tx));
      }
      u_out[s] = ux;
      u_out[Sz + s] = uy;
    }
  }
}

template <int SUB, int TY, bool FLUX>
cudaError_t launch_one(lbm_handle *h, int part, const KParams<float> &p, const float *phi_in, const float *u_in,
                       float *phi_out, const float *hin, float *hout, float *u_out) {
  using G = FStep<SUB, TY>;
  const dim3 grid((p.Lx + G::TX - 1) / G::TX, (p.Ly + TY - 1) / TY);
  // While a launch leaves SMs free, the next one is scheduled beside it (it
  // waits for its end before it reads anything): 64^2 5.7 -> 5.4 us a step, 384^2
  // 8.0 -> 7.6, 509 x 251 9.5 -> 9.0.
  const bool beside = (int)(grid.x * grid.y) <= sm_count();
  auto go = [&](auto kernel) {
    return launch_ex(false, beside, kernel, grid, dim3(G::NT), G::smem, h->stream, phi_in, u_in, phi_out, hin, hout,
                     u_out, p);
  };
  if (part == (FS_FD | FS_COLLIDE)) return go(step2d_kernel<SUB, TY, FLUX, FS_FD | FS_COLLIDE>);
  if (part == FS_COLLIDE) return go(step2d_kernel<SUB, TY, FLUX, FS_COLLIDE>);
  return go(step2d_kernel<SUB, TY, FLUX, FS_FD>);
}

cudaError_t step2d(lbm_handle *h, int part, int in, int force_on, const float *u_in, float *u_out) {
  const KParams<float> p = make_params<float>(h, force_on);
  // collide of time t reads h[in], phi[in]; the FD before it forms phi[in] from phi[1 - in].
  // An FD alone forms phi[1 - in] from phi[in].
  const bool fd = (part & FS_FD) != 0, coll = (part & FS_COLLIDE) != 0;
  const float *src = static_cast<const float *>(h->phi[fd && coll ? 1 - in : in]);
  float *dst = static_cast<float *>(h->phi[fd && coll ? in : 1 - in]);
  const float *hin = static_cast<const float *>(h->h[in]);
  float *hout = static_cast<float *>(h->h[1 - in]);
  const bool flux = p.adv_variant == LBM_ADV_FLUX;
#define FS_GO(SB, TYY)                                                                            \
  return flux ? launch_one<SB, TYY, true>(h, part, p, src, u_in, dst, hin, hout, u_out)        \
              : launch_one<SB, TYY, false>(h, part, p, src, u_in, dst, hin, hout, u_out);
#define FS_SUB(SB)                       \
  if (h->m == SB) {                      \
    if (h->fd_rows == 16) { FS_GO(SB, 16) } \
    FS_GO(SB, 32)                        \
  }
  FS_SUB(1)
  FS_SUB(2)
  FS_SUB(3)
  FS_SUB(4)
#undef FS_SUB
#undef FS_GO
  return cudaErrorInvalidValue;
}

}  // namespace

bool step2d_eligible(const lbm_handle *h) {
  return h->dims == 2 && h->P.precision == LBM_F32DEV && h->m <= 4 && h->P.T == 1.0 / 3.0 && h->P.stencil_fd == 0;
}

// u_pp: the plane pair that the collide writes (0: the handle's u, 1: the pair in the staging buffer)
static float *u_planes(lbm_handle *h, int u_pp) {
  return u_pp ? reinterpret_cast<float *>(h->staging) : static_cast<float *>(h->u);
}
cudaError_t step2d_fd_collide(lbm_handle *h, int in, int force_on, int u_pp) {
  return step2d(h, FS_FD | FS_COLLIDE, in, force_on, u_planes(h, 1 - u_pp), u_planes(h, u_pp));
}
cudaError_t step2d_collide(lbm_handle *h, int in, int force_on, int u_pp) {
  return step2d(h, FS_COLLIDE, in, force_on, nullptr, u_planes(h, u_pp));
}
cudaError_t step2d_fd(lbm_handle *h, int in) { return step2d(h, FS_FD, in, 0, u_planes(h, 0), nullptr); }

static_assert(FStep<4, 32>::smem <= 48 * 1024, "the largest region needs no shared-memory opt-in");

}  // namespace hlbm
