// kernels_2d_f64.cu -- D2Q9 step with FP64 populations in small tiles.
//
// FP64 operations issue at about two per clock and SM on the GB300, so the
// FP64 step costs its operation count divided by the SMs that have work: the
// 32 x 16 to 32 x 32 tiles of the FP32-minded kernels put 128^2 on 16 to 32 of
// the 152 SMs.  Here a CTA takes 16 x 8 sites (128^2: 128 CTAs of four warps,
// one per scheduler), or 32 x 16 where the lattice fills the SMs anyway and
// the smaller halo share wins (the FD update; the autotuner times both).  The
// expressions use the fewest FP64 operations: upwind sides from the sign bit,
// shared diagonal differences, one reciprocal, no products with zero
// components of e_i.
// One LB step on a GB300, before (best of the other kernels) and now:
//   128^2, paper's fluid (m = 1): step 42.9 -> 11.0 us (collide 35 -> 11 by events);
//   512^2, m = 4: step 187 -> 146 us; 300 x 211, flux form: 88 -> 50 us.
#include "lbm_common.cuh"

namespace hlbm {

namespace {

constexpr int D_NT = 128;             // threads of the 16 x 8 tiles
constexpr int D_TX = 16, D_TY = 8;

__device__ __forceinline__ bool neg(double v) { return __double2hiint(v) < 0; }

// Derivative pair of Eq. 30 from a tile with row pitch W, at k: the diagonal
// differences P = f(+,+) - f(-,-), D = f(+,-) - f(-,+) serve both.
__device__ __forceinline__ void grad2(const double *f, int k, int W, const KParams<double> &p, double &gx, double &gy) {
  const double P = f[k + W + 1] - f[k - W - 1], D = f[k - W + 1] - f[k + W - 1];
  gx = fma(p.M, P + D, p.N * (f[k + 1] - f[k - 1]));
  gy = fma(p.M, P - D, p.N * (f[k + W] - f[k - W]));
}

// lap_D of Eq. 31
__device__ __forceinline__ double lapD(const double *f, int k, int W, const KParams<double> &p) {
  const double faces = (f[k - W] + f[k + W]) + (f[k - 1] + f[k + 1]);
  const double corners = (f[k - W - 1] + f[k - W + 1]) + (f[k + W - 1] + f[k + W + 1]);
  return fma(p.Q, faces, fma(p.R, corners, p.C0 * f[k]));
}

// Steps 1-4 of a 16 x 8 tile (or its moments), one site per thread.  The pair
// algebra is that of the FP64 3D kernel: f_i = (1 - 1/tau) f_i + E + O and
// f_ib = (1 - 1/tau) f_ib + E - O with O = q + r, q = 3 A n (e.u), r = 3 B (e.F),
// E = A base - 3 B u.F + 1.5 (e.u)(q + 2 r), A = w / tau, B = w (1 - 1/2tau).
template <bool TGEN, int MODE>
__global__ void __launch_bounds__(D_NT, 4)
    collide2d_f64_kernel(const double *__restrict__ hin, double *__restrict__ hout, const double *__restrict__ phi,
                         const double *__restrict__ dn, double *__restrict__ uout, double *__restrict__ stg,
                         KParams<double> p) {
  constexpr int PX = D_TX + 4, PY = D_TY + 4, MX = D_TX + 2, MY = D_TY + 2;
  __shared__ double sphi[PX * PY], smu[MX * MY], spn[TGEN ? MX * MY : 1];
  const int Lx = p.Lx, Ly = p.Ly, tid = threadIdx.x;
  const long long Sz = (long long)Lx * Ly;
  const int x0 = blockIdx.x * D_TX, y0 = blockIdx.y * D_TY;
  const int lx = tid % D_TX, ly = tid / D_TX;
  const bool ok = x0 + lx < Lx && y0 + ly < Ly;
  const int x = ok ? x0 + lx : 0, y = ok ? y0 + ly : 0;
  // f_i(r, t) = buf_i(r - e_i), in flight during the stencil phase
  const int xm = x == 0 ? Lx - 1 : x - 1, xp = x == Lx - 1 ? 0 : x + 1;
  const double *rc = hin + (long long)y * Lx, *rm = hin + (long long)(y == 0 ? Ly - 1 : y - 1) * Lx,
               *rp = hin + (long long)(y == Ly - 1 ? 0 : y + 1) * Lx;
  const double h0 = __ldg(rc + x);
  const double h1 = __ldg(rc + Sz + xm), h2 = __ldg(rm + 2 * Sz + x), h3 = __ldg(rc + 3 * Sz + xp),
               h4 = __ldg(rp + 4 * Sz + x), h5 = __ldg(rm + 5 * Sz + xm), h6 = __ldg(rm + 6 * Sz + xp),
               h7 = __ldg(rp + 7 * Sz + xp), h8 = __ldg(rp + 8 * Sz + xm);
  for (int k = tid; k < PX * PY; k += D_NT) {
    const int ry = k / PX, rx = k - ry * PX;
    sphi[k] = __ldg(phi + (long long)wrapi(y0 + ry - 2, Ly) * Lx + wrapi(x0 + rx - 2, Lx));
  }
  if constexpr (TGEN)
    for (int k = tid; k < MX * MY; k += D_NT) {
      const int ry = k / MX, rx = k - ry * MX;
      spn[k] = __ldg(dn + (long long)wrapi(y0 + ry - 1, Ly) * Lx + wrapi(x0 + rx - 1, Lx));
    }
  __syncthreads();
  // mu = a phi + b phi^3 - kappa lap_D phi (Eqs. 5, 31) on the tile + 1
  for (int k = tid; k < MX * MY; k += D_NT) {
    const int my = k / MX, mx = k - my * MX, q = (my + 1) * PX + mx + 1;
    const double c = sphi[q];
    smu[k] = fma(fma(p.b, c * c, p.a), c, -p.kappa * lapD(sphi, q, PX, p));
  }
  __syncthreads();
  if (!ok) return;
  // F (Eq. 28), n, u* (Eqs. 12, 18)
  double gx, gy;
  const int km = (ly + 1) * MX + lx + 1;
  grad2(smu, km, MX, p, gx, gy);
  const double ph = sphi[(ly + 2) * PX + lx + 2];
  double Fx = -ph * gx, Fy = -ph * gy;
  if constexpr (TGEN) {  // + d_D((cs^2 - T) n); the constant part of n drops out
    grad2(spn, km, MX, p, gx, gy);
    Fx = fma(p.cs2mT, gx, Fx);
    Fy = fma(p.cs2mT, gy, Fy);
  }
  const double dens = (h0 + ((h1 + h3) + (h2 + h4))) + ((h5 + h7) + (h6 + h8));
  const double d5 = h5 - h7, d6 = h6 - h8;
  const double jx = (h1 - h3) + (d5 - d6), jy = (h2 - h4) + (d5 + d6);
  const double n = 1.0 + dens;
  Fx = fma(n, p.gx, Fx);
  Fy = fma(n, p.gy, Fy);
  const double inv_n = 1.0 / n;
  const double ux = fma(0.5, Fx, jx) * inv_n, uy = fma(0.5, Fy, jy) * inv_n;
  const long long s = (long long)y * Lx + x;
  if constexpr (MODE == COLLIDE_MOMENTS) {
    stg[s] = n;
    stg[Sz + s] = ph;
    stg[2 * Sz + s] = ux;
    stg[3 * Sz + s] = uy;
    return;
  }
  const double om = p.tau_inv, keep = 1.0 - om, uF = fma(ux, Fx, uy * Fy);
  const double base = fma(-1.5 * n, fma(ux, ux, uy * uy), dens);
  const double iso = fma(om, base, (-3.0 * p.pref) * uF);  // w iso = A base - 3 B u.F
  const double an3 = (3.0 * om) * n, b3 = 3.0 * p.pref;
  const double w0 = q9_w(0), w1 = q9_w(1), w2 = q9_w(5);
  double *dst = hout + s;
  dst[0] = fma(keep, h0, w0 * iso);
  auto pair = [&](int i, double hi, double hb, double iw, double q, double r, double eu15) {
    const double O = q + r, E = fma(eu15, fma(2.0, r, q), iw);
    dst[i * Sz] = fma(keep, hi, E) + O;
    dst[(i + 2) * Sz] = fma(keep, hb, E) - O;
  };
  const double tx = 1.5 * ux, ty = 1.5 * uy;
  {
    const double A = w1 * an3, B = w1 * b3, iw = w1 * iso;
    pair(1, h1, h3, iw, A * ux, B * Fx, tx);
    pair(2, h2, h4, iw, A * uy, B * Fy, ty);
  }
  {  // e = (1, 1) and (-1, 1)
    const double A = w2 * an3, B = w2 * b3, iw = w2 * iso;
    const double qx = A * ux, qy = A * uy, rx = B * Fx, ry = B * Fy;
    pair(5, h5, h7, iw, qx + qy, rx + ry, tx + ty);
    pair(6, h6, h8, iw, qy - qx, ry - rx, ty - tx);
  }
  uout[s] = ux;
  uout[Sz + s] = uy;
}

// One substep of Eqs. 32-36 on a TX x TY tile: phi and u* staged with halo 3,
// phih on the tile + 2, psi on the tile + 1, the new phi on the tile.
// STENCIL: the operators of Eqs. 30-31 (printed advection form only).
template <int TX, int TY, int NT, bool FLUX, bool STENCIL>
__global__ void __launch_bounds__(NT)
    fd2d_f64_kernel(const double *__restrict__ phi, const double *__restrict__ u, double *__restrict__ out,
                    KParams<double> p) {
  constexpr int W = TX + 6, H = TY + 6, WA = TX + 4, HA = TY + 4, WP = TX + 2, HP = TY + 2;
  __shared__ double sp[W * H], su[W * H], sv[W * H], sa[WA * HA];
  double *sq = su;  // psi takes u's place once phih is formed
  const int Lx = p.Lx, Ly = p.Ly, tid = threadIdx.x;
  const long long Sz = (long long)Lx * Ly;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  for (int k = tid; k < W * H; k += NT) {
    const int ry = k / W, rx = k - ry * W;
    const long long g = (long long)wrapi(y0 + ry - 3, Ly) * Lx + wrapi(x0 + rx - 3, Lx);
    sp[k] = __ldg(phi + g);
    su[k] = __ldg(u + g);
    sv[k] = __ldg(u + Sz + g);
  }
  __syncthreads();
  auto lap = [&](const double *f, int k, int pitch) {
    if constexpr (STENCIL) return lapD(f, k, pitch, p);
    return fma(-4.0, f[k], (f[k - pitch] + f[k + pitch]) + (f[k - 1] + f[k + 1]));
  };
  for (int j = tid; j < WA * HA; j += NT) {
    const int ay = j / WA, ax = j - ay * WA, k = (ay + 1) * W + ax + 1;
    const double ph = sp[k], uc = su[k], vc = sv[k];
    const double pl = sp[k - 1], pr = sp[k + 1], pd = sp[k - W], pu = sp[k + W];
    if constexpr (!FLUX) {
      double d;
      if constexpr (STENCIL) {
        const double dux = fma(p.M, (su[k - W + 1] - su[k - W - 1]) + (su[k + W + 1] - su[k + W - 1]),
                               p.N * (su[k + 1] - su[k - 1]));
        const double dvy = fma(p.M, (sv[k + W + 1] - sv[k - W + 1]) + (sv[k + W - 1] - sv[k - W - 1]),
                               p.N * (sv[k + W] - sv[k - W]));
        d = (dux + dvy) + (fabs(uc) + fabs(vc));
      } else {
        d = fma(0.5, (su[k + 1] - su[k - 1]) + (sv[k + W] - sv[k - W]), fabs(uc) + fabs(vc));
      }
      double t = -d * ph;
      t = fma(fabs(uc), neg(uc) ? pr : pl, t);
      t = fma(fabs(vc), neg(vc) ? pu : pd, t);
      sa[j] = fma(p.dt, t, ph);
    } else {  // face velocities doubled, dt halved
      const double Upx = uc + su[k + 1], Umx = su[k - 1] + uc, Upy = vc + sv[k + W], Umy = sv[k - W] + vc;
      double t = -Upx * (neg(Upx) ? pr : ph);
      t = fma(Umx, neg(Umx) ? ph : pl, t);
      t = fma(-Upy, neg(Upy) ? pu : ph, t);
      t = fma(Umy, neg(Umy) ? ph : pd, t);
      sa[j] = fma(0.5 * p.dt, t, ph);
    }
  }
  __syncthreads();
  for (int j = tid; j < WP * HP; j += NT) {
    const int qy = j / WP, qx = j - qy * WP, k = (qy + 1) * WA + qx + 1;
    const double h = sa[k], c = p.cubic_at_half ? h : sp[(qy + 2) * W + qx + 2];
    sq[j] = fma(p.a, h, fma(p.b, c * c * c, -p.kappa * lap(sa, k, WA)));
  }
  __syncthreads();
  for (int j = tid; j < TX * TY; j += NT) {
    const int ly = j / TX, lx = j - ly * TX, x = x0 + lx, y = y0 + ly;
    if (x < Lx && y < Ly)
      out[(long long)y * Lx + x] = fma(p.dtG, lap(sq, (ly + 1) * WP + lx + 1, WP), sa[(ly + 2) * WA + lx + 2]);
  }
}

template <int TX, int TY, int NT>
cudaError_t fd2d_f64_tiles(const KParams<double> &p, const double *src, const double *u, double *dst, cudaStream_t s) {
  const dim3 grid((p.Lx + TX - 1) / TX, (p.Ly + TY - 1) / TY);
  if (p.adv_variant == LBM_ADV_FLUX)
    fd2d_f64_kernel<TX, TY, NT, true, false><<<grid, NT, 0, s>>>(src, u, dst, p);
  else if (p.stencil_fd)
    fd2d_f64_kernel<TX, TY, NT, false, true><<<grid, NT, 0, s>>>(src, u, dst, p);
  else
    fd2d_f64_kernel<TX, TY, NT, false, false><<<grid, NT, 0, s>>>(src, u, dst, p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t collide2d_f64(lbm_handle *h, int in, int force_on, int mode) {
  const KParams<double> p = make_params<double>(h, force_on);
  const dim3 grid((p.Lx + D_TX - 1) / D_TX, (p.Ly + D_TY - 1) / D_TY);
  const double *hin = static_cast<const double *>(h->h[in]), *phi = static_cast<const double *>(h->phi[in]);
  const double *dn = static_cast<const double *>(h->dn);
  double *hout = static_cast<double *>(h->h[1 - in]), *u = static_cast<double *>(h->u);
  auto launch = [&](auto kernel) { kernel<<<grid, D_NT, 0, h->stream>>>(hin, hout, phi, dn, u, h->staging, p); };
  const bool tgen = p.cs2mT != 0.0;
  if (mode == COLLIDE_STEP)
    tgen ? launch(collide2d_f64_kernel<true, COLLIDE_STEP>) : launch(collide2d_f64_kernel<false, COLLIDE_STEP>);
  else
    tgen ? launch(collide2d_f64_kernel<true, COLLIDE_MOMENTS>) : launch(collide2d_f64_kernel<false, COLLIDE_MOMENTS>);
  return cudaGetLastError();
}

// rows: output rows of a tile, 8 (16 x 8) or 16 (32 x 16)
cudaError_t fd2d_f64(lbm_handle *h, const KParams<double> &p, const double *src, double *dst, int rows) {
  const double *u = static_cast<const double *>(h->u);
  return rows == 8 ? fd2d_f64_tiles<16, 8, 128>(p, src, u, dst, h->stream)
                   : fd2d_f64_tiles<32, 16, 256>(p, src, u, dst, h->stream);
}

}  // namespace hlbm
