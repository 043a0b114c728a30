// kernels_3d_f64.cu -- the D3Q19 step with FP64 populations (the accuracy path).
//
// The GB300 issues about two FP64 operations per clock and SM, 1/64 of its
// FP32 rate, so these kernels are bound by their FP64 operation count and by
// how evenly the sites fall on the SMs; bytes, index arithmetic and loads are
// free beside it.  Hence, unlike the FP32 kernels:
//   - no halo is ever recomputed: every field is formed once per site (mu,
//     phih, psi and the new phi each in a pass of its own, their planes living
//     in the handle's FP64 staging buffer between the passes);
//   - one site per thread over a flat site index, 128 threads a block, so any
//     shape spreads over all SMs (64^3: 2048 blocks, the fullest SM 4 % over
//     the mean);
//   - the expressions are arranged for the fewest FP64 operations: upwind
//     sides from the sign bit (integer pipe), the two gradients of a plane
//     from shared diagonal differences, no products with zero components of
//     e_i, the even and odd parts of opposite directions formed once.
// 64^3, one LB step with m = 8 on a GB300: FD 1397 us (shared-memory tile
// kernel, halo 3 recomputed 7.4 times) -> 152 us, collide 222 -> 121 us.
#include "lbm_common.cuh"

namespace hlbm {

namespace {

constexpr int F64_THREADS = 128;

// Site of this thread and the offsets of its periodic neighbours.
struct Site3 {
  unsigned s;
  int x, y, z;
  long long xm, xp, ym, yp, zm, zp;  // offsets from s
};

__device__ __forceinline__ bool site3(const KParams<double> &p, Site3 &n) {
  const unsigned Lx = p.Lx, Ly = p.Ly, Lz = p.Lz;
  const unsigned long long s = blockIdx.x * (unsigned long long)F64_THREADS + threadIdx.x;
  if (s >= (unsigned long long)Lx * Ly * Lz) return false;
  n.s = (unsigned)s;  // at most 2^31 sites
  const unsigned r = n.s / Lx;
  n.x = n.s - r * Lx;
  n.z = r / Ly;
  n.y = r - n.z * Ly;
  const long long row = Lx, pl = (long long)Lx * Ly;
  n.xm = n.x == 0 ? (long long)Lx - 1 : -1;
  n.xp = n.x == (int)Lx - 1 ? 1 - (long long)Lx : 1;
  n.ym = n.y == 0 ? (Ly - 1) * row : -row;
  n.yp = n.y == (int)Ly - 1 ? -(long long)(Ly - 1) * row : row;
  n.zm = n.z == 0 ? (Lz - 1) * pl : -pl;
  n.zp = n.z == (int)Lz - 1 ? -(long long)(Lz - 1) * pl : pl;
  return true;
}

// the sign bit, on the integer pipe (a zero velocity of either sign picks a
// side whose product is zero)
__device__ __forceinline__ bool neg(double v) { return __double2hiint(v) < 0; }

// phih (Eqs. 32-35), printed form: phi + dt (|u| phi_up,x + |v| phi_up,y +
// |w| phi_up,z - phi (div u + |u| + |v| + |w|)); flux form: phi - dt (sum of
// face fluxes), the face velocities doubled and dt halved.
template <bool FLUX>
__global__ void __launch_bounds__(F64_THREADS)
    fd3_adv_f64_kernel(const double *__restrict__ phi, const double *__restrict__ u, double *__restrict__ A,
                       KParams<double> p) {
  Site3 n;
  if (!site3(p, n)) return;
  const long long Sz = (long long)p.Lx * p.Ly * p.Lz;
  const double *f = phi + n.s, *uu = u + n.s, *vv = uu + Sz, *ww = vv + Sz;
  const double ph = __ldg(f);
  const double pxm = __ldg(f + n.xm), pxp = __ldg(f + n.xp), pym = __ldg(f + n.ym), pyp = __ldg(f + n.yp),
               pzm = __ldg(f + n.zm), pzp = __ldg(f + n.zp);
  const double uc = __ldg(uu), um = __ldg(uu + n.xm), up = __ldg(uu + n.xp);
  const double vc = __ldg(vv), vm = __ldg(vv + n.ym), vp = __ldg(vv + n.yp);
  const double wc = __ldg(ww), wm = __ldg(ww + n.zm), wp = __ldg(ww + n.zp);
  double r;
  if constexpr (!FLUX) {
    const double div2 = ((up - um) + (vp - vm)) + (wp - wm);
    const double d = fma(0.5, div2, (fabs(uc) + fabs(vc)) + fabs(wc));
    double t = -d * ph;
    t = fma(fabs(uc), neg(uc) ? pxp : pxm, t);
    t = fma(fabs(vc), neg(vc) ? pyp : pym, t);
    t = fma(fabs(wc), neg(wc) ? pzp : pzm, t);
    r = fma(p.dt, t, ph);
  } else {
    double t = 0.0;
    auto flux = [&](double cm, double cc, double cp, double fm, double fp) {
      const double Up = cc + cp, Um = cm + cc;
      t = fma(-Up, neg(Up) ? fp : ph, t);
      t = fma(Um, neg(Um) ? ph : fm, t);
    };
    flux(um, uc, up, pxm, pxp);
    flux(vm, vc, vp, pym, pyp);
    flux(wm, wc, wp, pzm, pzp);
    r = fma(0.5 * p.dt, t, ph);
  }
  A[n.s] = r;
}

__device__ __forceinline__ double lap7(const double *f, const Site3 &n, double c) {
  const double sum = ((__ldg(f + n.xm) + __ldg(f + n.xp)) + (__ldg(f + n.ym) + __ldg(f + n.yp))) +
                     (__ldg(f + n.zm) + __ldg(f + n.zp));
  return fma(-6.0, c, sum);
}

// psi = a phih + b phi^3 - kappa lap phih (Eq. 36)
__global__ void __launch_bounds__(F64_THREADS)
    fd3_psi_f64_kernel(const double *__restrict__ A, const double *__restrict__ phi, double *__restrict__ P,
                       KParams<double> p) {
  Site3 n;
  if (!site3(p, n)) return;
  const double h = __ldg(A + n.s), c = p.cubic_at_half ? h : __ldg(phi + n.s);
  const double lap = lap7(A + n.s, n, h);
  P[n.s] = fma(p.a, h, fma(p.b, c * c * c, -p.kappa * lap));
}

// phi^{n+1} = phih + dt Gamma lap psi (Eq. 36)
__global__ void __launch_bounds__(F64_THREADS)
    fd3_phi_f64_kernel(const double *__restrict__ P, const double *__restrict__ A, double *__restrict__ out,
                       KParams<double> p) {
  Site3 n;
  if (!site3(p, n)) return;
  out[n.s] = fma(p.dtG, lap7(P + n.s, n, __ldg(P + n.s)), __ldg(A + n.s));
}

// mu = a phi + b phi^3 - kappa lap_D phi (Eqs. 5, 31)
__global__ void __launch_bounds__(F64_THREADS)
    mu3_f64_kernel(const double *__restrict__ phi, double *__restrict__ mu, KParams<double> p) {
  Site3 n;
  if (!site3(p, n)) return;
  const double *f = phi + n.s;
  const double c = __ldg(f);
  const double faces = ((__ldg(f + n.xm) + __ldg(f + n.xp)) + (__ldg(f + n.ym) + __ldg(f + n.yp))) +
                       (__ldg(f + n.zm) + __ldg(f + n.zp));
  auto ring = [&](long long am, long long ap, long long bm, long long bp) {
    return (__ldg(f + am + bm) + __ldg(f + am + bp)) + (__ldg(f + ap + bm) + __ldg(f + ap + bp));
  };
  const double edges = (ring(n.xm, n.xp, n.ym, n.yp) + ring(n.xm, n.xp, n.zm, n.zp)) + ring(n.ym, n.yp, n.zm, n.zp);
  const double lap = fma(p.Q, faces, fma(p.R, edges, p.C0 * c));
  mu[n.s] = fma(fma(p.b, c * c, p.a), c, -p.kappa * lap);
}

// d_D f (Eq. 30): the four edge neighbours of a plane (a, b) give the
// differences P = f(+,+) - f(-,-) and D = f(+,-) - f(-,+), whose sum belongs
// to the a derivative and whose difference to the b derivative.
template <typename F>
__device__ __forceinline__ void grad3(const KParams<double> &p, const Site3 &n, F &&at, double &gx, double &gy,
                                      double &gz) {
  const double pxy = at(n.xp + n.yp) - at(n.xm + n.ym), dxy = at(n.xp + n.ym) - at(n.xm + n.yp);
  const double pxz = at(n.xp + n.zp) - at(n.xm + n.zm), dxz = at(n.xp + n.zm) - at(n.xm + n.zp);
  const double pyz = at(n.yp + n.zp) - at(n.ym + n.zm), dyz = at(n.yp + n.zm) - at(n.ym + n.zp);
  gx = fma(p.M, (pxy + dxy) + (pxz + dxz), p.N * (at(n.xp) - at(n.xm)));
  gy = fma(p.M, (pxy - dxy) + (pyz + dyz), p.N * (at(n.yp) - at(n.ym)));
  gz = fma(p.M, (pxz - dxz) + (pyz - dyz), p.N * (at(n.zp) - at(n.zm)));
}

// Force, moments, collision and streaming of one site per thread (steps 2-4),
// or its moments.  An opposite pair (i, i + 1) takes
//   f_i  = (1 - 1/tau) f_i  + E + O,  f_ib = (1 - 1/tau) f_ib + E - O,
//   O = q + r,  q = 3 A n (e.u),  r = 3 B (e.F),
//   E = A base - 3 B u.F + 1.5 (e.u)(q + 2 r),
// with A = w / tau, B = w (1 - 1/2tau), base = n - 1 - 1.5 n u^2 (Eqs. 15, 29).
template <bool TGEN, int MODE>
__global__ void __launch_bounds__(F64_THREADS, 4)
    collide3_f64_kernel(const double *__restrict__ hin, double *__restrict__ hout, const double *__restrict__ phi,
                        const double *__restrict__ mu, const double *__restrict__ dn, double *__restrict__ uout,
                        double *__restrict__ stg, KParams<double> p) {
  Site3 n;
  if (!site3(p, n)) return;
  const long long Sz = (long long)p.Lx * p.Ly * p.Lz;
  const unsigned s = n.s;
  // f_i(r) = buf_i(r - e_i)
  double h[19];
  const double *src = hin + s;
#define LD(i, off) h[i] = __ldg(src + (i)*Sz + (off))
  LD(0, 0);
  LD(1, n.xm);
  LD(2, n.xp);
  LD(3, n.ym);
  LD(4, n.yp);
  LD(5, n.zm);
  LD(6, n.zp);
  LD(7, n.xm + n.ym);    // (1,1,0)
  LD(8, n.xp + n.yp);    // (-1,-1,0)
  LD(9, n.xm + n.yp);    // (1,-1,0)
  LD(10, n.xp + n.ym);   // (-1,1,0)
  LD(11, n.xm + n.zm);   // (1,0,1)
  LD(12, n.xp + n.zp);   // (-1,0,-1)
  LD(13, n.xm + n.zp);   // (1,0,-1)
  LD(14, n.xp + n.zm);   // (-1,0,1)
  LD(15, n.ym + n.zm);   // (0,1,1)
  LD(16, n.yp + n.zp);   // (0,-1,-1)
  LD(17, n.ym + n.zp);   // (0,1,-1)
  LD(18, n.yp + n.zm);   // (0,-1,1)
#undef LD
  // F = -phi d_D mu (Eq. 28)
  double gx, gy, gz;
  grad3(p, n, [&](long long o) { return __ldg(mu + s + o); }, gx, gy, gz);
  const double ph = __ldg(phi + s);
  double Fx = -ph * gx, Fy = -ph * gy, Fz = -ph * gz;
  if constexpr (TGEN) {  // + d_D((cs^2 - T) n); the constant part of n drops out
    grad3(p, n, [&](long long o) { return __ldg(dn + s + o); }, gx, gy, gz);
    Fx = fma(p.cs2mT, gx, Fx);
    Fy = fma(p.cs2mT, gy, Fy);
    Fz = fma(p.cs2mT, gz, Fz);
  }
  double dens = h[0];
#pragma unroll
  for (int i = 1; i < 19; i += 2) dens += h[i] + h[i + 1];
  auto d = [&](int i) { return h[i] - h[i + 1]; };
  const double d7 = d(7), d9 = d(9), d11 = d(11), d13 = d(13), d15 = d(15), d17 = d(17);
  const double jx = d(1) + ((d7 + d9) + (d11 + d13));
  const double jy = d(3) + ((d7 - d9) + (d15 + d17));
  const double jz = d(5) + ((d11 - d13) + (d15 - d17));
  const double nn = 1.0 + dens;
  Fx = fma(nn, p.gx, Fx);
  Fy = fma(nn, p.gy, Fy);
  Fz = fma(nn, p.gz, Fz);
  // u* (Eq. 18)
  const double inv_n = 1.0 / nn;
  const double ux = fma(0.5, Fx, jx) * inv_n, uy = fma(0.5, Fy, jy) * inv_n, uz = fma(0.5, Fz, jz) * inv_n;
  if constexpr (MODE == COLLIDE_MOMENTS) {
    stg[s] = nn;
    stg[Sz + s] = ph;
    stg[2 * Sz + s] = ux;
    stg[3 * Sz + s] = uy;
    stg[4 * Sz + s] = uz;
    return;
  }
  const double usq = fma(ux, ux, fma(uy, uy, uz * uz)), uF = fma(ux, Fx, fma(uy, Fy, uz * Fz));
  const double om = p.tau_inv, keep = 1.0 - om;
  const double base = fma(-1.5 * nn, usq, dens), m3uF = -3.0 * uF;
  // per weight class (rest, faces, edges): the isotropic part and the factors of e.u and e.F
  const double w0 = q19_w(0), w1 = q19_w(1), w2 = q19_w(7);
  const double iso = fma(om, base, p.pref * m3uF);  // w iso = A base - 3 B u.F
  const double an3 = 3.0 * om * nn, b3 = 3.0 * p.pref;
  double *dst = hout + s;
  dst[0] = fma(keep, h[0], w0 * iso);
  auto pair = [&](int i, double iso_w, double q, double r, double eu15) {
    const double O = q + r, E = fma(eu15, fma(2.0, r, q), iso_w);
    dst[i * Sz] = fma(keep, h[i], E) + O;
    dst[(i + 1) * Sz] = fma(keep, h[i + 1], E) - O;
  };
  {
    const double A = w1 * an3, B = w1 * b3, iw = w1 * iso;
    pair(1, iw, A * ux, B * Fx, 1.5 * ux);
    pair(3, iw, A * uy, B * Fy, 1.5 * uy);
    pair(5, iw, A * uz, B * Fz, 1.5 * uz);
  }
  {
    // q, r and 1.5 e.u are linear in e: the edges add or subtract the axes' parts
    const double A = w2 * an3, B = w2 * b3, iw = w2 * iso;
    const double qx = A * ux, qy = A * uy, qz = A * uz, rx = B * Fx, ry = B * Fy, rz = B * Fz;
    const double tx = 1.5 * ux, ty = 1.5 * uy, tz = 1.5 * uz;
    pair(7, iw, qx + qy, rx + ry, tx + ty);
    pair(9, iw, qx - qy, rx - ry, tx - ty);
    pair(11, iw, qx + qz, rx + rz, tx + tz);
    pair(13, iw, qx - qz, rx - rz, tx - tz);
    pair(15, iw, qy + qz, ry + rz, ty + tz);
    pair(17, iw, qy - qz, ry - rz, ty - tz);
  }
  uout[s] = ux;
  uout[Sz + s] = uy;
  uout[2 * Sz + s] = uz;
}

unsigned blocks_of(const lbm_handle *h) { return (unsigned)((h->S + F64_THREADS - 1) / F64_THREADS); }

}  // namespace

// Staging planes between the passes (the entry points that use the buffer for
// their own data, lbm_init_fields and the read-backs, leave nothing in it):
// phih in plane 0, psi in plane 1, mu in the scratch plane 5 (a moments pass
// writes planes 0 to 4 while it reads mu).
cudaError_t fd3_f64(lbm_handle *h, int in) {
  const KParams<double> p = make_params<double>(h, 0);
  const unsigned nb = blocks_of(h);
  const double *u = static_cast<const double *>(h->u), *src = static_cast<const double *>(h->phi[in]);
  double *A = h->staging, *P = h->staging + h->S;
  for (int j = 0; j < h->m; ++j) {
    double *dst = static_cast<double *>(((h->m - 1 - j) % 2 == 0) ? h->phi[1 - in] : h->phi[2]);
    if (p.adv_variant == LBM_ADV_FLUX)
      fd3_adv_f64_kernel<true><<<nb, F64_THREADS, 0, h->stream>>>(src, u, A, p);
    else
      fd3_adv_f64_kernel<false><<<nb, F64_THREADS, 0, h->stream>>>(src, u, A, p);
    fd3_psi_f64_kernel<<<nb, F64_THREADS, 0, h->stream>>>(A, src, P, p);
    fd3_phi_f64_kernel<<<nb, F64_THREADS, 0, h->stream>>>(P, A, dst, p);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    src = dst;
  }
  return cudaSuccess;
}

cudaError_t collide3_f64(lbm_handle *h, int in, int force_on, int mode) {
  const KParams<double> p = make_params<double>(h, force_on);
  const unsigned nb = blocks_of(h);
  const double *hin = static_cast<const double *>(h->h[in]), *phi = static_cast<const double *>(h->phi[in]);
  const double *dn = static_cast<const double *>(h->dn);
  double *hout = static_cast<double *>(h->h[1 - in]), *u = static_cast<double *>(h->u), *stg = h->staging;
  double *mu = stg + 5 * h->S;
  mu3_f64_kernel<<<nb, F64_THREADS, 0, h->stream>>>(phi, mu, p);
  const bool tgen = p.cs2mT != 0.0;
  if (mode == COLLIDE_STEP) {
    if (tgen)
      collide3_f64_kernel<true, COLLIDE_STEP><<<nb, F64_THREADS, 0, h->stream>>>(hin, hout, phi, mu, dn, u, stg, p);
    else
      collide3_f64_kernel<false, COLLIDE_STEP><<<nb, F64_THREADS, 0, h->stream>>>(hin, hout, phi, mu, dn, u, stg, p);
  } else {
    if (tgen)
      collide3_f64_kernel<true, COLLIDE_MOMENTS><<<nb, F64_THREADS, 0, h->stream>>>(hin, hout, phi, mu, dn, u, stg, p);
    else
      collide3_f64_kernel<false, COLLIDE_MOMENTS><<<nb, F64_THREADS, 0, h->stream>>>(hin, hout, phi, mu, dn, u, stg, p);
  }
  return cudaGetLastError();
}

}  // namespace hlbm
