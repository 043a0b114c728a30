// kernels_3d.cu -- D3Q19 hot path on sm_103a (the 3D generalisation of the
// paper's D2Q9 scheme).  Same structure as the 2D kernels:
//   collide3d : phi tile + halo 2 in shared memory -> mu (Eq. 5, 19-point lap_D)
//               -> F (Eq. 28, 19-point d_D) -> pull streaming -> n, u* -> BGK
//               with the Guo forcing term (Eqs. 15, 17, 29).
//   fd3d      : `sub` substeps of Eqs. 32-36 (7-point Laplacian) per launch,
//               blocked in shared memory with halo 3 per substep.
//   density3d : n - 1 for the T != 1/3 force term.
// Stencils (3D reading of Eqs. 30-31): d_D has N on the two face neighbours
// along the axis and M on the eight edge neighbours with a non-zero component
// along it (2N + 8M = 1); lap_D has Q on the six faces, R on the twelve edges
// and -(6Q + 12R) at the centre (Q + 4R = 1).
#include <algorithm>
#include <cstdlib>

#include "lbm_common.cuh"

namespace hlbm {

// FP64 populations (kernels_3d_f64.cu)
cudaError_t collide3_f64(lbm_handle *h, int in, int force_on, int mode);
cudaError_t fd3_f64(lbm_handle *h, int in);

namespace {

constexpr int C3_TX = 32, C3_TY = 8, C3_TZ = 8;  // block 32 x 8; z-planes per thread

// Wraps x in [-L, 2L) into [0, L).
__device__ __forceinline__ int wrap1_3(int x, int L) { return x < 0 ? x + L : (x >= L ? x - L : x); }

template <typename S, typename C, bool TGEN, int MODE, int MINB>
__global__ void __launch_bounds__(256, MINB)
    collide3d_kernel(const S *__restrict__ hin, S *__restrict__ hout, const C *__restrict__ phi,
                     const C *__restrict__ dn, C *__restrict__ uout, double *__restrict__ stg,
                     KParams<C> p) {
  constexpr int PX = C3_TX + 4, PY = C3_TY + 4, PZ = C3_TZ + 4;
  constexpr int MX = C3_TX + 2, MY = C3_TY + 2, MZ = C3_TZ + 2;
  __shared__ C sphi[PZ][PY][PX];
  __shared__ C smu[MZ][MY][MX];
  const int Lx = p.Lx, Ly = p.Ly, Lz = p.Lz;
  const long long Sz = (long long)Lx * Ly * Lz;
  const int x0 = blockIdx.x * C3_TX, y0 = blockIdx.y * C3_TY, z0 = blockIdx.z * C3_TZ;
  const int tid = threadIdx.y * 32 + threadIdx.x;
  const int lx = threadIdx.x, ly = threadIdx.y, x = x0 + lx, y = y0 + ly;
  const bool site_ok = x < Lx && y < Ly;
  const int xc = site_ok ? x : 0, yc_ = site_ok ? y : 0;
  const int xm = xc == 0 ? Lx - 1 : xc - 1, xp = xc == Lx - 1 ? 0 : xc + 1;
  const int ym = yc_ == 0 ? Ly - 1 : yc_ - 1, yp = yc_ == Ly - 1 ? 0 : yc_ + 1;
  const long long pl = (long long)Lx * Ly;
  const long long yc = (long long)yc_ * Lx, ymo = (long long)ym * Lx, ypo = (long long)yp * Lx;
  // f_i(r) = buf_i(r - e_i) of plane z (clamped into the lattice for threads
  // without a site; their values are never used)
  // FP16 storage: the populations stay in their stored scale 2^s through the
  // sums and the collision (the scale is folded into the moments and the
  // weights), which is exact for a power of two and saves a multiply per
  // population read and written
  constexpr bool FOLD = !std::is_same<S, C>::value;
  const C ld_scale = FOLD ? C(1) : p.inv_scale, st_scale = FOLD ? C(1) : p.scale;
  const C wsc = FOLD ? p.scale : C(1);  // weights in the stored scale
  auto load_plane = [&](C (&hv)[19], int z) {
    const int zm = z == 0 ? Lz - 1 : z - 1, zp = z == Lz - 1 ? 0 : z + 1;
    const long long zc = (long long)z * pl, zmo = (long long)zm * pl, zpo = (long long)zp * pl;
#define LD(i, zz, yy, xx) hv[i] = Store<S, C>::ld(hin + (i)*Sz + (zz) + (yy) + (xx), ld_scale)
    LD(0, zc, yc, xc);
    LD(1, zc, yc, xm);
    LD(2, zc, yc, xp);
    LD(3, zc, ymo, xc);
    LD(4, zc, ypo, xc);
    LD(5, zmo, yc, xc);
    LD(6, zpo, yc, xc);
    LD(7, zc, ymo, xm);    // (1,1,0)
    LD(8, zc, ypo, xp);    // (-1,-1,0)
    LD(9, zc, ypo, xm);    // (1,-1,0)
    LD(10, zc, ymo, xp);   // (-1,1,0)
    LD(11, zmo, yc, xm);   // (1,0,1)
    LD(12, zpo, yc, xp);   // (-1,0,-1)
    LD(13, zpo, yc, xm);   // (1,0,-1)
    LD(14, zmo, yc, xp);   // (-1,0,1)
    LD(15, zmo, ymo, xc);  // (0,1,1)
    LD(16, zpo, ypo, xc);  // (0,-1,-1)
    LD(17, zpo, ymo, xc);  // (0,1,-1)
    LD(18, zmo, ypo, xc);  // (0,-1,1)
#undef LD
  };
  // the first plane's populations are in flight while phi and mu are staged
  C hv[19], hn[19];
  if (z0 < Lz) load_plane(hv, z0);
  const bool big = Lx >= PX && Ly >= PY && Lz >= PZ;
  // phi on the tile + halo 2: one (x, y) column per thread, the z loop inside
  for (int k = tid; k < PX * PY; k += 256) {
    const int ry = k / PX, rx = k - ry * PX;
    const int gx = big ? wrap1_3(x0 + rx - 2, Lx) : wrapi(x0 + rx - 2, Lx);
    const int gy = big ? wrap1_3(y0 + ry - 2, Ly) : wrapi(y0 + ry - 2, Ly);
    const C *col = phi + (long long)gy * Lx + gx;
    C v[PZ];  // the whole column in flight before any of it is stored
#pragma unroll
    for (int rz = 0; rz < PZ; ++rz) {
      const int gz = big ? wrap1_3(z0 + rz - 2, Lz) : wrapi(z0 + rz - 2, Lz);
      v[rz] = col[(long long)gz * pl];
    }
#pragma unroll
    for (int rz = 0; rz < PZ; ++rz) sphi[rz][ry][rx] = v[rz];
  }
  __syncthreads();
  // mu on the tile + 1: one (x, y) column per thread marching in z, the 3 x 3
  // neighbourhoods of phi on planes z - 1, z, z + 1 in registers (9 new
  // loads per site)
  for (int k = tid; k < MX * MY; k += 256) {
    const int my = k / MX, mx = k - my * MX, cy = my + 1, cx = mx + 1;
    C w[3][3][3];  // [plane][dy][dx]
#pragma unroll
    for (int pz = 0; pz < 2; ++pz)
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) w[pz + 1][a][b] = sphi[pz][cy - 1 + a][cx - 1 + b];
#pragma unroll 2
    for (int mz = 0; mz < MZ; ++mz) {
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          w[0][a][b] = w[1][a][b];
          w[1][a][b] = w[2][a][b];
          w[2][a][b] = sphi[mz + 2][cy - 1 + a][cx - 1 + b];
        }
      const C c = w[1][1][1];
      const C faces = ((w[1][1][0] + w[1][1][2]) + (w[1][0][1] + w[1][2][1])) + (w[0][1][1] + w[2][1][1]);
      const C edges = ((w[1][0][0] + w[1][0][2]) + (w[1][2][0] + w[1][2][2])) +
                      ((w[0][1][0] + w[0][1][2]) + (w[2][1][0] + w[2][1][2])) +
                      ((w[0][0][1] + w[0][2][1]) + (w[2][0][1] + w[2][2][1]));
      const C lap = p.Q * faces + p.R * edges + p.C0 * c;
      smu[mz][my][mx] = p.a * c + p.b * c * c * c - p.kappa * lap;
    }
  }
  __syncthreads();

  if (!site_ok) return;
#pragma unroll 1
  for (int lz = 0; lz < C3_TZ; ++lz) {
    const int z = z0 + lz;
    if (z >= Lz) break;
    // the next plane's populations are issued before this plane is computed
    if (lz + 1 < C3_TZ && z + 1 < Lz) load_plane(hn, z + 1);
    const int mx = lx + 1, my = ly + 1, mz = lz + 1;
    // d_D mu along x, y, z
    auto grad = [&](const C (*f)[MY][MX], C &gx_, C &gy_, C &gz_) {
      gx_ = p.N * (f[mz][my][mx + 1] - f[mz][my][mx - 1]) +
            p.M * (((f[mz][my - 1][mx + 1] - f[mz][my - 1][mx - 1]) +
                    (f[mz][my + 1][mx + 1] - f[mz][my + 1][mx - 1])) +
                   ((f[mz - 1][my][mx + 1] - f[mz - 1][my][mx - 1]) +
                    (f[mz + 1][my][mx + 1] - f[mz + 1][my][mx - 1])));
      gy_ = p.N * (f[mz][my + 1][mx] - f[mz][my - 1][mx]) +
            p.M * (((f[mz][my + 1][mx - 1] - f[mz][my - 1][mx - 1]) +
                    (f[mz][my + 1][mx + 1] - f[mz][my - 1][mx + 1])) +
                   ((f[mz - 1][my + 1][mx] - f[mz - 1][my - 1][mx]) +
                    (f[mz + 1][my + 1][mx] - f[mz + 1][my - 1][mx])));
      gz_ = p.N * (f[mz + 1][my][mx] - f[mz - 1][my][mx]) +
            p.M * (((f[mz + 1][my][mx - 1] - f[mz - 1][my][mx - 1]) +
                    (f[mz + 1][my][mx + 1] - f[mz - 1][my][mx + 1])) +
                   ((f[mz + 1][my - 1][mx] - f[mz - 1][my - 1][mx]) +
                    (f[mz + 1][my + 1][mx] - f[mz - 1][my + 1][mx])));
    };
    C gmx, gmy, gmz;
    grad(smu, gmx, gmy, gmz);
    const C ph = sphi[lz + 2][ly + 2][lx + 2];
    C Fx = -ph * gmx, Fy = -ph * gmy, Fz = -ph * gmz;
    if constexpr (TGEN) {
      // d_D((cs2 - T) n) from the density pass, read directly (rare path)
      auto pn = [&](int dx, int dy, int dz) {
        const long long g = ((long long)wrapi(z + dz, Lz) * Ly + wrapi(y + dy, Ly)) * Lx +
                            wrapi(x + dx, Lx);
        return p.cs2mT * (C(1) + dn[g]);
      };
      Fx += p.N * (pn(1, 0, 0) - pn(-1, 0, 0)) +
            p.M * (((pn(1, -1, 0) - pn(-1, -1, 0)) + (pn(1, 1, 0) - pn(-1, 1, 0))) +
                   ((pn(1, 0, -1) - pn(-1, 0, -1)) + (pn(1, 0, 1) - pn(-1, 0, 1))));
      Fy += p.N * (pn(0, 1, 0) - pn(0, -1, 0)) +
            p.M * (((pn(-1, 1, 0) - pn(-1, -1, 0)) + (pn(1, 1, 0) - pn(1, -1, 0))) +
                   ((pn(0, 1, -1) - pn(0, -1, -1)) + (pn(0, 1, 1) - pn(0, -1, 1))));
      Fz += p.N * (pn(0, 0, 1) - pn(0, 0, -1)) +
            p.M * (((pn(-1, 0, 1) - pn(-1, 0, -1)) + (pn(1, 0, 1) - pn(1, 0, -1))) +
                   ((pn(0, -1, 1) - pn(0, -1, -1)) + (pn(0, 1, 1) - pn(0, 1, -1))));
    }
    const long long zc = (long long)z * pl;
    C dens = hv[0];
#pragma unroll
    for (int i = 1; i < 19; ++i) dens += hv[i];
    C jx = C(0), jy = C(0), jz = C(0);
#pragma unroll
    for (int i = 1; i < 19; ++i) {
      if (q19_ex(i) > 0) jx += hv[i];
      if (q19_ex(i) < 0) jx -= hv[i];
      if (q19_ey(i) > 0) jy += hv[i];
      if (q19_ey(i) < 0) jy -= hv[i];
      if (q19_ez(i) > 0) jz += hv[i];
      if (q19_ez(i) < 0) jz -= hv[i];
    }
    if constexpr (FOLD) {
      dens *= p.inv_scale;
      jx *= p.inv_scale;
      jy *= p.inv_scale;
      jz *= p.inv_scale;
    }
    const C n = C(1) + dens;
    Fx += n * p.gx;
    Fy += n * p.gy;
    Fz += n * p.gz;
    const C inv_n = C(1) / n;
    const C ux = (jx + C(0.5) * Fx) * inv_n;
    const C uy = (jy + C(0.5) * Fy) * inv_n;
    const C uz = (jz + C(0.5) * Fz) * inv_n;
    const long long s = zc + yc + x;
    if constexpr (MODE == COLLIDE_MOMENTS) {
      stg[s] = (double)n;
      stg[Sz + s] = (double)ph;
      stg[2 * Sz + s] = (double)ux;
      stg[3 * Sz + s] = (double)uy;
      stg[4 * Sz + s] = (double)uz;
#pragma unroll
      for (int i = 0; i < 19; ++i) hv[i] = hn[i];
      continue;
    }
    const C usq = ux * ux + uy * uy + uz * uz;
    const C uF = ux * Fx + uy * Fy + uz * Fz;
    const C om = p.tau_inv, keep = C(1) - p.tau_inv;
    const C base = dens - n * (C(1.5) * usq);  // the u-independent and |u|^2 parts
    if constexpr (FOLD) {
      // BGK + Guo source (Eqs. 15, 17, 29) per opposite pair (i, i + 1): with
      // A = w / tau and B = w (1 - 1/2tau) per weight class, the part even in
      // e_i is E = A (base + 4.5 n (e.u)^2) + B (9 (e.u)(e.F) - 3 u.F) and the
      // odd part O = 3 A n (e.u) + 3 B (e.F); f_i = (1 - 1/tau) f_i + E + O,
      // f_ib = (1 - 1/tau) f_ib + E - O.  e.u and e.F take only the non-zero
      // components of e_i (the compiler may not drop a product with a zero
      // component under IEEE rules).  FP16 storage only: the kernel is
      // issue-bound there (417 against 444 us a launch at 256^3), while the
      // FP32 kernel, closer to the memory roof, ran slower with this form
      // (473 against 464 us), so it keeps the one below.
      const C n45 = C(4.5) * n, m3uF = C(-3) * uF;
      const C A0 = om * C(q19_w(0)) * wsc, B0 = p.pref * C(q19_w(0)) * wsc;
      const C A1 = om * C(q19_w(1)) * wsc, B1 = p.pref * C(q19_w(1)) * wsc;  // faces
      const C A2 = om * C(q19_w(7)) * wsc, B2 = p.pref * C(q19_w(7)) * wsc;  // edges
      const C An3_1 = C(3) * A1 * n, An3_2 = C(3) * A2 * n;
      Store<S, C>::st(hout + s, keep * hv[0] + (A0 * base + B0 * m3uF), st_scale);
      auto edot = [](int ex, int ey, int ez, C a, C b, C c) {
        C r = ex > 0 ? a : (ex < 0 ? -a : C(0));
        if (ey != 0) r = ex != 0 ? (ey > 0 ? r + b : r - b) : (ey > 0 ? b : -b);
        if (ez != 0) r = (ex != 0 || ey != 0) ? (ez > 0 ? r + c : r - c) : (ez > 0 ? c : -c);
        return r;
      };
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const int i = 2 * k + 1, ib = i + 1;  // e_ib = -e_i
        const bool face = k < 3;
        const C A = face ? A1 : A2, B = face ? B1 : B2, An3 = face ? An3_1 : An3_2;
        const C eu = edot(q19_ex(i), q19_ey(i), q19_ez(i), ux, uy, uz);
        const C eF = edot(q19_ex(i), q19_ey(i), q19_ez(i), Fx, Fy, Fz);
        const C se = n45 * eu * eu + base;
        const C fe = C(9) * eu * eF + m3uF;
        const C E = A * se + B * fe;
        const C O = An3 * eu + C(3) * B * eF;
        Store<S, C>::st(hout + i * Sz + s, (keep * hv[i] + E) + O, st_scale);
        Store<S, C>::st(hout + ib * Sz + s, (keep * hv[ib] + E) - O, st_scale);
      }
    } else {
      // BGK + Guo source (Eqs. 15, 17, 29) per opposite pair (i, i + 1): the
      // parts even and odd in e_i are formed once and added / subtracted
      const C n3 = C(3) * n, n45 = C(4.5) * n;
      const C pF3 = C(3) * p.pref, pF9 = C(9) * p.pref, puF = C(3) * p.pref * uF;
      {
        const C w = C(q19_w(0));
        Store<S, C>::st(hout + s, keep * hv[0] + om * (w * base) + w * (-puF), st_scale);
      }
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const int i = 2 * k + 1, ib = i + 1;  // e_ib = -e_i
        const C w = C(q19_w(i));
        const C eu = C(q19_ex(i)) * ux + C(q19_ey(i)) * uy + C(q19_ez(i)) * uz;
        const C eF = C(q19_ex(i)) * Fx + C(q19_ey(i)) * Fy + C(q19_ez(i)) * Fz;
        const C even = w * (base + n45 * eu * eu);
        const C odd = w * (n3 * eu);
        const C Feven = w * (pF9 * eu * eF - puF);
        const C Fodd = w * (pF3 * eF);
        Store<S, C>::st(hout + i * Sz + s, keep * hv[i] + om * (even + odd) + (Feven + Fodd), st_scale);
        Store<S, C>::st(hout + ib * Sz + s, keep * hv[ib] + om * (even - odd) + (Feven - Fodd), st_scale);
      }
    }
    uout[s] = ux;
    uout[Sz + s] = uy;
    uout[2 * Sz + s] = uz;
#pragma unroll
    for (int i = 0; i < 19; ++i) hv[i] = hn[i];
  }
}

template <typename C, int TX, int TY, int TZ>
__global__ void __launch_bounds__(256)
    fd3d_kernel(const C *__restrict__ phi_in, const C *__restrict__ u, C *__restrict__ phi_out,
                KParams<C> p, int sub) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C *sm = reinterpret_cast<C *>(smem_raw);
  const int H = 3 * sub, RX = TX + 2 * H, RY = TY + 2 * H, RZ = TZ + 2 * H;
  const int R = RX * RY * RZ, PL = RX * RY;
  C *sp = sm, *sh = sm + R, *sq = sm + 2 * R, *su = sm + 3 * R, *sv = sm + 4 * R,
    *sw = sm + 5 * R;
  const int Lx = p.Lx, Ly = p.Ly, Lz = p.Lz;
  const long long Sz = (long long)Lx * Ly * Lz;
  const int x0 = blockIdx.x * TX - H, y0 = blockIdx.y * TY - H, z0 = blockIdx.z * TZ - H;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int rz = 0; rz < RZ; ++rz)
    for (int ry = ty; ry < RY; ry += 8) {
      const long long row = ((long long)wrapi(z0 + rz, Lz) * Ly + wrapi(y0 + ry, Ly)) * Lx;
      for (int rx = tx; rx < RX; rx += 32) {
        const long long g = row + wrapi(x0 + rx, Lx);
        const int k = rz * PL + ry * RX + rx;
        sp[k] = phi_in[g];
        su[k] = u[g];
        sv[k] = u[Sz + g];
        sw[k] = u[2 * Sz + g];
      }
    }
  __syncthreads();
  const C dt = p.dt, dtG = p.dtG;
#pragma unroll 1
  for (int s = 1; s <= sub; ++s) {
    int lo = 3 * s - 2;
    for (int rz = lo; rz < RZ - lo; ++rz)
      for (int ry = lo + ty; ry < RY - lo; ry += 8)
        for (int rx = lo + tx; rx < RX - lo; rx += 32) {
          const int k = rz * PL + ry * RX + rx;
          const C ph = sp[k];
          C tend;
          if (p.adv_variant == LBM_ADV_PAPER) {
            const C ua = su[k], va = sv[k], wa = sw[k];
            const C dux = (su[k + 1] - su[k - 1]) / C(2);
            const C dpx = ua < C(0) ? sp[k + 1] - ph : ph - sp[k - 1];
            const C duy = (sv[k + RX] - sv[k - RX]) / C(2);
            const C dpy = va < C(0) ? sp[k + RX] - ph : ph - sp[k - RX];
            const C duz = (sw[k + PL] - sw[k - PL]) / C(2);
            const C dpz = wa < C(0) ? sp[k + PL] - ph : ph - sp[k - PL];
            tend = (ph * dux + ua * dpx);
            tend += (ph * duy + va * dpy);
            tend += (ph * duz + wa * dpz);
          } else {
            auto flux = [&](const C *uu, int st) {
              const C Up = C(0.5) * (uu[k] + uu[k + st]);
              const C Um = C(0.5) * (uu[k - st] + uu[k]);
              const C Jp = Up > C(0) ? Up * ph : Up * sp[k + st];
              const C Jm = Um > C(0) ? Um * sp[k - st] : Um * ph;
              return Jp - Jm;
            };
            tend = flux(su, 1);
            tend += flux(sv, RX);
            tend += flux(sw, PL);
          }
          sh[k] = ph - dt * tend;
        }
    __syncthreads();
    lo = 3 * s - 1;
    for (int rz = lo; rz < RZ - lo; ++rz)
      for (int ry = lo + ty; ry < RY - lo; ry += 8)
        for (int rx = lo + tx; rx < RX - lo; rx += 32) {
          const int k = rz * PL + ry * RX + rx;
          const C hk = sh[k];
          const C c = p.cubic_at_half ? hk : sp[k];
          C lap = sh[k - PL];
          lap += sh[k - RX];
          lap += sh[k - 1];
          lap += C(-6) * hk;
          lap += sh[k + 1];
          lap += sh[k + RX];
          lap += sh[k + PL];
          sq[k] = p.a * hk + p.b * (c * c * c) - p.kappa * lap;
        }
    __syncthreads();
    lo = 3 * s;
    for (int rz = lo; rz < RZ - lo; ++rz)
      for (int ry = lo + ty; ry < RY - lo; ry += 8)
        for (int rx = lo + tx; rx < RX - lo; rx += 32) {
          const int k = rz * PL + ry * RX + rx;
          C lap = sq[k - PL];
          lap += sq[k - RX];
          lap += sq[k - 1];
          lap += C(-6) * sq[k];
          lap += sq[k + 1];
          lap += sq[k + RX];
          lap += sq[k + PL];
          sp[k] = sh[k] + dtG * lap;
        }
    __syncthreads();
  }
  for (int rz = H; rz < H + TZ; ++rz) {
    const int gz = z0 + rz;
    if (gz >= Lz) break;
    for (int ry = H + ty; ry < H + TY; ry += 8) {
      const int gy = y0 + ry;
      if (gy >= Ly) break;
      for (int rx = H + tx; rx < H + TX; rx += 32) {
        const int gx = x0 + rx;
        if (gx < Lx) phi_out[((long long)gz * Ly + gy) * Lx + gx] = sp[rz * PL + ry * RX + rx];
      }
    }
  }
}

// ---- FD 3D, FP32: three passes per substep --------------------------------------
// One site per thread over the whole lattice, periodic neighbours by index
// arithmetic; no halo is recomputed.  Pass 1: phih (Eqs. 32-35) from the
// 7-point neighbourhood of phi and u*; pass 2: psi = a phih + b phi^3 -
// kappa lap phih (Eq. 36); pass 3: phi^{n+1} = phih + dt Gamma lap psi.  The
// expressions are those of fd3d_kernel, in the same order.
struct Nbr3 {
  long long s, xm, xp, ym, yp, zm, zp;
};

__device__ __forceinline__ bool nbr3(const KParams<float> &p, Nbr3 &n) {
  const int Lx = p.Lx, Ly = p.Ly, Lz = p.Lz;
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y, z = blockIdx.z;
  if (x >= Lx || y >= Ly) return false;
  const long long PL = (long long)Lx * Ly;
  n.s = z * PL + (long long)y * Lx + x;
  n.xm = n.s + (x == 0 ? Lx - 1 : -1);
  n.xp = n.s + (x == Lx - 1 ? 1 - Lx : 1);
  n.ym = n.s + (y == 0 ? (long long)(Ly - 1) * Lx : -(long long)Lx);
  n.yp = n.s + (y == Ly - 1 ? -(long long)(Ly - 1) * Lx : (long long)Lx);
  n.zm = n.s + (z == 0 ? (Lz - 1) * PL : -PL);
  n.zp = n.s + (z == Lz - 1 ? -(Lz - 1) * PL : PL);
  return true;
}

template <bool FLUX>
__global__ void __launch_bounds__(256)
    fd3_adv_kernel(const float *__restrict__ phi, const float *__restrict__ u,
                   float *__restrict__ A, KParams<float> p) {
  Nbr3 n;
  if (!nbr3(p, n)) return;
  const long long Sz = (long long)p.Lx * p.Ly * p.Lz;
  const float *v = u + Sz, *w = u + 2 * Sz;
  const float ph = __ldg(phi + n.s);
  float tend;
  if constexpr (!FLUX) {
    const float ua = __ldg(u + n.s), va = __ldg(v + n.s), wa = __ldg(w + n.s);
    const float dux = (__ldg(u + n.xp) - __ldg(u + n.xm)) / 2.f;
    const float dpx = ua < 0.f ? __ldg(phi + n.xp) - ph : ph - __ldg(phi + n.xm);
    const float duy = (__ldg(v + n.yp) - __ldg(v + n.ym)) / 2.f;
    const float dpy = va < 0.f ? __ldg(phi + n.yp) - ph : ph - __ldg(phi + n.ym);
    const float duz = (__ldg(w + n.zp) - __ldg(w + n.zm)) / 2.f;
    const float dpz = wa < 0.f ? __ldg(phi + n.zp) - ph : ph - __ldg(phi + n.zm);
    tend = (ph * dux + ua * dpx);
    tend += (ph * duy + va * dpy);
    tend += (ph * duz + wa * dpz);
  } else {
    auto flux = [&](const float *uu, long long m, long long q) {
      const float uc = __ldg(uu + n.s);
      const float Up = 0.5f * (uc + __ldg(uu + q));
      const float Um = 0.5f * (__ldg(uu + m) + uc);
      const float Jp = Up > 0.f ? Up * ph : Up * __ldg(phi + q);
      const float Jm = Um > 0.f ? Um * __ldg(phi + m) : Um * ph;
      return Jp - Jm;
    };
    tend = flux(u, n.xm, n.xp);
    tend += flux(v, n.ym, n.yp);
    tend += flux(w, n.zm, n.zp);
  }
  A[n.s] = ph - p.dt * tend;
}

__global__ void __launch_bounds__(256)
    fd3_psi_kernel(const float *__restrict__ A, const float *__restrict__ phi,
                   float *__restrict__ P, KParams<float> p) {
  Nbr3 n;
  if (!nbr3(p, n)) return;
  const float hk = __ldg(A + n.s);
  const float c = p.cubic_at_half ? hk : __ldg(phi + n.s);
  float lap = __ldg(A + n.zm);
  lap += __ldg(A + n.ym);
  lap += __ldg(A + n.xm);
  lap += -6.f * hk;
  lap += __ldg(A + n.xp);
  lap += __ldg(A + n.yp);
  lap += __ldg(A + n.zp);
  P[n.s] = p.a * hk + p.b * (c * c * c) - p.kappa * lap;
}

__global__ void __launch_bounds__(256)
    fd3_phi_kernel(const float *__restrict__ P, const float *__restrict__ A,
                   float *__restrict__ phi_out, KParams<float> p) {
  Nbr3 n;
  if (!nbr3(p, n)) return;
  float lap = __ldg(P + n.zm);
  lap += __ldg(P + n.ym);
  lap += __ldg(P + n.xm);
  lap += -6.f * __ldg(P + n.s);
  lap += __ldg(P + n.xp);
  lap += __ldg(P + n.yp);
  lap += __ldg(P + n.zp);
  phi_out[n.s] = __ldg(A + n.s) + p.dtG * lap;
}

// ---- the same three passes, four x-sites per thread, marching in z ------------
// (Lx a multiple of 4.)  A warp covers 128 consecutive x (float4 per lane, the
// x neighbours by shuffles; lanes at a warp or lattice edge load their wrapped
// neighbour), a block 8 rows of y, and each thread marches nz planes in z
// (at most F3V_NZ, fewer when the lattice is too small to fill the GPU)
// keeping the z-1, z, z+1 values of the marched field in registers.
constexpr int F3V_NZ = 16;

struct Vq {
  int x4, xc, y, z0, z1, lane;
  bool ok;
};

__device__ __forceinline__ Vq vq_of(const KParams<float> &p, int nz) {
  Vq q;
  q.lane = threadIdx.x;
  q.x4 = 4 * (blockIdx.x * 32 + threadIdx.x);
  q.xc = min(q.x4, p.Lx - 4);  // loads of lanes past the lattice edge stay in bounds
  q.ok = q.x4 < p.Lx;
  q.y = blockIdx.y * 8 + threadIdx.y;
  q.z0 = blockIdx.z * nz;
  q.z1 = min(q.z0 + nz, p.Lz);
  return q;
}

__device__ __forceinline__ const float *row_of(const float *a, int y, int z, const KParams<float> &p) {
  return a + ((long long)z * p.Ly + y) * p.Lx;
}

__device__ __forceinline__ float4 ld4g(const float *row, int x) {
  return __ldg(reinterpret_cast<const float4 *>(row + x));
}

// values at x4 - 1 and x4 + 4 of `row`, whose quad at x4 is c
__device__ __forceinline__ void xnbr4(const float *row, float4 c, const Vq &q, int Lx, float &l,
                                      float &r) {
  l = __shfl_up_sync(0xffffffffu, c.w, 1);
  r = __shfl_down_sync(0xffffffffu, c.x, 1);
  if (q.lane == 0 || q.x4 == 0) l = __ldg(row + (q.x4 == 0 ? Lx - 1 : q.xc - 1));
  if (q.lane == 31 || q.x4 + 4 >= Lx) r = __ldg(row + (q.x4 + 4 >= Lx ? 0 : q.x4 + 4));
}

__device__ __forceinline__ float cmp4(const float4 &v, int j) {
  return j == 0 ? v.x : (j == 1 ? v.y : (j == 2 ? v.z : v.w));
}

// phih of one site in flux form: phi at the site and its six neighbours, the u*
// components along each axis at the neighbours that the face velocities need
__device__ __forceinline__ float adv_site_flux(float ph, float pxm, float pxp, float pym, float pyp, float pzm,
                                               float pzp, float uxm, float ua, float uxp, float vym, float va,
                                               float vyp, float wzm, float wa, float wzp, float dt) {
  auto flux = [&](float cm, float cc, float cp, float fm, float fp) {
    const float Up = 0.5f * (cc + cp);
    const float Um = 0.5f * (cm + cc);
    const float Jp = Up > 0.f ? Up * ph : Up * fp;
    const float Jm = Um > 0.f ? Um * fm : Um * ph;
    return Jp - Jm;
  };
  float tend = flux(uxm, ua, uxp, pxm, pxp);
  tend += flux(vym, va, vyp, pym, pyp);
  tend += flux(wzm, wa, wzp, pzm, pzp);
  return ph - dt * tend;
}

// packed FP32 pairs (sites 0,1 and 2,3 of a quad)
__device__ __forceinline__ float2 pf2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }

// phih of a quad (Eqs. 32-35), in the printed form on packed pairs where the
// neighbours are pairs, each operation explicitly rounded.  Of an axis's phi (u_+ -
// u_-)/2 + u dphi, dphi the upwind difference, the second product is rounded and the
// first fused along x and y, the other way round along z; phi is halved instead of
// the difference.  (Central and second differences would save the selects, but round
// differently.)
template <bool FLUX>
__device__ __forceinline__ float4 adv_quad(const float4 &pc, float pl, float pr, const float4 &pym, const float4 &pyp,
                                           const float4 &pzm, const float4 &pzp, const float4 &uc, float ul, float ur,
                                           const float4 &vym, const float4 &vc, const float4 &vyp, const float4 &wzm,
                                           const float4 &wc, const float4 &wzp, float dt) {
  if constexpr (!FLUX) {
    const float2 m1 = pf2(-1.f, -1.f);
    auto sub = [&](float2 a, float2 b) { return pfma(m1, b, a); };
    // the upwind difference of phi (scalar: packed differences under the selects
    // take more registers, 256^3 step 1247 against 1237 us)
    auto upw = [](float2 u, float2 c, float2 m, float2 q) {
      return pf2(u.x < 0.f ? __fsub_rn(q.x, c.x) : __fsub_rn(c.x, m.x),
                 u.y < 0.f ? __fsub_rn(q.y, c.y) : __fsub_rn(c.y, m.y));
    };
    auto half = [&](float2 c, float2 xm, float2 xp, float2 u, float2 um, float2 up, float2 ym, float2 yp, float2 v,
                    float2 vm, float2 vp, float2 zm, float2 zp, float2 w, float2 wm, float2 wp) {
      const float2 h = pmul(pf2(0.5f, 0.5f), c);
      float2 t = pfma(h, sub(up, um), pmul(u, upw(u, c, xm, xp)));
      t = padd(t, pfma(h, sub(vp, vm), pmul(v, upw(v, c, ym, yp))));
      t = padd(t, pfma(w, upw(w, c, zm, zp), pmul(h, sub(wp, wm))));
      return pfma(pf2(-dt, -dt), t, c);
    };
    const float2 a = half(lo2(pc), pf2(pl, pc.x), pf2(pc.y, pc.z), lo2(uc), pf2(ul, uc.x), pf2(uc.y, uc.z), lo2(pym),
                          lo2(pyp), lo2(vc), lo2(vym), lo2(vyp), lo2(pzm), lo2(pzp), lo2(wc), lo2(wzm), lo2(wzp));
    const float2 b = half(hi2(pc), pf2(pc.y, pc.z), pf2(pc.w, pr), hi2(uc), pf2(uc.y, uc.z), pf2(uc.w, ur), hi2(pym),
                          hi2(pyp), hi2(vc), hi2(vym), hi2(vyp), hi2(pzm), hi2(pzp), hi2(wc), hi2(wzm), hi2(wzp));
    return make_float4(a.x, a.y, b.x, b.y);
  } else {
    float e[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      e[j] = adv_site_flux(cmp4(pc, j), j == 0 ? pl : cmp4(pc, j - 1), j == 3 ? pr : cmp4(pc, j + 1), cmp4(pym, j),
                           cmp4(pyp, j), cmp4(pzm, j), cmp4(pzp, j), j == 0 ? ul : cmp4(uc, j - 1), cmp4(uc, j),
                           j == 3 ? ur : cmp4(uc, j + 1), cmp4(vym, j), cmp4(vc, j), cmp4(vyp, j), cmp4(wzm, j),
                           cmp4(wc, j), cmp4(wzp, j), dt);
    return make_float4(e[0], e[1], e[2], e[3]);
  }
}

// Asks for `bytes` (a multiple of 16) from the 16-byte aligned f on in L2.
__device__ __forceinline__ void l2_prefetch(const float *f, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(f), "r"(bytes) : "memory");
}

// Advection pass.  A row takes 2^lw lanes of a block of 256 threads (a warp
// may hold several short rows); with WRAP the whole row fits in them and the
// periodic x neighbours come from shuffles, otherwise the outermost lanes load
// theirs.  Offsets advance by planes instead of being recomputed per load.
// Bound by HBM on large lattices (57 us a launch at 256^3, 20 B/site at 0.87 of the
// copy bandwidth) and by load latency and the L1 pipe where L2 holds the fields (200 x
// 144 x 112: 11.7 us).  L2 prefetches, cache hints for u* and a reversed sweep changed
// nothing.  The loop over planes is unrolled by two: LB step at 256^3 1268 -> 1237 us
// (1257 by four; 1306 with registers for 3 or for 5 CTAs an SM).
template <bool FLUX, bool WRAP>
__global__ void __launch_bounds__(256, 4)
    fd3v_adv_kernel(const float *__restrict__ phi, const float *__restrict__ u,
                    float *__restrict__ A, KParams<float> p, int nz, int lw) {
  const int Lx = p.Lx, Ly = p.Ly, Lz = p.Lz, nq = Lx >> 2, LW = 1 << lw;
  const int lane = threadIdx.x & (LW - 1), qx = blockIdx.x * LW + lane;
  const int yr = blockIdx.y * (256 >> lw) + (threadIdx.x >> lw);
  const bool ok = qx < nq && yr < Ly;
  const int qc = min(qx, nq - 1), y = min(yr, Ly - 1);  // loads of idle lanes stay in bounds
  const int z0 = blockIdx.z * nz, z1 = min(z0 + nz, Lz);
  // element offsets in 32 bits (at most 2^31 sites); arithmetic wraps modulo 2^32
  const unsigned PL = (unsigned)Lx * Ly, Sz = PL * Lz;
  const unsigned ymo = y == 0 ? PL - Lx : 0u - Lx, ypo = y == Ly - 1 ? Lx - PL : (unsigned)Lx;
  const int xlo = qc == 0 ? Lx - 1 : -1, xro = qc == nq - 1 ? 4 - Lx : 4;  // x neighbours of the quad
  const int sl = WRAP && lane == 0 ? nq - 1 : lane - 1, sr = WRAP && lane == nq - 1 ? 0 : lane + 1;
  const bool el = !WRAP && (lane == 0 || qc == 0), er = !WRAP && (lane == LW - 1 || qc == nq - 1);
  auto ldq = [](const float *f, unsigned o) { return __ldg(reinterpret_cast<const float4 *>(f + o)); };
  auto xn = [&](const float *f, unsigned o, const float4 &c, float &l, float &r) {
    l = __shfl_sync(0xffffffffu, c.w, sl, LW);
    r = __shfl_sync(0xffffffffu, c.x, sr, LW);
    if (el) l = __ldg(f + (o + xlo));
    if (er) r = __ldg(f + (o + xro));
  };
  const float *v = u + Sz, *w = v + Sz;
  unsigned o = z0 * PL + (unsigned)y * Lx + 4 * qc;  // the quad in plane z
  const unsigned ob = z0 == 0 ? o + (Sz - PL) : o - PL;
  float4 pm = ldq(phi, ob), pc = ldq(phi, o), wm = ldq(w, ob), wc = ldq(w, o);
#pragma unroll 2
  for (int z = z0; z < z1; ++z) {
    const unsigned on = z == Lz - 1 ? o - (Sz - PL) : o + PL;
    const float4 pp = ldq(phi, on), wp = ldq(w, on);
    const float4 pym = ldq(phi, o + ymo), pyp = ldq(phi, o + ypo);
    const float4 uc = ldq(u, o), vc = ldq(v, o), vym = ldq(v, o + ymo), vyp = ldq(v, o + ypo);
    float pl, pr, ul, ur;
    xn(phi, o, pc, pl, pr);
    xn(u, o, uc, ul, ur);
    const float4 r = adv_quad<FLUX>(pc, pl, pr, pym, pyp, pm, pp, uc, ul, ur, vym, vc, vyp, wm, wc, wp, p.dt);
    if (ok) *reinterpret_cast<float4 *>(A + o) = r;
    o = on;
    pm = pc;
    pc = pp;
    wm = wc;
    wc = wp;
  }
}

// LAP7 of a field with the quad c at (y, z) and its neighbours, in the order
// z-1, y-1, x-1, centre, x+1, y+1, z+1 of the scalar kernels
template <bool PSI>
__global__ void __launch_bounds__(256)
    fd3v_lap_kernel(const float *__restrict__ F, const float *__restrict__ G,
                    float *__restrict__ out, KParams<float> p, int nz) {
  // PSI:  out = a F + b c^3 - kappa lap F, c = (cubic_at_half ? F : G)
  // else: out = G + dtG lap F
  const Vq q = vq_of(p, nz);
  if (q.y >= p.Ly) return;
  const int Lx = p.Lx, Ly = p.Ly, Lz = p.Lz;
  const int ym = q.y == 0 ? Ly - 1 : q.y - 1, yp = q.y == Ly - 1 ? 0 : q.y + 1;
  const int zb = q.z0 == 0 ? Lz - 1 : q.z0 - 1;
  float4 fm = ld4g(row_of(F, q.y, zb, p), q.xc), fc = ld4g(row_of(F, q.y, q.z0, p), q.xc);
  for (int z = q.z0; z < q.z1; ++z) {
    const int zn = z == Lz - 1 ? 0 : z + 1;
    const float *frow = row_of(F, q.y, z, p);
    const float4 fp = ld4g(row_of(F, q.y, zn, p), q.xc);
    const float4 fym = ld4g(row_of(F, ym, z, p), q.xc), fyp = ld4g(row_of(F, yp, z, p), q.xc);
    const float4 gc = ld4g(row_of(G, q.y, z, p), q.xc);
    float fl, fr;
    xnbr4(frow, fc, q, Lx, fl, fr);
    float e[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float hk = cmp4(fc, j);
      float lap = cmp4(fm, j);
      lap += cmp4(fym, j);
      lap += j == 0 ? fl : cmp4(fc, j - 1);
      lap += -6.f * hk;
      lap += j == 3 ? fr : cmp4(fc, j + 1);
      lap += cmp4(fyp, j);
      lap += cmp4(fp, j);
      if constexpr (PSI) {
        const float c = p.cubic_at_half ? hk : cmp4(gc, j);
        e[j] = p.a * hk + p.b * (c * c * c) - p.kappa * lap;
      } else {
        e[j] = cmp4(gc, j) + p.dtG * lap;
      }
    }
    if (q.ok)
      *reinterpret_cast<float4 *>(out + ((long long)z * Ly + q.y) * Lx + q.x4) =
          make_float4(e[0], e[1], e[2], e[3]);
    fm = fc;
    fc = fp;
  }
}

// ---- psi and the new phi in one z-marching kernel (whole rows: Lx % 4 == 0, Lx <= 256) ------
// The second and third passes of a substep fused: a CTA of 512 threads holds
// R = 512 / 2^lw rows of which R - 2 are written; a row takes 2^lw lanes with
// V quads (float4) each, quad q of lane l at x = 4 (q nl + l), nl lanes in use,
// so the periodic x neighbours come from shuffles.  Each thread computes psi =
// a phih + b phi^3 - kappa lap phih (Eq. 36) of its quads and marches in z
// with phih of planes z, z + 1, z + 2 in registers.  psi goes to a four-plane
// shared-memory ring; after one barrier the inner rows form phi^{n+1} = phih +
// dt Gamma lap psi (Eq. 36) of plane z from the ring.  psi never reaches
// global memory: a substep moves the advection pass's 20 B/site plus about 12
// B/site here, instead of 44 B.
// The arithmetic runs on packed FP32 pairs.  SEQ: in the order and with the fused
// products of the three-pass kernels; rows of 128 and 256 have an order of their
// own.  FP16 storage rounds a stored population to the other neighbour where phi
// or u* differ in a last bit (4e-5 of the populations and 1e-7 of phi after four
// steps of 200 x 144 x 112), so a row length keeps its operations and their order
// whichever kernel runs them; here they cost nothing measurable.
// Each iteration waits for loads issued one plane before; one thread asks for
// the CTA's rows (a contiguous range) in L2 two planes earlier still, which
// covers the latency of HBM: 40 us a launch at 256^3 against 62 us without
// (12 B/site at 0.74 of the copy bandwidth; with 16 warps an SM the rest is
// issue and shared-memory latency).
constexpr int F3F_NW = 16;

template <int V>
__device__ __forceinline__ void xnbr_row(const float4 (&c)[V], float (&l)[V], float (&r)[V]) {
  const int lane = threadIdx.x & 31;
  float sl[V], sr[V];
#pragma unroll
  for (int q = 0; q < V; ++q) {
    sl[q] = __shfl_sync(0xffffffffu, c[q].w, (lane + 31) & 31);
    sr[q] = __shfl_sync(0xffffffffu, c[q].x, (lane + 1) & 31);
  }
#pragma unroll
  for (int q = 0; q < V; ++q) {
    l[q] = lane == 0 ? sl[(q + V - 1) % V] : sl[q];
    r[q] = lane == 31 ? sr[(q + 1) % V] : sr[q];
  }
}

// The loads of iteration z + 1 (phih of plane z + 3, phih of plane z + 2 on
// the rows y -+ 1 and phi of plane z + 2) are issued before iteration z
// computes, so that they are in flight across its barrier (1.16x over
// loading them at the top of their own iteration).
// 7-point Laplacian of the quad c (x neighbours l, r of its ends; m, p in z,
// ym, yp in y) as two packed pairs: the z and y neighbours and the centre as
// pairs, the x neighbour sums (which straddle the pairs) scalar.  SEQ: one
// neighbour after the other, in the order of the scalar kernels.
template <bool SEQ>
__device__ __forceinline__ void lap7_quad(const float4 &c, const float4 &m, const float4 &p, const float4 &ym,
                                          const float4 &yp, float l, float r, float2 &lo, float2 &hi) {
  const float2 m6 = pf2(-6.f, -6.f), mid = pf2(c.y, c.z);
  if constexpr (SEQ) {
    lo = pfma(m6, lo2(c), padd(padd(lo2(m), lo2(ym)), pf2(l, c.x)));
    hi = pfma(m6, hi2(c), padd(padd(hi2(m), hi2(ym)), mid));
    lo = padd(padd(padd(lo, mid), lo2(yp)), lo2(p));
    hi = padd(padd(padd(hi, pf2(c.w, r)), hi2(yp)), hi2(p));
  } else {
    lo = pfma(m6, lo2(c), padd(padd(padd(lo2(m), lo2(p)), padd(lo2(ym), lo2(yp))), pf2(l + c.y, c.x + c.z)));
    hi = pfma(m6, hi2(c), padd(padd(padd(hi2(m), hi2(p)), padd(hi2(ym), hi2(yp))), pf2(c.y + c.w, c.z + r)));
  }
}

// A load that stays where it is written relative to barriers.
__device__ __forceinline__ float4 ldg4_here(const float *f) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(f));
  return v;
}

template <int V, int MINB, bool SEQ>
__global__ void __launch_bounds__(F3F_NW * 32, MINB)
    fd3f_kernel(const float *__restrict__ A, const float *__restrict__ G, float *__restrict__ out,
                KParams<float> p, int nz, int lw) {
  constexpr int NT = F3F_NW * 32;
  extern __shared__ __align__(16) float f3f_smem[];
  float4 *const sq = reinterpret_cast<float4 *>(f3f_smem);  // [4 planes][V][NT threads]
  const int LW = 1 << lw, lane = threadIdx.x & (LW - 1), row = threadIdx.x >> lw, R = NT >> lw;
  const int Lx = p.Lx, Ly = p.Ly, Lz = p.Lz, nq = Lx >> 2, nl = (nq + V - 1) / V;
  const unsigned plane = (unsigned)Lx * Ly, Sz = plane * Lz;  // element offsets in 32 bits, modulo 2^32
  const int yr = (int)blockIdx.y * (R - 2) - 1 + row;  // this thread's psi row (wrapped below)
  const int y = wrapi(yr, Ly);
  const unsigned ymo = y == 0 ? plane - Lx : 0u - Lx, ypo = y == Ly - 1 ? Lx - plane : (unsigned)Lx;
  const bool outr = row >= 1 && row <= R - 2 && yr < Ly && lane < nl;
  const int z0 = blockIdx.z * nz, z1 = min(z0 + nz, Lz);
  // columns of the quads (idle lanes and the missing last quad of an odd row
  // load a valid one and are never used)
  const unsigned x0 = 4 * min(lane, nl - 1), dx = 4 * (min(nl + min(lane, nl - 1), nq - 1) - min(lane, nl - 1));
  auto xo = [&](int q) { return q == 0 ? 0u : dx; };
  // x neighbours: quad j of the row is (q, lane) with j = q nl + lane; the
  // first quad's left neighbour is the last quad, lane e1 of q = V - 1
  const int e1 = nq - 1 - (V - 1) * nl;
  auto xn = [&](const float4 (&c)[V], float (&l)[V], float (&r)[V]) {
    if constexpr (V == 1) {
      l[0] = __shfl_sync(0xffffffffu, c[0].w, lane == 0 ? e1 : lane - 1, LW);
      r[0] = __shfl_sync(0xffffffffu, c[0].x, lane == e1 ? 0 : lane + 1, LW);
    } else {
      const float l0 = __shfl_sync(0xffffffffu, c[0].w, lane == 0 ? nl - 1 : lane - 1, LW);
      const float l1 = __shfl_sync(0xffffffffu, c[1].w, lane == 0 ? e1 : lane - 1, LW);
      const float r0 = __shfl_sync(0xffffffffu, c[0].x, lane == e1 ? 0 : lane + 1, LW);
      const float r1 = __shfl_sync(0xffffffffu, c[1].x, lane == nl - 1 ? 0 : lane + 1, LW);
      // an odd row's lane nl - 2 is the last of q = 1 but not of q = 0
      const float r0n = e1 == nl - 1 ? r0 : __shfl_sync(0xffffffffu, c[0].x, lane + 1, LW);
      l[0] = lane == 0 ? l1 : l0;
      l[1] = lane == 0 ? l0 : l1;
      r[0] = lane == nl - 1 ? r1 : r0n;
      r[1] = lane == e1 ? r0 : r1;
    }
  };
  auto ld = [&](const float *f, unsigned o, float4 (&v)[V]) {
#pragma unroll
    for (int q = 0; q < V; ++q) v[q] = ldg4_here(f + (o + xo(q)));
  };
  auto mv = [](float4 (&d)[V], const float4 (&s2)[V]) {
#pragma unroll
    for (int q = 0; q < V; ++q) d[q] = s2[q];
  };
  auto at = [&](int z) { return (unsigned)wrapi(z, Lz) * plane + (unsigned)y * Lx + x0; };
  float4 hm[V], hc[V], hp[V];     // phih of this row at planes z, z + 1, z + 2
  float4 hym[V], hyp[V], gc[V];   // phih of plane z + 1 on rows y -+ 1, phi of plane z + 1
  ld(A, at(z0 - 2), hm);
  ld(A, at(z0 - 1), hc);
  ld(A, at(z0), hp);
  ld(A, at(z0 - 1) + ymo, hym);
  ld(A, at(z0 - 1) + ypo, hyp);
  ld(G, at(z0 - 1), gc);
  // the CTA's rows of a plane (those that do not wrap) are one contiguous
  // range; one thread asks for them in L2 two iterations before they are loaded
  const int yb = max((int)blockIdx.y * (R - 2) - 1, 0), ye = min((int)blockIdx.y * (R - 2) + R - 1, Ly);
  const unsigned pf_off = (unsigned)yb * Lx, pf_bytes = (unsigned)(ye - yb) * Lx * 4;
  auto prefetch = [&](const float *f, int zz) {
    l2_prefetch(f + ((unsigned)wrap1(zz, Lz) * plane + pf_off), pf_bytes);
  };
  unsigned o2 = at(z0), o3 = at(z0 + 1);  // this row in planes z + 2 and z + 3
  int zn = wrapi(z0 + 1, Lz);
  for (int z = z0 - 2; z < z1; ++z) {
    float4 nhp[V], nym[V], nyp[V], ngc[V];
    if (threadIdx.x == 0 && z + 5 < z1 + 2 && z + 5 < 2 * Lz) {
      prefetch(A, z + 5);
      prefetch(G, z + 4);
    }
    ld(A, o3, nhp);
    ld(A, o2 + ymo, nym);
    ld(A, o2 + ypo, nyp);
    ld(G, o2, ngc);
    o2 = o3;
    zn = zn + 1 == Lz ? 0 : zn + 1;
    o3 += zn == 0 ? plane - Sz : plane;
    // psi of plane z + 1 on this row
    {
      float l[V], r[V];
      xn(hc, l, r);
      float4 *dst = sq + ((z + 1) & 3) * V * NT + threadIdx.x;
#pragma unroll
      for (int q = 0; q < V; ++q) {
        float2 L[2], o[2];
        lap7_quad<SEQ>(hc[q], hm[q], hp[q], hym[q], hyp[q], l[q], r[q], L[0], L[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float2 hk = k ? hi2(hc[q]) : lo2(hc[q]);
          const float2 cb = p.cubic_at_half ? hk : (k ? hi2(gc[q]) : lo2(gc[q]));
          const float2 a = pf2(p.a, p.a), b = pf2(p.b, p.b), mk = pf2(-p.kappa, -p.kappa), c3 = pmul(pmul(cb, cb), cb);
          o[k] = SEQ ? pfma(mk, L[k], pfma(a, hk, pmul(b, c3))) : pfma(a, hk, pfma(b, c3, pmul(mk, L[k])));
        }
        dst[q * NT] = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
      }
    }
    __syncthreads();
    // phi^{n+1} of plane z (psi planes z - 1, z, z + 1 are in the ring); the
    // first and last rows of the CTA take part in the shuffles only
    if (z >= z0) {
      auto sld = [&](int slot, int q, int rows) { return sq[(slot & 3) * V * NT + q * NT + threadIdx.x + rows * LW]; };
      const int dm = row >= 1 ? -1 : 0, dp = row <= R - 2 ? 1 : 0;
      float4 qc[V];
#pragma unroll
      for (int q = 0; q < V; ++q) qc[q] = sld(z, q, 0);
      float l[V], r[V];
      xn(qc, l, r);
      float *dst = out + ((unsigned)z * plane + (unsigned)y * Lx + x0);
#pragma unroll
      for (int q = 0; q < V; ++q) {
        const float4 qm = sld(z + 3, q, 0), qp = sld(z + 1, q, 0);
        const float4 qym = sld(z, q, dm), qyp = sld(z, q, dp);
        float2 L[2];
        lap7_quad<SEQ>(qc[q], qm, qp, qym, qyp, l[q], r[q], L[0], L[1]);
        const float2 g = pf2(p.dtG, p.dtG);
        const float2 o0 = pfma(g, L[0], lo2(hm[q])), o1 = pfma(g, L[1], hi2(hm[q]));
        if (outr && (q == 0 || lane <= e1)) *reinterpret_cast<float4 *>(dst + xo(q)) = make_float4(o0.x, o0.y, o1.x, o1.y);
      }
    }
    mv(hm, hc);
    mv(hc, hp);
    mv(hp, nhp);
    mv(hym, nym);
    mv(hyp, nyp);
    mv(gc, ngc);
  }
}

// ---- one whole FD substep, software-pipelined in z (Lx = 128 V, V = 1 or 2) ----
// The advection of Eqs. 32-35 fused with psi and the new phi of Eq. 36, with
// one barrier per plane.  A CTA of F3P_NW warps owns F3P_NW - 4 output rows;
// warp w owns row y0 - 2 + w, the whole row (V float4 per lane, quad q of
// lane l at x = 128 q + 4 l; periodic x neighbours by shuffles), and marches
// in z.  Iteration k runs three phases, each reading only what earlier
// iterations wrote, so that one barrier at its end orders them all:
//   C (warps 2 .. NW - 3): phi^{n+1} of plane k - 2 = phih + dt Gamma lap psi,
//     from psi of planes k - 3 .. k - 1 (three-slot ring; rows w -+ 1 of plane
//     k - 2) and phih of plane k - 2 (own row);
//   B (warps 1 .. NW - 2): psi of plane k = a phih + b phi^3 - kappa lap phih,
//     from phih of planes k - 1 .. k + 1 (four-slot ring; rows w -+ 1 of
//     plane k) into the psi ring;
//   A (all warps): phih of plane a = k + 2 into the phih ring.
// A warp writes only its own row of a ring, and the only same-iteration
// reuse of a slot is by the writing warp itself (C reads its own phih of
// plane k - 2 and psi of plane k - 3 before A and B overwrite those slots).
// The advection inputs arrive one plane ahead: u of the warps' 16 rows and v
// of 18 rows (y -+ 1) by bulk copies into a two-slot shared-memory ring (one
// mbarrier a slot; warp 0 issues plane a + 1 at the top of iteration k, after
// the barrier that ended the reads of its slot), phi and w of the own row in
// registers marching in z, and phi of rows y -+ 1 and the next planes' own-row
// phi and w loaded at the end of phase A, so that they are in flight across
// the barrier and phases C and B.  A substep reads phi and u* and writes the
// new phi (20 B/site, against 32 B/site for the advection pass followed by
// fd3f); the arithmetic per site is that of those two kernels (the same
// device functions and packed operations), so the results are equal bitwise.
// Every copy wait is bounded: a wait that gives up is reported through the
// barrier (all threads learn it together), the copies in flight are drained
// with a bound, and the CTA returns; the host reports LBM_ETIMEOUT.
constexpr int F3P_NW = 16;

__device__ int g_fd3p_err = 0;
__device__ unsigned long long g_fd3p_wait_ns = 500000000ull;

template <int V>
struct F3P {
  static constexpr int W = 128 * V;
  static constexpr int U_OFF = 0;                                // [2][NW][W]     u rows
  static constexpr int V_OFF = U_OFF + 2 * F3P_NW * W;           // [2][NW + 2][W] v rows
  static constexpr int H_OFF = V_OFF + 2 * (F3P_NW + 2) * W;     // [4][NW][W]     phih
  static constexpr int Q_OFF = H_OFF + 4 * F3P_NW * W;           // [3][NW][W]     psi
  static constexpr int FLOATS = Q_OFF + 3 * F3P_NW * W;
  static constexpr uint32_t TX_BYTES = (2 * F3P_NW + 2) * W * sizeof(float);  // one plane's copies
  static constexpr size_t smem = sizeof(float) * FLOATS + 16;    // + two mbarriers
};

template <bool FLUX, int V>
__global__ void __launch_bounds__(F3P_NW * 32, 1)
    fd3p_kernel(const float *__restrict__ G, const float *__restrict__ u, float *__restrict__ out,
                KParams<float> p, int nz) {
  constexpr int NW = F3P_NW, W = 128 * V;
  using L = F3P<V>;
  extern __shared__ __align__(16) float f3p_smem[];
  float(*su)[NW][W] = reinterpret_cast<float(*)[NW][W]>(f3p_smem + L::U_OFF);
  float(*sv)[NW + 2][W] = reinterpret_cast<float(*)[NW + 2][W]>(f3p_smem + L::V_OFF);
  float(*sh)[NW][W] = reinterpret_cast<float(*)[NW][W]>(f3p_smem + L::H_OFF);
  float(*sq)[NW][W] = reinterpret_cast<float(*)[NW][W]>(f3p_smem + L::Q_OFF);
  const uint32_t bar0 = su32(f3p_smem + L::FLOATS);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Ly = p.Ly, Lz = p.Lz;
  const long long plane = (long long)W * Ly, Sz = plane * Lz;
  const float *vv = u + Sz, *ww = u + 2 * Sz;
  const int y0 = blockIdx.y * (NW - 4);
  const int yr = y0 - 2 + warp;  // this warp's row (wrapped below)
  const int y = wrapi(yr, Ly), ym = wrapi(yr - 1, Ly), yp = wrapi(yr + 1, Ly);
  const bool psiw = warp >= 1 && warp <= NW - 2;             // warp-uniform
  const bool outw = warp >= 2 && warp <= NW - 3 && yr < Ly;  // warp-uniform
  const int z0 = blockIdx.z * nz, z1 = min(z0 + nz, Lz);
  const int a0 = z0 - 2, a1 = z1 + 1;  // planes phase A advects
  const bool cubic_half = p.cubic_at_half != 0;
  auto g4 = [&](const float *f, int yy, int zz, int q) {
    return __ldg(reinterpret_cast<const float4 *>(f + wrapi(zz, Lz) * plane + (long long)yy * W + 128 * q +
                                                  4 * lane));
  };
  auto ldrow = [&](const float *f, int yy, int zz, float4(&v)[V]) {
#pragma unroll
    for (int q = 0; q < V; ++q) v[q] = g4(f, yy, zz, q);
  };
  auto put = [&](float(*ring)[NW][W], int slot, const float4(&v)[V]) {
#pragma unroll
    for (int q = 0; q < V; ++q) *reinterpret_cast<float4 *>(&ring[slot][warp][128 * q + 4 * lane]) = v[q];
  };
  auto get = [&](const float *row, int q) { return *reinterpret_cast<const float4 *>(row + 128 * q + 4 * lane); };
  // u and v rows of plane pl (warp 0): 16 + 18 bulk copies of one row each
  auto issue = [&](int pl) {
    const int s = pl & 1;
    const uint32_t bar = bar0 + 8 * s;
    if (lane == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier reads of the slot first
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(L::TX_BYTES)
                   : "memory");
    }
    __syncwarp();
    const long long zo = (long long)wrapi(pl, Lz) * plane;
    for (int i = lane; i < 2 * NW + 2; i += 32) {
      const float *src;
      uint32_t dst;
      if (i < NW) {
        src = u + zo + (long long)wrapi(y0 - 2 + i, Ly) * W;
        dst = su32(&su[s][i][0]);
      } else {
        src = vv + zo + (long long)wrapi(y0 - 3 + (i - NW), Ly) * W;
        dst = su32(&sv[s][i - NW][0]);
      }
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
          "l"(src), "r"((uint32_t)(W * sizeof(float))), "r"(bar)
          : "memory");
    }
  };
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (warp == 0) {
    issue(a0);
    if (a0 + 1 <= a1) issue(a0 + 1);
  }
  // own-row phi of planes a - 1, a, a + 1 and w of the same (a = the plane
  // phase A advects next), phi of plane a on rows y -+ 1, and phi of plane k
  // (the cube of phase B)
  float4 P0[V], P1[V], P2[V], Pym[V], Pyp[V], W0[V], W1[V], W2[V], Pk[V];
  ldrow(G, y, a0 - 1, P0);
  ldrow(G, y, a0, P1);
  ldrow(G, y, a0 + 1, P2);
  ldrow(G, ym, a0, Pym);
  ldrow(G, yp, a0, Pyp);
  ldrow(ww, y, a0 - 1, W0);
  ldrow(ww, y, a0, W1);
  ldrow(ww, y, a0 + 1, W2);
#pragma unroll
  for (int q = 0; q < V; ++q) Pk[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  const float2 g2 = pf2(p.dtG, p.dtG);
  for (int k = z0 - 4; k <= z1 + 1; ++k) {
    if (warp == 0 && k >= z0 - 3 && k + 3 <= a1) issue(k + 3);
    // C: phi^{n+1} of plane k - 2
    if (k >= z0 + 2 && outw) {
      const int zc = k - 2;
      const float *qrow = &sq[(zc + 6) % 3][warp][0];
      float4 qc[V];
#pragma unroll
      for (int q = 0; q < V; ++q) qc[q] = get(qrow, q);
      float l[V], r[V];
      xnbr_row<V>(qc, l, r);
      float *orow = out + (long long)zc * plane + (long long)yr * W;
#pragma unroll
      for (int q = 0; q < V; ++q) {
        const float4 qm = get(&sq[(zc + 5) % 3][warp][0], q), qp = get(&sq[(zc + 7) % 3][warp][0], q);
        const float4 qym = get(&sq[(zc + 6) % 3][warp - 1][0], q), qyp = get(&sq[(zc + 6) % 3][warp + 1][0], q);
        const float4 hm = get(&sh[zc & 3][warp][0], q);
        float2 Lp[2];
        lap7_quad<false>(qc[q], qm, qp, qym, qyp, l[q], r[q], Lp[0], Lp[1]);
        const float2 o0 = pfma(g2, Lp[0], lo2(hm)), o1 = pfma(g2, Lp[1], hi2(hm));
        *reinterpret_cast<float4 *>(orow + 128 * q + 4 * lane) = make_float4(o0.x, o0.y, o1.x, o1.y);
      }
    }
    // B: psi of plane k
    if (k >= z0 - 1 && k <= z1 && psiw) {
      float4 hc[V];
#pragma unroll
      for (int q = 0; q < V; ++q) hc[q] = get(&sh[k & 3][warp][0], q);
      float l[V], r[V];
      xnbr_row<V>(hc, l, r);
      float4 o4[V];
#pragma unroll
      for (int q = 0; q < V; ++q) {
        const float4 hm = get(&sh[(k + 3) & 3][warp][0], q), hp = get(&sh[(k + 1) & 3][warp][0], q);
        const float4 hym = get(&sh[k & 3][warp - 1][0], q), hyp = get(&sh[k & 3][warp + 1][0], q);
        float2 Lp[2];
        lap7_quad<false>(hc[q], hm, hp, hym, hyp, l[q], r[q], Lp[0], Lp[1]);
        float2 o[2];
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
          const float2 hk = kk ? hi2(hc[q]) : lo2(hc[q]);
          const float2 cb = cubic_half ? hk : (kk ? hi2(Pk[q]) : lo2(Pk[q]));
          o[kk] = pfma(pf2(p.a, p.a), hk,
                       pfma(pf2(p.b, p.b), pmul(pmul(cb, cb), cb), pmul(pf2(-p.kappa, -p.kappa), Lp[kk])));
        }
        o4[q] = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
      }
      put(sq, (k + 6) % 3, o4);
    }
    // A: phih of plane a = k + 2, then the loads of plane a + 1
    bool ok = true;
    const int a = k + 2;
    if (a <= a1) {
      const int s = a & 1;
      ok = bar_wait(bar0 + 8 * s, (uint32_t)((a - a0) >> 1) & 1u, g_fd3p_wait_ns);
      float4 uc[V];
#pragma unroll
      for (int q = 0; q < V; ++q) uc[q] = get(&su[s][warp][0], q);
      float pl[V], pr[V], ul[V], ur[V];
      xnbr_row<V>(P1, pl, pr);
      xnbr_row<V>(uc, ul, ur);
      float4 h[V];
#pragma unroll
      for (int q = 0; q < V; ++q) {
        const float4 vc = get(&sv[s][warp + 1][0], q), vym = get(&sv[s][warp][0], q),
                     vyp = get(&sv[s][warp + 2][0], q);
        h[q] = adv_quad<FLUX>(P1[q], pl[q], pr[q], Pym[q], Pyp[q], P0[q], P2[q], uc[q], ul[q], ur[q], vym, vc, vyp,
                              W0[q], W1[q], W2[q], p.dt);
      }
      put(sh, a & 3, h);
      // march: phi of plane a - 1 becomes the cube of the next phase B
#pragma unroll
      for (int q = 0; q < V; ++q) {
        Pk[q] = P0[q];
        P0[q] = P1[q];
        P1[q] = P2[q];
        W0[q] = W1[q];
        W1[q] = W2[q];
      }
      if (a + 1 <= a1) {
        ldrow(G, y, a + 2, P2);
        ldrow(G, ym, a + 1, Pym);
        ldrow(G, yp, a + 1, Pyp);
        ldrow(ww, y, a + 2, W2);
      }
    } else {
      // no plane left to advect: phi of plane k + 1 for the last phase B
#pragma unroll
      for (int q = 0; q < V; ++q) {
        Pk[q] = P0[q];
        P0[q] = P1[q];
      }
    }
    if (!__syncthreads_and(ok)) {
      // a copy did not land within the bound: report, drain what is in
      // flight (planes a and a + 1, with the 0.5 s bound), leave
      if (threadIdx.x == 0) {
        atomicExch(&g_fd3p_err, 1);
        for (int pl = a; pl <= min(a + 1, a1); ++pl)
          bar_wait(bar0 + 8 * (pl & 1), (uint32_t)((pl - a0) >> 1) & 1u, 500000000ull);
      }
      return;
    }
  }
}

// resident CTAs of the pipelined substep kernel on this device (queried once per V)
template <int V>
int fd3p_resident_v() {
  static const int g = [] {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fd3p_kernel<false, V>, F3P_NW * 32, F3P<V>::smem);
    return std::max(1, sms * std::max(per, 1));
  }();
  return g;
}

template <typename S, typename C>
__global__ void __launch_bounds__(256)
    density3d_kernel(const S *__restrict__ hin, C *__restrict__ dn, KParams<C> p) {
  const int Lx = p.Lx, Ly = p.Ly, Lz = p.Lz;
  const long long Sz = (long long)Lx * Ly * Lz;
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y, z = blockIdx.z;
  if (x >= Lx || y >= Ly) return;
  C d = C(0);
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const int sx = wrapi(x - q19_ex(i), Lx), sy = wrapi(y - q19_ey(i), Ly),
              sz = wrapi(z - q19_ez(i), Lz);
    d += Store<S, C>::ld(hin + i * Sz + ((long long)sz * Ly + sy) * Lx + sx, p.inv_scale);
  }
  dn[((long long)z * Ly + y) * Lx + x] = d;
}

template <typename S, typename C>
cudaError_t collide3d(lbm_handle *h, int in, int force_on, int mode) {
  KParams<C> p = make_params<C>(h, force_on);
  dim3 grid((p.Lx + C3_TX - 1) / C3_TX, (p.Ly + C3_TY - 1) / C3_TY, (p.Lz + C3_TZ - 1) / C3_TZ);
  dim3 block(32, C3_TY);
  const S *hin = static_cast<const S *>(h->h[in]);
  S *hout = static_cast<S *>(h->h[1 - in]);
  const C *phi = static_cast<const C *>(h->phi[in]);
  const C *dn = static_cast<const C *>(h->dn);
  C *u = static_cast<C *>(h->u);
  const bool tgen = p.cs2mT != C(0);
  // registers budgeted for 3 CTAs per SM (85 a thread, no spill in FP32): 576 us
  // at 256^3 against 698 us for 2 and 618 us for 4 (spilling)
  if (mode == COLLIDE_STEP) {
    if (tgen)
      collide3d_kernel<S, C, true, COLLIDE_STEP, 3><<<grid, block, 0, h->stream>>>(hin, hout, phi, dn, u, h->staging, p);
    else
      collide3d_kernel<S, C, false, COLLIDE_STEP, 3><<<grid, block, 0, h->stream>>>(hin, hout, phi, dn, u, h->staging, p);
  } else {
    if (tgen)
      collide3d_kernel<S, C, true, COLLIDE_MOMENTS, 3><<<grid, block, 0, h->stream>>>(hin, hout, phi, dn, u, h->staging, p);
    else
      collide3d_kernel<S, C, false, COLLIDE_MOMENTS, 3><<<grid, block, 0, h->stream>>>(hin, hout, phi, dn, u, h->staging, p);
  }
  return cudaGetLastError();
}

// resident blocks of a kernel on this device
template <typename K>
int resident_blocks(K kernel, int threads, size_t smem) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
  return std::max(1, sms * std::max(per, 1));
}

// log2 of the lanes that a row of nq quads takes in the advection pass: 32, or
// 16 or 8 where that leaves clearly fewer lanes idle (short rows share a warp;
// every 2^lw lanes the outermost ones load their x neighbours)
int adv_lanes_log2(int nq) {
  int best = 5;
  double cost = 0;
  for (int lw = 5; lw >= 3; --lw) {
    const int L = 1 << lw, used = (nq + L - 1) / L * L;
    const double c = used * (nq <= L ? 1.0 : 1.0 + 0.05 * (5 - lw));
    if (lw == 5 || c < 0.9 * cost) {
      best = lw;
      cost = c;
    }
  }
  return best;
}

// the m substeps of an LB step as three passes each (FP32)
cudaError_t fd3d_passes(lbm_handle *h, int in) {
  KParams<float> p = make_params<float>(h, 0);
  dim3 grid((p.Lx + 31) / 32, (p.Ly + 7) / 8, p.Lz), block(32, 8);
  const float *u = static_cast<const float *>(h->u);
  float *A = static_cast<float *>(h->fd_a), *P = static_cast<float *>(h->fd_p);
  const float *src = static_cast<const float *>(h->phi[in]);
  const bool flux = p.adv_variant == LBM_ADV_FLUX;
  const bool vec = p.Lx % 4 == 0 && p.Lx >= 4 && std::getenv("HLBM_FD3_SCALAR") == nullptr;
  const int nq = p.Lx / 4, alw = adv_lanes_log2(std::max(nq, 1)), aL = 1 << alw;
  // planes per thread (at most F3V_NZ): the kernels run a few waves of
  // resident blocks, and a partial last wave leaves most SMs idle while its
  // blocks march their planes, so nz minimises waves x (nz + 2), the planes a
  // block loads (its first two are the z neighbours of the first output)
  auto planes_per_block = [&](long long bxy, long long res) {
    int nz = 1;
    long long best = -1;
    for (int c = 1; c <= std::min(F3V_NZ, p.Lz); ++c) {
      const long long waves = (bxy * ((p.Lz + c - 1) / c) + res - 1) / res;
      if (best < 0 || waves * (c + 2) < best) {
        best = waves * (c + 2);
        nz = c;
      }
    }
    return nz;
  };
  static const int res_adv = resident_blocks(fd3v_adv_kernel<false, false>, 256, 0);
  static const int res_flux = resident_blocks(fd3v_adv_kernel<true, false>, 256, 0);
  const bool wrap = nq <= aL;
  const int abx = (nq + aL - 1) / aL, aby = (p.Ly + (256 >> alw) - 1) / (256 >> alw);
  const int nz = planes_per_block((long long)abx * aby, flux ? res_flux : res_adv);
  dim3 grida(abx, aby, (p.Lz + nz - 1) / nz);
  auto advect = [&](const float *from) {
    if (flux && wrap) fd3v_adv_kernel<true, true><<<grida, 256, 0, h->stream>>>(from, u, A, p, nz, alw);
    else if (flux) fd3v_adv_kernel<true, false><<<grida, 256, 0, h->stream>>>(from, u, A, p, nz, alw);
    else if (wrap) fd3v_adv_kernel<false, true><<<grida, 256, 0, h->stream>>>(from, u, A, p, nz, alw);
    else fd3v_adv_kernel<false, false><<<grida, 256, 0, h->stream>>>(from, u, A, p, nz, alw);
  };
  const int nzl = planes_per_block((long long)((nq + 31) / 32) * ((p.Ly + 7) / 8), res_adv);
  dim3 gridl((nq + 31) / 32, (p.Ly + 7) / 8, (p.Lz + nzl - 1) / nzl);
  // psi and the new phi fused (whole rows, Lx <= 256): one wave of CTAs, as
  // many chunks of planes as fit beside each other
  const bool fused = vec && p.Lx <= 256 && std::getenv("HLBM_FD3_UNFUSED") == nullptr;
  const int V = nq <= 32 ? 1 : 2;
  const int flw = nq <= 8 ? 3 : (nq <= 16 ? 4 : 5), fR = (F3F_NW * 32) >> flw;
  const size_t smf = sizeof(float4) * 4 * V * F3F_NW * 32;
  static const int res_f1 = resident_blocks(fd3f_kernel<1, 2, true>, F3F_NW * 32, sizeof(float4) * 4 * F3F_NW * 32);
  static const int res_f2 = resident_blocks(fd3f_kernel<2, 1, true>, F3F_NW * 32, sizeof(float4) * 8 * F3F_NW * 32);
  const int rows_f = (p.Ly + fR - 3) / (fR - 2);
  const int chunks = std::max(1, std::min(p.Lz, (V == 1 ? res_f1 : res_f2) / rows_f));
  const int nzf = (p.Lz + chunks - 1) / chunks;
  dim3 gridf(1, rows_f, (p.Lz + nzf - 1) / nzf);
  // the advection fused as well, one software-pipelined kernel per substep
  // (opt-in; one CTA per SM, within one wave of z chunks)
  const bool fusedp = fused && (p.Lx == 128 || p.Lx == 256) && std::getenv("HLBM_FD3_FUSED_ADV") != nullptr;
  const int rows_p = (p.Ly + F3P_NW - 5) / (F3P_NW - 4);
  const int zch = std::max(1, std::min(p.Lz, (p.Lx == 128 ? fd3p_resident_v<1>() : fd3p_resident_v<2>()) / rows_p));
  const int nzp = (p.Lz + zch - 1) / zch;
  dim3 gridp(1, rows_p, (p.Lz + nzp - 1) / nzp);
  for (int j = 0; j < h->m; ++j) {
    float *dst = static_cast<float *>(((h->m - 1 - j) % 2 == 0) ? h->phi[1 - in] : h->phi[2]);
    if (fusedp) {
      if (p.Lx == 128) {
        if (flux) fd3p_kernel<true, 1><<<gridp, F3P_NW * 32, F3P<1>::smem, h->stream>>>(src, u, dst, p, nzp);
        else fd3p_kernel<false, 1><<<gridp, F3P_NW * 32, F3P<1>::smem, h->stream>>>(src, u, dst, p, nzp);
      } else {
        if (flux) fd3p_kernel<true, 2><<<gridp, F3P_NW * 32, F3P<2>::smem, h->stream>>>(src, u, dst, p, nzp);
        else fd3p_kernel<false, 2><<<gridp, F3P_NW * 32, F3P<2>::smem, h->stream>>>(src, u, dst, p, nzp);
      }
    } else if (vec) {
      advect(src);
      if (fused) {
        auto psi_phi = [&](auto kernel) { kernel<<<gridf, F3F_NW * 32, smf, h->stream>>>(A, src, dst, p, nzf, flw); };
        if (p.Lx == 128) psi_phi(fd3f_kernel<1, 2, false>);
        else if (p.Lx == 256) psi_phi(fd3f_kernel<2, 1, false>);
        else if (V == 1) psi_phi(fd3f_kernel<1, 2, true>);
        else psi_phi(fd3f_kernel<2, 1, true>);
      } else {
        fd3v_lap_kernel<true><<<gridl, block, 0, h->stream>>>(A, src, P, p, nzl);
        fd3v_lap_kernel<false><<<gridl, block, 0, h->stream>>>(P, A, dst, p, nzl);
      }
    } else {
      if (flux) fd3_adv_kernel<true><<<grid, block, 0, h->stream>>>(src, u, A, p);
      else fd3_adv_kernel<false><<<grid, block, 0, h->stream>>>(src, u, A, p);
      fd3_psi_kernel<<<grid, block, 0, h->stream>>>(A, src, P, p);
      fd3_phi_kernel<<<grid, block, 0, h->stream>>>(P, A, dst, p);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    src = dst;
  }
  return cudaSuccess;
}

template <typename C, int TX, int TY, int TZ>
cudaError_t fd3d(lbm_handle *h, int in) {
  KParams<C> p = make_params<C>(h, 0);
  dim3 grid((p.Lx + TX - 1) / TX, (p.Ly + TY - 1) / TY, (p.Lz + TZ - 1) / TZ), block(32, 8);
  const int launches = (h->m + h->sub - 1) / h->sub;
  const C *u = static_cast<const C *>(h->u);
  const C *src = static_cast<const C *>(h->phi[in]);
  for (int j = 0; j < launches; ++j) {
    const int sub = (j == launches - 1) ? h->m - h->sub * (launches - 1) : h->sub;
    C *dst = static_cast<C *>(((launches - 1 - j) % 2 == 0) ? h->phi[1 - in] : h->phi[2]);
    const int H = 3 * sub;
    const size_t smem = sizeof(C) * 6 * (size_t)(TX + 2 * H) * (TY + 2 * H) * (TZ + 2 * H);
    fd3d_kernel<C, TX, TY, TZ><<<grid, block, smem, h->stream>>>(src, u, dst, p, sub);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    src = dst;
  }
  return cudaSuccess;
}

}  // namespace

// FD tile (HLBM_FD3_TILE=1): FP32 32 x 4 x 4 (one substep per launch: halo 3).
constexpr int FD3_TX_F = 32, FD3_TY = 4, FD3_TZ = 4;

size_t fd3d_smem_bytes(int sub) {
  const int H = 3 * sub;
  return sizeof(float) * 6 * (size_t)(FD3_TX_F + 2 * H) * (FD3_TY + 2 * H) * (FD3_TZ + 2 * H);
}

// FP32 storage and arithmetic; the FP64 kernels use no shared memory
cudaError_t fd3d_configure(int precision, size_t smem) {
  if (precision == LBM_F64) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(fd3d_kernel<float, FD3_TX_F, FD3_TY, FD3_TZ>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int smf1 = (int)(sizeof(float) * 4 * F3F_NW * 128), smf2 = 2 * smf1;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fd3f_kernel<1, 2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smf1);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fd3f_kernel<1, 2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smf1);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fd3f_kernel<2, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smf2);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fd3f_kernel<2, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smf2);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fd3p_kernel<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F3P<1>::smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fd3p_kernel<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F3P<1>::smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fd3p_kernel<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F3P<2>::smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fd3p_kernel<true, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F3P<2>::smem);
  return e;
}

int fd3p_set_wait_ns(unsigned long long ns) {
  return cudaMemcpyToSymbol(g_fd3p_wait_ns, &ns, sizeof ns) == cudaSuccess ? 0 : -1;
}

int fd3p_error(bool reset) {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_fd3p_err, sizeof v) != cudaSuccess) return -1;
  if (reset && v != 0) {
    const int zero = 0;
    cudaMemcpyToSymbol(g_fd3p_err, &zero, sizeof zero);
  }
  return v;
}

cudaError_t collide3d_launch(lbm_handle *h, int in, int force_on, int mode) {
  switch (h->P.precision) {
    case LBM_F64: return collide3_f64(h, in, force_on, mode);
    case LBM_F32DEV: return collide3d<float, float>(h, in, force_on, mode);
    default: return collide3d<__half, float>(h, in, force_on, mode);
  }
}

cudaError_t fd3d_launch(lbm_handle *h, int in) {
  if (h->P.precision == LBM_F64) return fd3_f64(h, in);
  if (h->fd_a != nullptr && std::getenv("HLBM_FD3_TILE") == nullptr) return fd3d_passes(h, in);
  return fd3d<float, FD3_TX_F, FD3_TY, FD3_TZ>(h, in);
}

cudaError_t density3d_launch(lbm_handle *h, int in) {
  dim3 grid((h->P.Lx + 31) / 32, (h->P.Ly + 7) / 8, h->P.Lz), block(32, 8);
  switch (h->P.precision) {
    case LBM_F64: {
      KParams<double> p = make_params<double>(h, 0);
      density3d_kernel<double, double><<<grid, block, 0, h->stream>>>(
          static_cast<const double *>(h->h[in]), static_cast<double *>(h->dn), p);
      break;
    }
    case LBM_F32DEV: {
      KParams<float> p = make_params<float>(h, 0);
      density3d_kernel<float, float><<<grid, block, 0, h->stream>>>(
          static_cast<const float *>(h->h[in]), static_cast<float *>(h->dn), p);
      break;
    }
    default: {
      KParams<float> p = make_params<float>(h, 0);
      density3d_kernel<__half, float><<<grid, block, 0, h->stream>>>(
          static_cast<const __half *>(h->h[in]), static_cast<float *>(h->dn), p);
    }
  }
  return cudaGetLastError();
}

}  // namespace hlbm
