// The near-image sum (A_else, Sec. 4.1) by spherical-wave expansions, for
// lattices whose nearest image stays clear of the body.
//
// With all sources y_s within r_s of the centre (0, 0, z_c) and all targets
// within r_t, an image displaced by D > r_s + r_t acts on the targets through
//   sum_s sigma_s G(x, c + y_s) = sum_{l,m} M_lm h_l(k|x - c|) Y_lm,
//   M_lm = i k sum_j j_l(k r_j) Pbar_l^m(cos theta_j) c_{m mod P, j}
// (the azimuthal sum of a ring's P points against e^{-i m phi} is the ring's
// coefficient of mode m mod P, so the P-point sum is reproduced with its
// aliases), and near the centre through regular waves L_lm j_l(k r) Y_lm.
// Degrees l <= p reach FP64 rounding (near_sph_degree); p is 72 for the k = 25
// cup. The direct sum costs M P N P kernel values per image, in FP64 on a
// part with 1/64-rate FP64; this one costs O(p^2 (N + M) + p^3) per wave, all
// of it small real-by-complex matrix products.
//
// Bound by the FP64 pipe (about 2.3e8 FMA for the cup with 16 waves: 0.38 ms
// at 1.2 TFLOP/s) and by the serial chains of length p. Cup, lattice of 13
// wavelengths, 7 digits asked for: 1.46 s by the direct split sum, 1.2 ms here
// with 16 waves (0.44 ms with one); its error against 64-bit sums over all
// pairs falls from 3.1e-14 to 1.3e-14.
//
// Steps (w = wave, images in pairs +-c of the four displacements):
//   1 sph_setup   S_m[l][j] = j_l Pbar_l^m at the sources, B_m[l][i] = its
//                 normal derivative at the targets, the rotation matrices
//                 Delta^l = d^l(pi/2), the sectorial translation coefficients
//   2 sph_p2m     M_lm, and (other CTAs) the translation coefficients T^m
//   3 sph_rot_fwd M' = the multipoles about axes turned so that z' points
//                 along the displacement: e^{i m phi_c}, then d^l(-pi/2)
//   4 sph_axial   L'_lm = sum_l' T^m_{l l'}(kD) M'_l'm
//   5 sph_rot_bwd L_lm = sum_c ph_w(c) e^{-i m phi_c} sum_m' d^l_{m'm} L'_lm'
//   6 sph_l2p     modal data at the rings, mode m folded to m mod P
//   7 sph_dft     samples at the P nodes of a ring
//
// Rotation: with Delta_{m',m} for m', m >= 0 only,
//   Delta_{m',-m} = (-1)^{l+m'} Delta_{m',m},  Delta_{-m',m} = (-1)^{l+m} Delta_{m',m},
// so the sums over even and odd m of (x_m +- x_-m) give rows +-m' at once; an
// image at -c has (-1)^m x_m, i.e. the same two sums subtracted. One quarter
// matrix times four pairs' columns replaces eight full matrices.
// Translation along z' commutes with d/dz and d/dx + i d/dy, which gives the
// recurrences (a_n = sqrt(((n+1)^2 - m^2)/((2n+1)(2n+3))))
//   a_n T_{l,n+1} = a_{n-1} T_{l,n-1} - a_l T_{l+1,n} + a_{l-1} T_{l-1,n}
// (Gumerov and Duraiswami, "Recursions for the computation of multipole
// translation and rotation coefficients for the 3-D Helmholtz equation", SIAM
// J. Sci. Comput. 25 (2003)), started from Gegenbauer's addition theorem for
// h_m(kR)/(kR)^m (the distance from the axis is the same in both frames):
//   T^m_{l,m} = sqrt((2m+1)!!/(2m)!! (2l+1) (l+m)!/(l-m)!) h_l(kD) / (kD)^m.
// Run upwards in n the recurrence loses digits at large k r where p nears kD
// (orders m of 4 to 16): against quadruple precision the error of one source's
// field, relative to the largest kernel value, over periods of 1.3 to 60 times
// r_s + r_t is below 2e-14 for k r = 20, 3e-14 for 35, 5e-14 for 45, 3e-13 for 55 and
// 1e-12 for 60 (k r is that of the larger radius). Measured, single sources at 1.3
// (r_s + r_t), against the direct sum of 7 digits: 6e-15 and 7e-15 for k r = 20, 1.7e-14
// and 1.0e-14 for 33, 2.0e-14 and 1.6e-14 for 45, 1.6e-13 and 1.7e-14 for 57; 6 digits
// keep 5e-13. So a caller who asks for 7 digits (2^-44 = 6e-14) takes this path up to
// k r = 45, with fewer up to 55 (near_sph_degree). T depends on |m|, and
// M'_{-m}(-c) = (-1)^l M'_m(c), so the sums over even and odd l' give (m, c)
// and (-m, -c) together.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "axi_internal.h"
#include "fft.cuh"

namespace axi {
namespace {

constexpr int kSphMaxDegree = 127;
constexpr double kPi = 3.14159265358979323846;

// Waves of order m start at packed index sph_off(m): degrees l = m .. p.
__host__ __device__ inline int sph_off(int m, int p) { return m * (p + 1) - m * (m - 1) / 2; }
// Delta^l is (l + 1) x (l + 1) at delta_off(l); T^m is (p + 1 - m)^2 at t_off(m).
__host__ __device__ inline int delta_off(int l) { return l * (l + 1) * (2 * l + 1) / 6; }
__host__ __device__ inline int t_off(int m, int p) {
  const int a = p + 1, b = p + 1 - m;             // sum of squares b+1 .. a
  return (a * (a + 1) * (2 * a + 1) - b * (b + 1) * (2 * b + 1)) / 6;
}

// Geometry and sizes of one call, by value.
struct SphArgs {
  int p, W, M, N, P, cols, ncls;
  double k, zc;
  double dist[3];          // distances of the displacement classes
  int cls[4];              // class of pair q
  double phi[4];           // azimuth of the pair's displacement
  double cx[4], cy[4];     // the displacement
};

struct SphBuf {
  double *S, *B, *delta;
  double2 *hank;           // [ncls][2p + 1] h_l(kD)
  double2 *turn, *bloch;   // [4][p + 1] e^{i m phi_q}, [4][W] e^{i k d_w . c_q}
  double2 *T, *mult, *rot, *loc_rot, *loc, *modes;
};

// prod_{i <= m} (2i + 1) / (2i) over a warp: the divisions in parallel (a
// division is some twenty FP64 instructions, each 64 cycles a warp).
__device__ __forceinline__ double warp_odd_even_product(int m) {
  double v = 1.0;
  for (int i = 1 + (threadIdx.x & 31); i <= m; i += 32) v *= (2.0 * i + 1.0) / (2.0 * i);
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) v *= __shfl_xor_sync(0xffffffffu, v, s);
  return v;
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// ---------------------------------------------------------------- step 1

constexpr int kTabWarps = 4;
constexpr int kSetupThreads = 32 * kTabWarps;

// Table of 32 points (lanes) and the orders m, p - m of each warp: value
// j_l(kr) Pbar_l^m or its normal derivative, out[(sph_off(m) + l - m) n + i].
// Miller's backward recurrence for j_l (as btilde_kernel), three-term
// recurrences for Pbar; the FP64 pipe bounds it (about 8 operations an entry).
// dPbar_l^m/dtheta is (l cos Pbar_l - c Pbar_{l-1}) / sin for m > 0, where both
// terms fall with sin^m; for m = 0 it would subtract nearly equal terms near the
// axis, so there -sin Pbar_l' with P_l' = P_{l-2}' + (2l - 1) P_{l-1}, a sum of
// like signs near the axis.
template <bool DERIV>
__device__ void wave_table(const double *__restrict__ pts, int stride, int n, double k, double zc, int p,
                           int grp, int part, double *__restrict__ out, double *sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int jn = p + 2;
  double *jl = sh;                                          // [jn][32]
  double *cf = sh + jn * 32 + warp * 6 * (p + 1);           // [2][3][p + 1]
  const int i = grp * 32 + lane;
  const bool live = i < n;
  const double *pt = pts + (size_t)(live ? i : n - 1) * stride;
  const double rho = pt[0], z = pt[1] - zc;
  const double r = hypot(rho, z), x = k * r, ix = 1.0 / x;
  const double st = rho / r, ct = z / r;
  if (warp == 0) {
    double xmax = x;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) xmax = fmax(xmax, __shfl_xor_sync(0xffffffffu, xmax, s));
    const int L0 = p + (int)xmax + 40;
    double f1 = 0.0, f0 = 1.0;
    double c = 2.0 * L0 + 1.0;                              // 2l + 1, exact
    for (int l = L0; l >= 1; --l) {
      const double fm = fma(c * ix, f0, -f1);
      c -= 2.0;
      f1 = f0;
      f0 = fm;
      if (l - 1 < jn) jl[(l - 1) * 32 + lane] = fm;
      if (((unsigned long long)__double_as_longlong(fm) & 0x7ff0000000000000ull) > 0x6970000000000000ull) {
        const double s = 0x1p-664;
        f0 *= s;
        f1 *= s;
        for (int u = l - 1; u < jn; ++u) jl[u * 32 + lane] *= s;
      }
    }
    double sn, cs;
    sincos(x, &sn, &cs);
    const double j0 = sn * ix, j1 = (sn * ix - cs) * ix;
    const double sc = fabs(j0) >= fabs(j1) ? j0 / jl[lane] : j1 / jl[32 + lane];
    for (int u = 0; u < jn; ++u) jl[u * 32 + lane] *= sc;
  }
  const int m0 = part * kTabWarps + warp, m1 = p - m0;
  const bool has0 = m0 <= m1, has1 = m0 < m1;
  for (int t = 0; t < 2; ++t) {
    if (!(t == 0 ? has0 : has1)) continue;
    const int m = t == 0 ? m0 : m1;
    double *c = cf + t * 3 * (p + 1);
    for (int l = m + lane; l <= p; l += 32) {
      double a = 0.0, b = 0.0, cc = 0.0;
      const double ll = (double)l * l, mm = (double)m * m, l1 = (double)(l - 1) * (l - 1);
      if (l == m + 1) {
        a = sqrt(2.0 * m + 3.0);
      } else if (l > m + 1) {
        a = sqrt((4.0 * ll - 1.0) / (ll - mm));
        b = sqrt((l1 - mm) / (4.0 * l1 - 1.0));
      }
      if (DERIV && l > m)
        cc = m > 0 ? sqrt((2.0 * l + 1.0) * (l - m) * (l + m) / (2.0 * l - 1.0))
                   : l > 2 ? sqrt((2.0 * l + 1.0) / (2.0 * l - 3.0)) : 0.0;      // of Pbar_{l-2}'
      c[l] = a;
      c[(p + 1) + l] = b;
      c[2 * (p + 1) + l] = cc;
    }
  }
  __syncthreads();
  double Ak = 0.0, Bk = 0.0, ist = 0.0;
  if (DERIV) {
    const double nr = pt[2], nz = pt[3];
    Ak = k * (nr * st + nz * ct);
    Bk = (nr * ct - nz * st) / r;
    ist = 1.0 / st;
  }
  for (int t = 0; t < 2; ++t) {
    if (!(t == 0 ? has0 : has1)) continue;
    const int m = t == 0 ? m0 : m1;
    const double *ca = cf + t * 3 * (p + 1), *cb = ca + (p + 1), *cc = ca + 2 * (p + 1);
    const double prod = warp_odd_even_product(m) / (4.0 * kPi);
    double spow = 1.0, sq = st;                             // sin(theta)^m by squaring
    for (int u = m; u > 0; u >>= 1) {
      if (u & 1) spow *= sq;
      sq *= sq;
    }
    double cur = ((m & 1) ? -sqrt(prod) : sqrt(prod)) * spow, prev = 0.0, dl = m;   // dl = l
    double *blk = out + (size_t)sph_off(m, p) * n;
    auto column = [&](auto zonal) {                         // two loops: no instruction of the other form
      double q0 = 0.0, q1 = 0.0;                            // m = 0: Pbar_l', Pbar_{l-1}'
      for (int l = m; l <= p; ++l) {
        if (l > m) {
          const double nxt = ca[l] * fma(ct, cur, -cb[l] * prev);
          prev = cur;
          cur = nxt;
          dl += 1.0;
          if constexpr (DERIV && zonal.value) {
            const double q2 = fma(dl * ca[l], prev, cc[l] * q1);
            q1 = q0;
            q0 = q2;
          }
        }
        const double j = jl[l * 32 + lane];
        double v;
        if constexpr (DERIV) {
          double dP;
          if constexpr (zonal.value)
            dP = -st * q0;
          else
            dP = fma(dl * ct, cur, -cc[l] * prev) * ist;
          const double dj = l == 0 ? -jl[32 + lane] : fma(-(dl + 1.0) * ix, j, jl[(l - 1) * 32 + lane]);
          v = fma(Ak * dj, cur, Bk * j * dP);
        } else {
          v = j * cur;
        }
        if (live) blk[(size_t)(l - m) * n + i] = v;
      }
    };
    if (DERIV && m == 0)
      column(std::true_type{});
    else
      column(std::false_type{});
  }
}

// Delta^l_{m',m}, 0 <= m', m <= l: d_{l,m} = (-1)^{l-m} sqrt(C(2l, l+m)) / 2^l,
// then downwards in m' (one thread per m), the stable direction:
//   d_{m'} = (2m d_{m'+1} - sqrt((l-m'-1)(l+m'+2)) d_{m'+2}) / sqrt((l-m')(l+m'+1)).
__device__ void delta_matrix(int l, double *__restrict__ out, double *sh) {
  double *inv = sh;                                         // [2l + 1] 1 / i
  double *c1 = inv + 2 * l + 1, *c2 = c1 + l + 1;           // [l + 1] each
  for (int i = threadIdx.x; i <= 2 * l; i += kSetupThreads) inv[i] = i ? 1.0 / i : 0.0;
  for (int i = threadIdx.x; i <= l; i += kSetupThreads) {
    const double q = i < l ? 1.0 / sqrt((double)(l - i) * (l + i + 1)) : 0.0;
    c1[i] = q;
    c2[i] = i + 1 < l ? sqrt((double)(l - i - 1) * (l + i + 2)) * q : 0.0;
  }
  __syncthreads();
  const int m = threadIdx.x;
  if (m > l) return;
  double v = 1.0;                                           // C(2l, l + m) / 4^l
  for (int i = 1; i <= l; ++i) v *= 1.0 - 0.5 * inv[i];     // (2i - 1) / (2i)
  for (int i = 1; i <= m; ++i) v *= (l - i + 1) * inv[l + i];
  double d1 = ((l - m) & 1) ? -sqrt(v) : sqrt(v), d2 = 0.0;
  double *o = out + delta_off(l) + m;
  o[(size_t)l * (l + 1)] = d1;
  for (int mp = l - 1; mp >= 0; --mp) {
    const double d0 = fma(2.0 * m * c1[mp], d1, -c2[mp] * d2);
    o[(size_t)mp * (l + 1)] = d0;
    d2 = d1;
    d1 = d0;
  }
}

// h_l(x), l = 0 .. 2p, of one distance, one thread each: y_l upwards; j_l upwards
// too where x is beyond the last degree (stable for l < x), else by Miller's
// recurrence from 40 degrees past the last one and the turning zone (a few
// x^{1/3} wide). At most 370 steps either way, whatever the period.
__device__ void hankel_row(double x, int p, double2 *__restrict__ out, double *sh) {
  const int L = 2 * p + 1;
  double *c = sh, *yl = c + L + 1, *jl = yl + L;            // c: (2l + 1) / x
  const double ix = 1.0 / x;
  double sn, cs;
  sincos(x, &sn, &cs);
  for (int i = threadIdx.x; i <= L; i += kSetupThreads) c[i] = (2.0 * i + 1.0) * ix;
  __syncthreads();
  if (threadIdx.x == 0) {
    double y0 = -cs * ix, y1 = (y0 - sn) * ix;
    for (int l = 0; l < L; ++l) {
      yl[l] = y0;
      const double y2 = fma(c[l + 1], y1, -y0);
      y0 = y1;
      y1 = y2;
    }
  } else if (threadIdx.x == 32 && x > L) {
    double j0 = sn * ix, j1 = (j0 - cs) * ix;
    for (int l = 0; l < L; ++l) {
      jl[l] = j0;
      const double j2 = fma(c[l + 1], j1, -j0);
      j0 = j1;
      j1 = j2;
    }
  } else if (threadIdx.x == 32) {
    const int L0 = max(L, (int)(x + 12.0 * cbrt(x))) + 40;
    double f1 = 0.0, f0 = 1.0;
    for (int l = L0; l >= 1; --l) {
      const double fm = fma(l <= L ? c[l] : (2.0 * l + 1.0) * ix, f0, -f1);
      f1 = f0;
      f0 = fm;
      if (l - 1 < L) jl[l - 1] = fm;
      if (((unsigned long long)__double_as_longlong(fm) & 0x7ff0000000000000ull) > 0x6970000000000000ull) {
        f0 *= 0x1p-664;
        f1 *= 0x1p-664;
        for (int u = l - 1; u < L; ++u) jl[u] *= 0x1p-664;
      }
    }
  }
  __syncthreads();
  const double j0 = sn * ix, j1 = (sn * ix - cs) * ix;
  const double sc = fabs(j0) >= fabs(j1) ? j0 / jl[0] : j1 / jl[1];
  for (int l = threadIdx.x; l < L; l += kSetupThreads) out[l] = make_double2(jl[l] * sc, yl[l]);
}

// CTAs: h_l of each distance, the phases, the target tables, the source
// tables, Delta^l.
__global__ void __launch_bounds__(kSetupThreads)
sph_setup_kernel(const ObsDev *__restrict__ od, SphArgs g, SphBuf b, const double *__restrict__ dirs, int parts) {
  extern __shared__ double sh[];
  const ObsDev &o = *od;
  int c = blockIdx.x;
  if (c < g.ncls) {
    hankel_row(g.k * g.dist[c], g.p, b.hank + (size_t)c * (2 * g.p + 1), sh);
    return;
  }
  c -= g.ncls;
  if (c < 4) {                                              // pair c's phases
    for (int e = threadIdx.x; e < g.p + 1 + g.W; e += kSetupThreads) {
      const int w = e - g.p - 1;
      double sn, cs;
      sincos(w < 0 ? e * g.phi[c] : g.k * (dirs[3 * w] * g.cx[c] + dirs[3 * w + 1] * g.cy[c]), &sn, &cs);
      (w < 0 ? b.turn[c * (g.p + 1) + e] : b.bloch[c * g.W + w]) = make_double2(cs, sn);
    }
    return;
  }
  c -= 4;
  const int nt = (g.M + 31) / 32 * parts, ns = (g.N + 31) / 32 * parts;
  if (c < nt) {
    wave_table<true>(o.coll, 4, g.M, g.k, g.zc, g.p, c / parts, c % parts, b.B, sh);
    return;
  }
  c -= nt;
  if (c < ns) {
    wave_table<false>(o.src, 2, g.N, g.k, g.zc, g.p, c / parts, c % parts, b.S, sh);
    return;
  }
  delta_matrix(g.p - (c - ns), b.delta, sh);
}

// ---------------------------------------------------------------- step 2

constexpr int kMatThreads = 128;

// T^m_{l,n} of one class, n = m .. p (stored [n - m][l - m]): rows of length
// 2p + 1 - n - m shrink by one per step.
__device__ void translation_block(int m, int p, double x, const double2 *__restrict__ h, double2 *__restrict__ out,
                                  double *sh) {
  const int L = 2 * p + 1, w = p + 1 - m;
  double *a = sh, *sq = sh + L;                             // [L] a_l, [2L + 1] sqrt(i / x)
  double2 *e0 = reinterpret_cast<double2 *>(sh + 3 * L + 1), *e1 = e0 + L, *e2 = e1 + L;
  const double ix = 1.0 / x;
  for (int i = threadIdx.x; i <= 2 * L; i += kMatThreads) sq[i] = sqrt(i * ix);
  const double f = sqrt(warp_odd_even_product(m));          // (2m + 1)!! / (2m)!!
  __syncthreads();
  for (int l = threadIdx.x; l < L; l += kMatThreads) {
    a[l] = l >= m ? sqrt((double)(l + 1 - m) * (l + 1 + m) / ((2.0 * l + 1.0) * (2.0 * l + 3.0))) : 0.0;
    e0[l] = make_double2(0.0, 0.0);
    double q = 0.0;
    if (l >= m && l <= 2 * p - m) {
      q = f * sqrt(2.0 * l + 1.0);
      for (int i = 1; i <= m; ++i) q *= sq[l - i + 1] * sq[l + i];
    }
    const double2 v = h[l];
    e1[l] = q != 0.0 ? make_double2(q * v.x, q * v.y) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int l = m + threadIdx.x; l <= p; l += kMatThreads) out[l - m] = e1[l];
  for (int n = m; n < p; ++n) {
    const double ia = 1.0 / a[n], an = n > m ? a[n - 1] : 0.0;
    double2 *o = out + (size_t)(n + 1 - m) * w;
    for (int l = m + threadIdx.x; l < 2 * p - n; l += kMatThreads) {
      const double2 hi = e1[l + 1], lo = l > m ? e1[l - 1] : make_double2(0.0, 0.0), pr = e0[l];
      const double al = a[l], am = l > m ? a[l - 1] : 0.0;
      const double2 v = make_double2(ia * fma(an, pr.x, fma(am, lo.x, -al * hi.x)),
                                     ia * fma(an, pr.y, fma(am, lo.y, -al * hi.y)));
      e2[l] = v;
      if (l <= p) o[l - m] = v;
    }
    __syncthreads();
    double2 *t = e0;
    e0 = e1;
    e1 = e2;
    e2 = t;
  }
}

// M_{l,+-m} of 32 degrees and TC waves: S and the coefficients staged 32 rings
// at a time, one degree per lane, the waves over the four warps.
template <int TC>
__device__ void p2m_tile(const SphArgs &g, const SphBuf &b, const double2 *__restrict__ coef, int m, int lt,
                         int wt, double *sh) {
  constexpr int NG = TC < 4 ? TC : 4, WG = TC / NG;        // warps in use, waves per warp
  double *ss = sh;                                          // [32 j][33]
  double2 *cs = reinterpret_cast<double2 *>(sh + 32 * 33);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int l0 = m + 32 * lt, nl = min(32, g.p + 1 - l0), w0 = wt * TC;
  const int np = m % g.P, nm = (g.P - np) % g.P;
  const double *S = b.S + (size_t)(sph_off(m, g.p) + 32 * lt) * g.N;
  double2 acc[2][WG];
#pragma unroll
  for (int q = 0; q < WG; ++q) acc[0][q] = acc[1][q] = make_double2(0.0, 0.0);
  for (int j0 = 0; j0 < g.N; j0 += 32) {
    const int nj = min(32, g.N - j0);
    __syncthreads();
    for (int r = warp; r < 32; r += kMatThreads / 32)
      ss[lane * 33 + r] = r < nl && lane < nj ? S[(size_t)r * g.N + j0 + lane] : 0.0;
    for (int e = warp; e < 2 * TC; e += kMatThreads / 32) {
      const int w = w0 + (e >> 1);
      cs[lane * 2 * TC + e] = w < g.W && lane < nj
                                  ? coef[((size_t)w * g.P + ((e & 1) ? nm : np)) * g.cols + j0 + lane]
                                  : make_double2(0.0, 0.0);
    }
    __syncthreads();
    if (warp < NG) {
#pragma unroll 4
      for (int j = 0; j < 32; ++j) {
        const double s = ss[j * 33 + lane];
#pragma unroll
        for (int q = 0; q < WG; ++q) {
          const double2 u = cs[j * 2 * TC + 2 * (warp * WG + q)], v = cs[j * 2 * TC + 2 * (warp * WG + q) + 1];
          acc[0][q].x = fma(s, u.x, acc[0][q].x);
          acc[0][q].y = fma(s, u.y, acc[0][q].y);
          acc[1][q].x = fma(s, v.x, acc[1][q].x);
          acc[1][q].y = fma(s, v.y, acc[1][q].y);
        }
      }
    }
  }
  if (warp >= NG || lane >= nl) return;
  const int l = l0 + lane;
  const double k = g.k, km = (m & 1) ? -k : k;
#pragma unroll
  for (int q = 0; q < WG; ++q) {
    const int w = w0 + warp * WG + q;
    if (w >= g.W) continue;
    b.mult[(size_t)(l * l + l + m) * g.W + w] = make_double2(-k * acc[0][q].y, k * acc[0][q].x);
    if (m > 0) b.mult[(size_t)(l * l + l - m) * g.W + w] = make_double2(-km * acc[1][q].y, km * acc[1][q].x);
  }
}

template <int TC>
__global__ void __launch_bounds__(kMatThreads)
sph_p2m_kernel(SphArgs g, SphBuf b, const double2 *__restrict__ coef) {
  extern __shared__ double sh[];
  const int p = g.p, m = blockIdx.x;
  const int ltiles = (p + 32) / 32, wtiles = (g.W + TC - 1) / TC;
  int c = blockIdx.y;
  if (c < g.ncls) {
    translation_block(m, p, g.k * g.dist[c], b.hank + (size_t)c * (2 * p + 1),
                      b.T + (size_t)c * t_off(p + 1, p) + t_off(m, p), sh);
    return;
  }
  c -= g.ncls;
  const int lt = c / wtiles, wt = c % wtiles;
  if (lt >= ltiles || m + 32 * lt > p) return;
  p2m_tile<TC>(g, b, coef, m, lt, wt, sh);
}

// ---------------------------------------------------------------- steps 3 - 5

// The three products run one row per kMatThreads / TC threads, TC waves
// across; a CTA takes one slab of that many rows, so the large degrees spread
// over several SMs (the FP64 pipe bounds each).

// Row sums over even and odd columns: e, o of d[0 .. n-1] times y[i TC + cc].
template <int TC>
__device__ __forceinline__ void parity_dot(const double *__restrict__ d, const double2 *y, int n, double2 &e,
                                           double2 &o) {
  int i = 0;
#pragma unroll 4
  for (; i + 1 < n; i += 2) {
    const double d0 = d[i], d1 = d[i + 1];
    const double2 a = y[i * TC], c = y[(i + 1) * TC];
    e.x = fma(d0, a.x, e.x);
    e.y = fma(d0, a.y, e.y);
    o.x = fma(d1, c.x, o.x);
    o.y = fma(d1, c.y, o.y);
  }
  if (i < n) {
    const double2 a = y[i * TC];
    e.x = fma(d[i], a.x, e.x);
    e.y = fma(d[i], a.y, e.y);
  }
}

// CTA: slab of rows m', degree l (largest first), pair q, TC waves.
// y[par][m] = (-1)^m (x_m +- x_-m), x_m = e^{i m phi} M_lm; both images of the pair.
template <int TC>
__global__ void __launch_bounds__(kMatThreads)
sph_rot_fwd_kernel(SphArgs g, SphBuf b, int wtiles) {
  extern __shared__ double2 shc[];
  constexpr int kRows = kMatThreads / TC;
  const int l = g.p - blockIdx.x, q = blockIdx.y, w0 = (blockIdx.z % wtiles) * TC, r0 = blockIdx.z / wtiles * kRows;
  if (r0 > l) return;
  double2 *yp = shc, *ym = shc + (l + 1) * TC;
  const double2 *M = b.mult + (size_t)l * l * g.W, *turn = b.turn + q * (g.p + 1);
  for (int e = threadIdx.x; e < (l + 1) * TC; e += kMatThreads) {
    const int m = e / TC, w = w0 + e % TC;
    double2 u = make_double2(0.0, 0.0), v = u;
    if (w < g.W) {
      const double2 t = turn[m];
      u = cmul(M[(size_t)(l + m) * g.W + w], t);
      if (m > 0) v = cmul(M[(size_t)(l - m) * g.W + w], make_double2(t.x, -t.y));
    }
    const double sg = (m & 1) ? -1.0 : 1.0;
    yp[e] = make_double2(sg * (u.x + v.x), sg * (u.y + v.y));
    ym[e] = make_double2(sg * (u.x - v.x), sg * (u.y - v.y));
  }
  __syncthreads();
  const int cc = threadIdx.x % TC, w = w0 + cc, mp = r0 + threadIdx.x / TC;
  if (mp > l || w >= g.W) return;
  double2 e = make_double2(0.0, 0.0), o = e;
  parity_dot<TC>(b.delta + delta_off(l) + (size_t)mp * (l + 1), (((l + mp) & 1) ? ym : yp) + cc, l + 1, e, o);
  const double s = (mp & 1) ? -1.0 : 1.0;
  double2 *r = b.rot + ((size_t)(sph_off(mp, g.p) + l - mp) * 8 + 2 * q) * g.W + w;
  r[0] = make_double2(s * (e.x + o.x), s * (e.y + o.y));
  r[g.W] = make_double2(s * (e.x - o.x), s * (e.y - o.y));
}

// CTA: slab of rows l, order m, image, TC waves: even and odd l' sums of
// T^m M' -> L'_m(c), L'_-m(-c).
template <int TC>
__global__ void __launch_bounds__(kMatThreads)
sph_axial_kernel(SphArgs g, SphBuf b, int wtiles) {
  extern __shared__ double2 shc[];
  constexpr int kRows = kMatThreads / TC;
  const int m = blockIdx.x, img = blockIdx.y, w0 = (blockIdx.z % wtiles) * TC, r0 = blockIdx.z / wtiles * kRows;
  const int n = g.p + 1 - m, nlt = sph_off(g.p + 1, g.p);
  if (r0 >= n) return;
  const double2 *R = b.rot + (size_t)sph_off(m, g.p) * 8 * g.W + (size_t)img * g.W;
  for (int e = threadIdx.x; e < n * TC; e += kMatThreads) {
    const int w = w0 + e % TC;
    shc[e] = w < g.W ? R[(size_t)(e / TC) * 8 * g.W + w] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const int cc = threadIdx.x % TC, w = w0 + cc, li = r0 + threadIdx.x / TC;
  if (li >= n || w >= g.W) return;
  const double2 *T = b.T + (size_t)g.cls[img >> 1] * t_off(g.p + 1, g.p) + t_off(m, g.p) + li;
  double2 e = make_double2(0.0, 0.0), o = e;
  int i = 0;
#pragma unroll 2
  for (; i + 1 < n; i += 2) {
    const double2 t0 = T[(size_t)i * n], t1 = T[(size_t)(i + 1) * n];
    const double2 a = shc[i * TC + cc], c = shc[(i + 1) * TC + cc];
    e.x = fma(t0.x, a.x, fma(-t0.y, a.y, e.x));
    e.y = fma(t0.x, a.y, fma(t0.y, a.x, e.y));
    o.x = fma(t1.x, c.x, fma(-t1.y, c.y, o.x));
    o.y = fma(t1.x, c.y, fma(t1.y, c.x, o.y));
  }
  if (i < n) {
    const double2 t0 = T[(size_t)i * n], a = shc[i * TC + cc];
    e.x = fma(t0.x, a.x, fma(-t0.y, a.y, e.x));
    e.y = fma(t0.x, a.y, fma(t0.y, a.x, e.y));
  }
  // index i counts l' - m: (-1)^{l'} = (-1)^m (-1)^i
  const double s = (m & 1) ? -1.0 : 1.0;
  const size_t at = (size_t)(sph_off(m, g.p) + li) * 8 * g.W + w;
  b.loc_rot[at + (size_t)img * g.W] = make_double2(e.x + o.x, e.y + o.y);
  b.loc_rot[(size_t)nlt * 8 * g.W + at + (size_t)(img ^ 1) * g.W] = make_double2(s * (e.x - o.x), s * (e.y - o.y));
}

// CTA: slab of rows m, degree l (largest first), TC waves; the four pairs'
// inputs in shared memory. Even rows m take ph(c) L'(c) + ph(-c) L'(-c), odd
// rows the difference.
template <int TC>
__global__ void __launch_bounds__(kMatThreads)
sph_rot_bwd_kernel(SphArgs g, SphBuf b) {
  extern __shared__ double2 shc[];
  constexpr int kRows = kMatThreads / TC;
  const int l = g.p - blockIdx.x, w0 = blockIdx.y * TC, r0 = blockIdx.z * kRows;
  if (r0 > l) return;
  const int nlt = sph_off(g.p + 1, g.p), sz = (l + 1) * TC;
  const double sl = (l & 1) ? -1.0 : 1.0;
  for (int e = threadIdx.x; e < 4 * sz; e += kMatThreads) {
    const int q = e / sz, i = e % sz, m = i / TC, w = w0 + i % TC;
    double2 ye = make_double2(0.0, 0.0), yo = ye;
    if (w < g.W) {
      const size_t at = ((size_t)(sph_off(m, g.p) + l - m) * 8 + 2 * q) * g.W + w;
      const double2 *Lp = b.loc_rot + at, *Lm = b.loc_rot + (size_t)nlt * 8 * g.W + at;
      const double2 ph = b.bloch[q * g.W + w], pc = make_double2(ph.x, -ph.y);
      double2 a = Lp[0], d = Lp[g.W], a2 = make_double2(0.0, 0.0), d2 = a2;
      if (m > 0) {
        a2 = Lm[0];
        d2 = Lm[g.W];
      }
      // even rows: (a + sl a2) ph + (d + sl d2) / ph; odd: (a - sl a2) ph - (d - sl d2) / ph
      const double2 ae = cmul(ph, make_double2(fma(sl, a2.x, a.x), fma(sl, a2.y, a.y)));
      const double2 de = cmul(pc, make_double2(fma(sl, d2.x, d.x), fma(sl, d2.y, d.y)));
      const double2 ao = cmul(ph, make_double2(fma(-sl, a2.x, a.x), fma(-sl, a2.y, a.y)));
      const double2 dd = cmul(pc, make_double2(fma(-sl, d2.x, d.x), fma(-sl, d2.y, d.y)));
      ye = make_double2(ae.x + de.x, ae.y + de.y);
      yo = make_double2(ao.x - dd.x, ao.y - dd.y);
    }
    shc[(2 * q) * sz + i] = ye;
    shc[(2 * q + 1) * sz + i] = yo;
  }
  __syncthreads();
  const int cc = threadIdx.x % TC, w = w0 + cc, m = r0 + threadIdx.x / TC;
  if (m > l || w >= g.W) return;
  double2 lp = make_double2(0.0, 0.0), lm = lp;
  for (int q = 0; q < 4; ++q) {
    double2 e = make_double2(0.0, 0.0), o = e;
    parity_dot<TC>(b.delta + delta_off(l) + (size_t)m * (l + 1), shc + (2 * q + (m & 1)) * sz + cc, l + 1, e, o);
    const double2 t = b.turn[q * (g.p + 1) + m];
    const double2 u = cmul(make_double2(t.x, -t.y), make_double2(e.x + o.x, e.y + o.y));
    const double2 v = cmul(t, make_double2(e.x - o.x, e.y - o.y));
    lp = make_double2(lp.x + u.x, lp.y + u.y);
    lm = make_double2(lm.x + v.x, lm.y + v.y);
  }
  b.loc[(size_t)(l * l + l + m) * g.W + w] = lp;
  if (m > 0) b.loc[(size_t)(l * l + l - m) * g.W + w] = make_double2(sl * lm.x, sl * lm.y);
}

// ---------------------------------------------------------------- steps 6, 7

// CTA: mode slot n, 32 rings (one per lane), TC waves over the warps: sum over
// m = n mod P.
template <int TC>
__global__ void __launch_bounds__(kMatThreads)
sph_l2p_kernel(SphArgs g, SphBuf b) {
  extern __shared__ double2 shc[];
  constexpr int NG = TC < 4 ? TC : 4, WG = TC / NG;        // warps in use, waves per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = blockIdx.x, i = blockIdx.y * 32 + lane, w0 = blockIdx.z * TC;
  const int ic = min(i, g.M - 1);
  double2 acc[WG];
#pragma unroll
  for (int w = 0; w < WG; ++w) acc[w] = make_double2(0.0, 0.0);
  for (int m = n - (n + g.p) / g.P * g.P; m <= g.p; m += g.P) {
    const int am = m < 0 ? -m : m, nl = g.p + 1 - am;
    const double sg = m < 0 && (am & 1) ? -1.0 : 1.0;
    __syncthreads();
    for (int e = threadIdx.x; e < nl * TC; e += kMatThreads) {
      const int l = am + e / TC, w = w0 + e % TC;
      const double2 v = w < g.W ? b.loc[(size_t)(l * l + l + m) * g.W + w] : make_double2(0.0, 0.0);
      shc[e] = make_double2(sg * v.x, sg * v.y);
    }
    __syncthreads();
    if (warp >= NG) continue;
    const double *B = b.B + (size_t)sph_off(am, g.p) * g.M + ic;
#pragma unroll 4
    for (int l = 0; l < nl; ++l) {
      const double v = B[(size_t)l * g.M];
#pragma unroll
      for (int w = 0; w < WG; ++w) {
        const double2 x = shc[l * TC + warp * WG + w];
        acc[w].x = fma(v, x.x, acc[w].x);
        acc[w].y = fma(v, x.y, acc[w].y);
      }
    }
  }
  if (i >= g.M || warp >= NG) return;
#pragma unroll
  for (int w = 0; w < WG; ++w) {
    const int ww = w0 + warp * WG + w;
    if (ww < g.W) b.modes[((size_t)ww * g.P + n) * g.M + i] = acc[w];
  }
}

// U[w][i][l] = sum_n modes[w][n][i] e^{2 pi i n l / P}: one warp per ring, 8 rings per CTA.
constexpr int kDftSeq = 8;
__global__ void __launch_bounds__(32 * kDftSeq)
sph_dft_kernel(const ObsDev *__restrict__ od, SphArgs g, const double2 *__restrict__ modes,
               double2 *__restrict__ U) {
  const ObsDev &o = *od;
  const int P = g.P;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = blockIdx.y, i0 = blockIdx.x * kDftSeq, i = i0 + warp;
  extern __shared__ double2 shc[];
  double2 *tw = shc;
  int *perm = reinterpret_cast<int *>(shc + P);
  double2 *seqs = shc + P + (P + 1) / 2, *seq = seqs + warp * P;
  const bool fft = o.fft_nst > 0;
  for (int l = threadIdx.x; l < P; l += 32 * kDftSeq) {
    tw[l] = o.tw_P[l];
    perm[l] = fft ? o.fft_perm[l] : l;
  }
  for (int e = threadIdx.x; e < P * kDftSeq; e += 32 * kDftSeq) {       // rings fastest: coalesced
    const int n = e / kDftSeq, q = e % kDftSeq;
    const double2 c = i0 + q < g.M ? modes[((size_t)w * P + n) * g.M + i0 + q] : make_double2(0.0, 0.0);
    seqs[q * P + n] = make_double2(c.x, -c.y);
  }
  __syncthreads();
  if (i >= g.M) return;
  double2 *out = U + ((size_t)w * g.M + i) * P;
  if (fft) {
    fft::warp_fft(seq, P, tw, o.fft_rad, o.fft_nst, lane);
    for (int l = lane; l < P; l += 32) {
      const double2 v = seq[perm[l]];
      out[l] = make_double2(v.x, -v.y);
    }
  } else {
    for (int l = lane; l < P; l += 32) {
      double2 s = make_double2(0.0, 0.0);
      int t = 0;                                            // n l mod P
      for (int n = 0; n < P; ++n) {
        const double2 a = seq[n], e = tw[t];
        s.x = fma(a.x, e.x, fma(-a.y, e.y, s.x));
        s.y = fma(a.x, e.y, fma(a.y, e.x, s.y));
        t += l;
        if (t >= P) t -= P;
      }
      out[l] = make_double2(s.x, -s.y);
    }
  }
}

// ---------------------------------------------------------------- host

// Binary exponents of |j_l(x)| and |h_l(x)|, l = 0 .. L (h_l of the order of
// its y part beyond the turning point, where it matters).
void bessel_exponents(double x, int L, int *ej, int *eh) {
  const double ix = 1.0 / x;
  int sc = 0;
  if (ej) {
    double f1 = 0.0, f0 = 1.0;
    for (int l = L + (int)x + 40; l >= 1; --l) {
      const double fm = (2.0 * l + 1.0) * ix * f0 - f1;
      f1 = f0;
      f0 = fm;
      if (l - 1 <= L) ej[l - 1] = sc + (fm != 0.0 ? std::ilogb(fm) : -1100);
      if (std::fabs(fm) > 0x1p500) {
        f0 *= 0x1p-500;
        f1 *= 0x1p-500;
        sc += 500;
      }
    }
    const double j0 = std::sin(x) * ix, j1 = (j0 - std::cos(x)) * ix;
    const bool zero = std::fabs(j0) >= std::fabs(j1);
    const int shift = std::ilogb(zero ? j0 : j1) - std::ilogb(zero ? f0 : f1) - sc;   // f0, f1 = f_0, f_1
    for (int l = 0; l <= L; ++l) ej[l] += shift;
  }
  if (!eh) return;
  double y0 = -std::cos(x) * ix, y1 = (y0 - std::sin(x)) * ix;
  sc = 0;
  for (int l = 0; l <= L; ++l) {
    eh[l] = sc + std::max(std::ilogb(std::fabs(y0) + std::fabs(y1) * 0.5), -1100);
    const double y2 = (2.0 * l + 3.0) * ix * y1 - y0;
    y0 = y1;
    y1 = y2;
    if (std::fabs(y1) > 0x1p500) {
      y0 *= 0x1p-500;
      y1 *= 0x1p-500;
      sc += 500;
    }
  }
}

size_t sph_align(size_t n) { return (n + 255) & ~(size_t)255; }

// Waves per CTA of the small products.
int wave_tile(int W) { return W >= 8 ? 8 : W > 2 ? 4 : W; }

size_t sph_layout(const ObsDev &h, int W, int p, int ncls, char *base, SphBuf *b) {
  const size_t nl = sph_off(p + 1, p), L = 2 * p + 1;
  size_t total = 0;
  auto put = [&](size_t n) {
    char *q = base ? base + total : nullptr;
    total += sph_align(n);
    return q;
  };
  SphBuf t;
  t.S = reinterpret_cast<double *>(put(sizeof(double) * nl * h.N));
  t.B = reinterpret_cast<double *>(put(sizeof(double) * nl * h.M));
  t.delta = reinterpret_cast<double *>(put(sizeof(double) * delta_off(p + 1)));
  t.hank = reinterpret_cast<double2 *>(put(sizeof(double2) * ncls * L));
  t.turn = reinterpret_cast<double2 *>(put(sizeof(double2) * 4 * (p + 1)));
  t.bloch = reinterpret_cast<double2 *>(put(sizeof(double2) * 4 * W));
  t.T = reinterpret_cast<double2 *>(put(sizeof(double2) * ncls * (size_t)t_off(p + 1, p)));
  t.mult = reinterpret_cast<double2 *>(put(sizeof(double2) * (size_t)(p + 1) * (p + 1) * W));
  t.rot = reinterpret_cast<double2 *>(put(sizeof(double2) * nl * 8 * W));
  t.loc_rot = reinterpret_cast<double2 *>(put(sizeof(double2) * nl * 16 * W));
  t.loc = reinterpret_cast<double2 *>(put(sizeof(double2) * (size_t)(p + 1) * (p + 1) * W));
  t.modes = reinterpret_cast<double2 *>(put(sizeof(double2) * (size_t)W * h.P * h.M));
  if (b) *b = t;
  return total;
}

int sph_classes(double ex, double ey) { return ex == ey ? 2 : 3; }

// One function a kernel, so that a kernel has one record of the shared memory it
// was granted: a second record (one per wave tile below) would let a smaller
// grant replace a larger one that the first still counts on.
cudaError_t launch_setup(const ObsDev *d_o, const SphArgs &g, const SphBuf &b, const double *dirs,
                         cudaStream_t st) {
  const int p = g.p, L = 2 * p + 1, parts = (p / 2 + 1 + kTabWarps - 1) / kTabWarps;
  const int blocks = g.ncls + 4 + ((g.M + 31) / 32 + (g.N + 31) / 32) * parts + p + 1;
  const size_t table = sizeof(double) * ((size_t)(p + 2) * 32 + (size_t)kTabWarps * 6 * (p + 1));
  const size_t smem = std::max(table, sizeof(double) * ((size_t)3 * L + 1));
  static size_t granted = 0;
  const cudaError_t e = ensure_dynamic_smem(sph_setup_kernel, smem, granted);
  if (e != cudaSuccess) return e;
  sph_setup_kernel<<<blocks, kSetupThreads, smem, st>>>(d_o, g, b, dirs, parts);
  return cudaGetLastError();
}

template <int TP>
cudaError_t launch_p2m(const SphArgs &g, const SphBuf &b, const double2 *coef, cudaStream_t st) {
  const int p = g.p, L = 2 * p + 1;
  const size_t block = sizeof(double) * (3 * L + 1) + 3 * sizeof(double2) * L;
  const size_t tile = sizeof(double) * 32 * 33 + sizeof(double2) * 32 * 2 * TP;
  const size_t smem = std::max(block, tile);
  static size_t granted = 0;
  const cudaError_t e = ensure_dynamic_smem(sph_p2m_kernel<TP>, smem, granted);
  if (e != cudaSuccess) return e;
  sph_p2m_kernel<TP><<<dim3(p + 1, g.ncls + (p + 32) / 32 * ((g.W + TP - 1) / TP)), kMatThreads, smem, st>>>(
      g, b, coef);
  return cudaGetLastError();
}

cudaError_t launch_dft(const ObsDev *d_o, const SphArgs &g, const SphBuf &b, double2 *U, cudaStream_t st) {
  const size_t smem = sizeof(double2) * ((size_t)g.P + (g.P + 1) / 2 + (size_t)kDftSeq * g.P);
  static size_t granted = 0;
  const cudaError_t e = ensure_dynamic_smem(sph_dft_kernel, smem, granted);
  if (e != cudaSuccess) return e;
  sph_dft_kernel<<<dim3((g.M + kDftSeq - 1) / kDftSeq, g.W), 32 * kDftSeq, smem, st>>>(d_o, g, b.modes, U);
  return cudaGetLastError();
}

template <int TC>
cudaError_t sph_launch(const ObsDev *d_o, const SphArgs &g, const SphBuf &b,
                       const double2 *coef, const double *dirs, double2 *U, cudaStream_t st) {
  const int p = g.p, wt = (g.W + TC - 1) / TC;
  const int slabs = (p + kMatThreads / TC) / (kMatThreads / TC);   // of the rows 0 .. p
  cudaError_t e;
  constexpr int TP = TC < 4 ? TC : 4;      // finer tiles: the orders' degree ranges are uneven
  if ((e = launch_setup(d_o, g, b, dirs, st)) != cudaSuccess) return e;
  if ((e = launch_p2m<TP>(g, b, coef, st)) != cudaSuccess) return e;
  {
    const size_t smem = 2 * sizeof(double2) * (p + 1) * TC;
    static size_t granted = 0;
    if ((e = ensure_dynamic_smem(sph_rot_fwd_kernel<TC>, smem, granted)) != cudaSuccess) return e;
    sph_rot_fwd_kernel<TC><<<dim3(p + 1, 4, wt * slabs), kMatThreads, smem, st>>>(g, b, wt);
  }
  {
    const size_t smem = sizeof(double2) * (p + 1) * TC;
    static size_t granted = 0;
    if ((e = ensure_dynamic_smem(sph_axial_kernel<TC>, smem, granted)) != cudaSuccess) return e;
    sph_axial_kernel<TC><<<dim3(p + 1, 8, wt * slabs), kMatThreads, smem, st>>>(g, b, wt);
  }
  {
    const size_t smem = 8 * sizeof(double2) * (p + 1) * TC;
    static size_t granted = 0;
    if ((e = ensure_dynamic_smem(sph_rot_bwd_kernel<TC>, smem, granted)) != cudaSuccess) return e;
    sph_rot_bwd_kernel<TC><<<dim3(p + 1, wt, slabs), kMatThreads, smem, st>>>(g, b);
  }
  {
    const size_t smem = sizeof(double2) * (p + 1) * TC;
    static size_t granted = 0;
    if ((e = ensure_dynamic_smem(sph_l2p_kernel<TC>, smem, granted)) != cudaSuccess) return e;
    sph_l2p_kernel<TC><<<dim3(g.P, (g.M + 31) / 32, wt), kMatThreads, smem, st>>>(g, b);
  }
  return launch_dft(d_o, g, b, U, st);
}

}  // namespace

// The degree p at which the truncated sums reach FP64 rounding, or 0 where the
// expansions do not serve: the first neglected terms of both expansions,
// (2l + 1) j_l(k r_s) h_l(k (D - r_t)) and (2l + 1) j_l(k r_t) h_l(k (D - r_s)),
// with the derivative's factor l, below 2^-58 of the largest. D is the shorter
// period. Refused: p above kSphMaxDegree (an image too close, or very large
// k r), k r beyond what the translation keeps of the caller's digits (the note at
// the head of this file), coefficients h_2p(kD) beyond the FP64 range (k D far below 1), k D of 2^19
// and more (the recurrences were compared with quadruple precision up to 7e5),
// and targets on the axis, where the derivative's recurrence divides by
// sin(theta).
int near_sph_degree(const ObsDev &h, double ex, double ey, int slices) {
  const double D = std::min(ex, ey), rs = h.sph_rs, rt = h.sph_rt;
  if (!(rs > 0.0) || !(rt > 0.0) || !(h.sph_rho_min > 1e-6 * rt) || !(D > 1.02 * (rs + rt))) return 0;
  const double r = std::max(rs, rt);
  if (!(h.k * r <= (slices >= 7 ? 45.0 : 55.0)) || !(h.k * std::hypot(ex, ey) < 0x1p19) || !(h.k * (D - r) > 0x1p-100)) return 0;
  constexpr int L = 2 * kSphMaxDegree + 2;
  int ja[L + 1], jb[L + 1], ha[L + 1], hb[L + 1];
  constexpr int L1 = kSphMaxDegree + 1;
  bessel_exponents(h.k * rs, L1, ja, nullptr);
  bessel_exponents(h.k * rt, L1, jb, nullptr);
  bessel_exponents(h.k * (D - rt), L1, nullptr, ha);
  bessel_exponents(h.k * (D - rs), L1, nullptr, hb);
  int top = -100000;
  for (int l = 0; l <= kSphMaxDegree; ++l) {
    const int w = std::ilogb(2.0 * l + 1.0);
    top = std::max(top, w + std::max(ja[l] + ha[l], jb[l] + hb[l]));
  }
  int p = kSphMaxDegree + 1;
  while (p > 0) {
    const int w = std::ilogb(2.0 * p + 1.0) + std::ilogb(p + 1.0);
    if (w + std::max(ja[p] + ha[p], jb[p] + hb[p]) > top - 58) break;
    --p;
  }
  if (p > kSphMaxDegree) return 0;
  if (p < 4) p = 4;
  bessel_exponents(h.k * D, L, nullptr, ha);
  return ha[2 * p + 1] + 16 < 1000 ? p : 0;
}

// Microseconds of the seven launches, measured: launches and serial chains of
// length p, then the products' FP64 operations.
double near_sph_estimate_us(const ObsDev &h, int W, int p) {
  const double n = p + 1.0, fma = W * n * n * (16.0 * n + 2.0 * (h.N + h.M));
  return 120.0 + p + fma / 4e5;
}

size_t near_sph_scratch_bytes(const ObsDev &h, int W, double ex, double ey, int p) {
  return sph_layout(h, W, p, sph_classes(ex, ey), nullptr, nullptr);
}

cudaError_t launch_near_sph(const ObsDev *d_o, const ObsDev &h, int W, const double2 *coef, double ex,
                            double ey, const double *dirs, int p, double2 *U, void *scratch,
                            cudaStream_t st) {
  SphArgs g;
  g.p = p; g.W = W; g.M = h.M; g.N = h.N; g.P = h.P; g.cols = h.cols;
  g.k = h.k; g.zc = h.sph_zc;
  g.ncls = sph_classes(ex, ey);
  const double dx[4] = {ex, 0.0, ex, ex}, dy[4] = {0.0, ey, ey, -ey};
  g.dist[0] = ex;
  g.dist[1] = std::hypot(ex, ey);
  g.dist[2] = ey;
  for (int q = 0; q < 4; ++q) {
    g.cx[q] = dx[q];
    g.cy[q] = dy[q];
    g.phi[q] = std::atan2(dy[q], dx[q]);
    g.cls[q] = q >= 2 ? 1 : (q == 1 && g.ncls == 3 ? 2 : 0);
  }
  SphBuf b;
  sph_layout(h, W, p, g.ncls, static_cast<char *>(scratch), &b);
  switch (wave_tile(W)) {
    case 1: return sph_launch<1>(d_o, g, b, coef, dirs, U, st);
    case 2: return sph_launch<2>(d_o, g, b, coef, dirs, U, st);
    case 4: return sph_launch<4>(d_o, g, b, coef, dirs, U, st);
    default: return sph_launch<8>(d_o, g, b, coef, dirs, U, st);
  }
}

}  // namespace axi
