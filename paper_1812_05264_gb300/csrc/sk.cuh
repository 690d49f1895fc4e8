// Slater-Koster two-centre blocks for an s/p/d basis (Slater & Koster, Phys. Rev. 94, 1498
// (1954), Table I), and the derivative of a weighted sum of a block's entries in the bond vector.
// Orbital order s, px, py, pz, dxy, dyz, dzx, dx2-y2, d3z2-r2;
// block(d)[i][j] couples orbital i on atom a with orbital j on atom b, d = R_b - R_a.
#pragma once
#include <math.h>

namespace tbk {

// Angular momentum of each orbital (parity of the reversed bond is (-1)^(la + lb)).
__host__ __device__ inline int sk_l(int i) { return i == 0 ? 0 : (i < 4 ? 1 : 2); }

__host__ __device__ inline void sk_block(const double d[3], const double V[10], double r0,
                                         double decay, double E[81]) {
  using T = double;
  const double s3 = 1.7320508075688772;  // sqrt(3)
  const T r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  const T l = d[0] / r, m = d[1] / r, n = d[2] / r;
  const T f = exp(-decay * (r / T(r0) - T(1.0)));
  T v[10];
  for (int i = 0; i < 10; ++i) v[i] = V[i] * f;
  const T &sss = v[0], &sps = v[1], &sds = v[2], &pps = v[3], &ppp = v[4], &pds = v[5],
          &pdp = v[6], &dds = v[7], &ddp = v[8], &ddd = v[9];
  const T ll = l * l, mm = m * m, nn = n * n, one(1.0);
  const T lm = l * m, mn = m * n, nl = n * l, lmn = lm * n;
  const T amb = ll - mm;                 // l^2 - m^2
  const T z2 = nn - 0.5 * (ll + mm);     // n^2 - (l^2 + m^2)/2
  const T dir[3] = {l, m, n};
  const T sq[3] = {ll, mm, nn};
  // s row
  E[0] = sss;
  for (int a = 0; a < 3; ++a) E[1 + a] = dir[a] * sps;
  E[4] = s3 * lm * sds;
  E[5] = s3 * mn * sds;
  E[6] = s3 * nl * sds;
  E[7] = (0.5 * s3) * amb * sds;
  E[8] = z2 * sds;
  // p-p: d_a d_b (pps - ppp) + delta_ab ppp
  for (int a = 0; a < 3; ++a)
    for (int b = a; b < 3; ++b) {
      T e = dir[a] * dir[b] * (pps - ppp);
      if (a == b) e = e + ppp;
      E[9 * (1 + a) + 1 + b] = e;
    }
  // p-d.  For p_a against d_xy-like orbitals (pairs (x,y)=4, (y,z)=5, (z,x)=6):
  //   p_a . d_bc = sqrt3 d_a d_b d_c pds + (delta_ab d_c + delta_ac d_b - 2 d_a d_b d_c) pdp
  const int pr[3][2] = {{0, 1}, {1, 2}, {2, 0}};
  for (int a = 0; a < 3; ++a)
    for (int q = 0; q < 3; ++q) {
      const int b = pr[q][0], c = pr[q][1];
      const T abc = dir[a] * dir[b] * dir[c];
      T e = s3 * abc * pds - 2.0 * abc * pdp;
      if (a == b) e = e + dir[c] * pdp;
      if (a == c) e = e + dir[b] * pdp;
      E[9 * (1 + a) + 4 + q] = e;
    }
  // p - d(x2-y2)
  E[9 * 1 + 7] = (0.5 * s3) * l * amb * pds + l * (one - amb) * pdp;
  E[9 * 2 + 7] = (0.5 * s3) * m * amb * pds - m * (one + amb) * pdp;
  E[9 * 3 + 7] = (0.5 * s3) * n * amb * pds - n * amb * pdp;
  // p - d(3z2-r2)
  E[9 * 1 + 8] = l * z2 * pds - s3 * l * nn * pdp;
  E[9 * 2 + 8] = m * z2 * pds - s3 * m * nn * pdp;
  E[9 * 3 + 8] = n * z2 * pds + s3 * n * (ll + mm) * pdp;
  // d_xy-like with d_xy-like (diagonal): 3 a^2 b^2 dds + (a^2 + b^2 - 4 a^2 b^2) ddp +
  // (c^2 + a^2 b^2) ddd, with (a, b, c) = (l, m, n), (m, n, l), (n, l, m)
  for (int q = 0; q < 3; ++q) {
    const int a = pr[q][0], b = pr[q][1], c = 3 - a - b;
    const T a2b2 = sq[a] * sq[b];
    E[9 * (4 + q) + 4 + q] = 3.0 * a2b2 * dds + (sq[a] + sq[b] - 4.0 * a2b2) * ddp + (sq[c] + a2b2) * ddd;
  }
  // off-diagonal d_xy-like pairs: (xy,yz), (xy,zx), (yz,zx).  For orbitals sharing the
  // coordinate k, with the other two coordinates i (first) and j (second):
  //   3 i k^2 j dds + i j (1 - 4 k^2) ddp + i j (k^2 - 1) ddd
  {
    // (xy, yz): shared y, others x, z
    E[9 * 4 + 5] = 3.0 * l * mm * n * dds + nl * (one - 4.0 * mm) * ddp + nl * (mm - one) * ddd;
    // (xy, zx): shared x, others y, z
    E[9 * 4 + 6] = 3.0 * ll * mn * dds + mn * (one - 4.0 * ll) * ddp + mn * (ll - one) * ddd;
    // (yz, zx): shared z, others y, x
    E[9 * 5 + 6] = 3.0 * lm * nn * dds + lm * (one - 4.0 * nn) * ddp + lm * (nn - one) * ddd;
  }
  // d_xy-like with d(x2-y2)
  E[9 * 4 + 7] = 1.5 * lm * amb * dds - 2.0 * lm * amb * ddp + 0.5 * lm * amb * ddd;
  E[9 * 5 + 7] = 1.5 * mn * amb * dds - mn * (one + 2.0 * amb) * ddp + mn * (one + 0.5 * amb) * ddd;
  E[9 * 6 + 7] = 1.5 * nl * amb * dds + nl * (one - 2.0 * amb) * ddp - nl * (one - 0.5 * amb) * ddd;
  // d_xy-like with d(3z2-r2)
  E[9 * 4 + 8] = s3 * lm * z2 * dds - 2.0 * s3 * lm * nn * ddp + (0.5 * s3) * lm * (one + nn) * ddd;
  E[9 * 5 + 8] = s3 * mn * z2 * dds + s3 * mn * (ll + mm - nn) * ddp - (0.5 * s3) * mn * (ll + mm) * ddd;
  E[9 * 6 + 8] = s3 * nl * z2 * dds + s3 * nl * (ll + mm - nn) * ddp - (0.5 * s3) * nl * (ll + mm) * ddd;
  // e_g block
  E[9 * 7 + 7] = 0.75 * amb * amb * dds + (ll + mm - amb * amb) * ddp + (nn + 0.25 * amb * amb) * ddd;
  E[9 * 7 + 8] = (0.5 * s3) * amb * z2 * dds - s3 * nn * amb * ddp + (0.25 * s3) * (one + nn) * amb * ddd;
  E[9 * 8 + 8] = z2 * z2 * dds + 3.0 * nn * (ll + mm) * ddp + 0.75 * (ll + mm) * (ll + mm) * ddd;
  // lower triangle from the parity of the reversed bond
  for (int i = 0; i < 9; ++i)
    for (int j = 0; j < i; ++j) {
      const T u = E[9 * j + i];
      E[9 * i + j] = ((sk_l(i) + sk_l(j)) & 1) ? -u : u;
    }
}

// t = sum_ij S_ij dE_ij/dd, E = sk_block(d), for a full 9 x 9 weight S: the derivative of the one number
// sum_ij S_ij E_ij, taken in reverse.  Weights of E_ij and E_ji = +-E_ij are added first; the number is then a
// polynomial in the direction cosines u (and their products q = u_a u_a, x = (lm, mn, nl), amb = l^2 - m^2,
// z2), whose adjoints g* are collected entry by entry.  l^2 + m^2 + n^2 = 1 is used throughout: only the part
// of du normal to u counts.  About 300 FP64 operations, where the forward mode over all entries takes 2,500.
// S(i, j) returns a weight.
template <class W>
__host__ __device__ inline void sk_bond_term(const double d[3], const double V[10], double r0, double decay,
                                             const W& S, double t[3]) {
  const double s3 = 1.7320508075688772;  // sqrt(3)
  const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]), ir = 1.0 / r;
  const double f = exp(-decay * (r / r0 - 1.0));
  const double u[3] = {d[0] * ir, d[1] * ir, d[2] * ir};
  const double q[3] = {u[0] * u[0], u[1] * u[1], u[2] * u[2]};
  const double x[3] = {u[0] * u[1], u[1] * u[2], u[2] * u[0]};
  const double amb = q[0] - q[1], z2 = 1.5 * q[2] - 0.5;
  const double sss = V[0], sps = V[1], sds = V[2], pps = V[3], ppp = V[4], pds = V[5], pdp = V[6], dds = V[7],
               ddp = V[8], ddd = V[9];
  auto even = [&](int i, int j) { return S(i, j) + S(j, i); };
  auto odd = [&](int i, int j) { return S(i, j) - S(j, i); };
  double gu[3], gq[3] = {0, 0, 0}, gx[3], ga = 0, phi;

  // s row (s3 lm sds, ..; (s3/2) amb sds; z2 sds)
  phi = S(0, 0) * sss;
  for (int a = 0; a < 3; ++a) {
    gu[a] = sps * odd(0, 1 + a);
    phi += gu[a] * u[a];
    gx[a] = s3 * sds * even(0, 4 + a);
    phi += gx[a] * x[a];
  }
  {
    const double w7 = 0.5 * s3 * sds * even(0, 7), w8 = sds * even(0, 8);
    phi += w7 * amb + w8 * z2;
    ga += w7;
    gq[2] += 1.5 * w8;
  }
  // p-p
  {
    const double D = pps - ppp;
    for (int a = 0; a < 3; ++a) {
      const double c = S(1 + a, 1 + a), w = D * c, w2 = D * even(1 + a, 1 + (a + 1) % 3);
      phi += w * q[a] + ppp * c + w2 * x[a];
      gq[a] += w;
      gx[a] += w2;
    }
  }
  // p-d: u_a x_b (s3 pds - 2 pdp) and the terms linear in u
  {
    const double A = s3 * pds - 2.0 * pdp;
    for (int b = 0; b < 3; ++b) {
      const int i = b, j = (b + 1) % 3;  // orbital 4 + b is the product u_i u_j
      double L = 0;
      for (int a = 0; a < 3; ++a) {
        const double w = odd(1 + a, 4 + b);
        L += w * u[a];
        gu[a] += A * x[b] * w;
        if (a == i) {
          gu[j] += pdp * w;
          phi += pdp * w * u[j];
        }
        if (a == j) {
          gu[i] += pdp * w;
          phi += pdp * w * u[i];
        }
      }
      phi += A * x[b] * L;
      gx[b] += A * L;
    }
    const double B = 0.5 * s3 * pds - pdp, H = z2 * pds - s3 * q[2] * pdp;
    double P7 = 0, P8 = 0;
    double w7[3], w8[3];
    for (int a = 0; a < 3; ++a) {
      w7[a] = odd(1 + a, 7);
      w8[a] = odd(1 + a, 8);
      P7 += w7[a] * u[a];
      P8 += w8[a] * u[a];
      gu[a] += B * amb * w7[a] + H * w8[a];
    }
    const double l0 = pdp * w7[0], l1 = -pdp * w7[1], l2 = s3 * pdp * w8[2];
    gu[0] += l0;
    gu[1] += l1;
    gu[2] += l2;
    phi += B * amb * P7 + H * P8 + l0 * u[0] + l1 * u[1] + l2 * u[2];
    ga += B * P7;
    gq[2] += P8 * (1.5 * pds - s3 * pdp);
  }
  // d-d
  {
    const double K = 3.0 * dds - 4.0 * ddp + ddd, D = ddd - ddp, M = 0.5 * (K * q[2] + ddd - dds);
    for (int b = 0; b < 3; ++b) {
      const int o = (b + 2) % 3;  // the coordinate that product b lacks
      const double c = S(4 + b, 4 + b);
      const double e = even(4 + b, 4 + (b + 1) % 3);  // K x_b x_{b+1} - D x_{b+2}
      const double cx = K * c * x[b], ex = K * e;
      phi += cx * x[b] + c * (D * q[o] + ddp) + ex * x[b] * x[(b + 1) % 3] - D * e * x[o];
      gx[b] += 2.0 * cx + ex * x[(b + 1) % 3];
      gx[(b + 1) % 3] += ex * x[b];
      gx[o] -= D * e;
      gq[o] += D * c;
    }
    double P7 = 0, P8 = 0;
    double w7[3], w8[3];
    for (int b = 0; b < 3; ++b) {
      w7[b] = even(4 + b, 7);
      w8[b] = s3 * even(4 + b, 8);
      P7 += w7[b] * x[b];
      P8 += w8[b] * x[b];
      gx[b] += 0.5 * K * amb * w7[b] + M * w8[b];
    }
    const double k1 = D * (w7[1] - w8[1]), k2 = -D * (w7[2] + w8[2]);
    gx[1] += k1;
    gx[2] += k2;
    phi += 0.5 * K * amb * P7 + M * P8 + k1 * x[1] + k2 * x[2];
    ga += 0.5 * K * P7;
    gq[2] += 0.5 * K * P8;
    const double c77 = S(7, 7), c78 = 0.5 * s3 * even(7, 8), c88 = S(8, 8), n1 = 1.0 - q[2];
    phi += c77 * (0.25 * K * amb * amb + n1 * ddp + q[2] * ddd) + c78 * amb * M +
           c88 * (z2 * z2 * dds + 3.0 * q[2] * n1 * ddp + 0.75 * n1 * n1 * ddd);
    ga += 0.5 * K * amb * c77 + c78 * M;
    gq[2] += D * c77 + 0.5 * K * c78 * amb + c88 * (3.0 * z2 * dds + (3.0 - 6.0 * q[2]) * ddp - 1.5 * n1 * ddd);
  }
  gq[0] += ga;
  gq[1] -= ga;
  for (int a = 0; a < 3; ++a) gu[a] += 2.0 * u[a] * gq[a] + gx[a] * u[(a + 1) % 3] + gx[(a + 2) % 3] * u[(a + 2) % 3];
  const double ug = u[0] * gu[0] + u[1] * gu[1] + u[2] * gu[2];
  const double radial = -f * (decay / r0) * phi, fr = f * ir;
  for (int a = 0; a < 3; ++a) t[a] = radial * u[a] + fr * (gu[a] - ug * u[a]);
}

}  // namespace tbk
