// Reverse-mode (vector-Jacobian) building blocks of the collide-stream update.
//
// The axis sweeps are products of commuting 3-point maps, which gives short transposes: with
// central moments k_abc and raw moments r_abc related by the shift u,
//     d r_abc / d u_x = a r_{a-1,b,c}      (unshift, inverse sweeps)
//     d k_abc / d u_x = -a k_{a-1,b,c}     (shift, forward sweeps)
// whatever the other axes do.  So the adjoint of u over all three axes needs one set of
// moments at each end of the collision (the post-collision raw ones, the pre-collision
// central ones) and 18 multiply-adds per axis and end, instead of every intermediate stage of
// every sweep, which would take three relaxations and six inverse sweeps more.  The equilibrium
// offsets are differentiated in reverse, not with dual numbers of four partials.  (Both
// together, all else equal: pass A at 128^3 272 -> 245 us.)
#pragma once
#include "lbm_device.cuh"

namespace lbm {

// Central moments about u back to raw moments (inverse of shift_axis).
template <int STRIDE>
__device__ __forceinline__ void unshift_axis(float (&v)[27], float u) {
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int b = line_base<STRIDE>(l);
    const float k0 = v[b], k1 = v[b + STRIDE], k2 = v[b + 2 * STRIDE];
    const float r1 = fmaf(u, k0, k1);
    v[b + STRIDE] = r1;
    v[b + 2 * STRIDE] = fmaf(u, k1 + r1, k2);
  }
}

// Transpose of the raw moments' inverse along one axis (f(-1) = (r2 - r1) / 2, f(0) = r0 - r2,
// f(+1) = (r2 + r1) / 2): adjoint of the populations -> adjoint of the raw moments.
template <int STRIDE>
__device__ __forceinline__ void raw_inverse_vjp(float (&A)[27]) {
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int b = line_base<STRIDE>(l);
    const float m = A[b], z = A[b + STRIDE], p = A[b + 2 * STRIDE];
    A[b] = z;
    A[b + STRIDE] = 0.5f * (p - m);
    A[b + 2 * STRIDE] = fmaf(0.5f, p + m, -z);
  }
}

// Transpose of unshift_axis (r1 = k1 + u k0, r2 = k2 + 2 u k1 + u^2 k0): adjoint of raw
// moments -> of central moments.  With -u it is the transpose of shift_axis.
template <int STRIDE>
__device__ __forceinline__ void unshift_axis_vjp(float (&A)[27], float u) {
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int b = line_base<STRIDE>(l);
    const float a2 = A[b + 2 * STRIDE];
    const float t = fmaf(u, a2, A[b + STRIDE]);
    A[b] = fmaf(u, t, A[b]);
    A[b + STRIDE] = fmaf(u, a2, t);
  }
}

// sum over the moments of A_abc d m_abc / d u along the axis of STRIDE: A_1 m_0 + 2 A_2 m_1
// per line (see the header).
template <int STRIDE>
__device__ __forceinline__ float shift_dot(const float (&A)[27], const float (&m)[27]) {
  float s1 = 0.0f, s2 = 0.0f;
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int b = line_base<STRIDE>(l);
    s1 = fmaf(A[b + STRIDE], m[b], s1);
    s2 = fmaf(A[b + 2 * STRIDE], m[b + STRIDE], s2);
  }
  return fmaf(2.0f, s2, s1);
}

// Transpose of raw_axis (a linear map with constant coefficients).
template <int STRIDE>
__device__ __forceinline__ void raw_axis_vjp(float (&A)[27]) {
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int b = line_base<STRIDE>(l);
    const float r0 = A[b], r1 = A[b + STRIDE], r02 = r0 + A[b + 2 * STRIDE];
    A[b] = r02 - r1;
    A[b + STRIDE] = r0;
    A[b + 2 * STRIDE] = r02 + r1;
  }
}

// Transpose of relax_to_equilibrium.  K: the node's keep factors; v: the central moments
// before relaxation; A: adjoint of the relaxed moments on entry, of v on return.  Adds the
// adjoints of (rho - 1, u) to bar[0..3] and of the high-order keep factors to kbar[0..3].
// out_i = Delta_i + K (v_i - Delta_i): dv_i = K o, dDelta_i = (1 - K) o, dK = o (v_i - Delta_i);
// the equilibrium offsets Delta(rho - 1, u) are differentiated in reverse through their shared
// subexpressions (squares and products of squares of u), whose adjoints (X2b, XYb, ...) are
// folded into u's at the end.
__device__ __forceinline__ void relax_vjp(const float (&v)[27], float (&A)[27], float dr, float X,
                                          float Y, float Z, const Keep& kf, float (&bar)[4],
                                          float (&kbar)[4]) {
  const float third = 1.0f / 3.0f, ninth = 1.0f / 9.0f;
  const float X2 = X * X, Y2 = Y * Y, Z2 = Z * Z;
  const float YZ = Y * Z, XZ = X * Z, XY = X * Y;
  float Xb, Yb, Zb, X2b, Y2b, Z2b, drb;
  auto one = [&](int i, float dl, int grp) {     // returns the adjoint of Delta_i
    const float o = A[i], p = kf.g[grp] * o;
    A[i] = p;
    kbar[grp] = fmaf(o, v[i] - dl, kbar[grp]);
    return o - p;
  };
  auto shear = [&](int i) {
    const float o = A[i], p = kf.nu * o;
    A[i] = p;
    return o - p;
  };
  {  // second order, off-diagonal: Delta = -u_a u_b
    const float a = shear(kap(1, 1, 0)), b = shear(kap(1, 0, 1)), c = shear(kap(0, 1, 1));
    Xb = -fmaf(a, Y, b * Z);
    Yb = -fmaf(a, X, c * Z);
    Zb = -fmaf(b, X, c * Y);
  }
  {  // second-order diagonal: deviators at the shear rate, trace at group 9..16
    const float dr3 = dr * third;
    const float Aa = v[kap(2, 0, 0)] - (dr3 - X2), Bb = v[kap(0, 2, 0)] - (dr3 - Y2);
    const float Cc = v[kap(0, 0, 2)] - (dr3 - Z2);
    const float o2 = A[kap(2, 0, 0)], o3 = A[kap(0, 2, 0)], o4 = A[kap(0, 0, 2)];
    const float trb = (o2 + o3 + o4) * third;
    const float d1b = fmaf(-2.0f, o3, o2 + o4) * third;
    const float d2b = fmaf(-2.0f, o4, o2 + o3) * third;
    const float gt = kf.g[0] * trb;
    const float Ab = fmaf(kf.nu, d1b + d2b, gt);
    const float Bb_ = fmaf(-kf.nu, d1b, gt);
    const float Cb = fmaf(-kf.nu, d2b, gt);
    kbar[0] = fmaf(trb, Aa + Bb + Cc, kbar[0]);
    A[kap(2, 0, 0)] = Ab;
    A[kap(0, 2, 0)] = Bb_;
    A[kap(0, 0, 2)] = Cb;
    X2b = Ab - o2;
    Y2b = Bb_ - o3;
    Z2b = Cb - o4;
    drb = -(X2b + Y2b + Z2b) * third;
  }
  {  // third order: Delta_120 = X (1/3 - dr Y2), ..., Delta_111 = -dr X Y Z
    const float qx = fmaf(-dr, X2, third), qy = fmaf(-dr, Y2, third), qz = fmaf(-dr, Z2, third);
    const float p120 = one(kap(1, 2, 0), X * qy, 0), p102 = one(kap(1, 0, 2), X * qz, 0);
    const float p210 = one(kap(2, 1, 0), Y * qx, 0), p012 = one(kap(0, 1, 2), Y * qz, 0);
    const float p201 = one(kap(2, 0, 1), Z * qx, 0), p021 = one(kap(0, 2, 1), Z * qy, 0);
    Xb = fmaf(p120, qy, fmaf(p102, qz, Xb));
    Yb = fmaf(p210, qx, fmaf(p012, qz, Yb));
    Zb = fmaf(p201, qx, fmaf(p021, qy, Zb));
    const float sx = fmaf(p210, Y, p201 * Z), sy = fmaf(p120, X, p021 * Z);
    const float sz = fmaf(p102, X, p012 * Y);
    const float XYZ = XY * Z;
    const float p111 = one(kap(1, 1, 1), -dr * XYZ, 0);
    const float t = -p111 * dr;
    Xb = fmaf(t, YZ, Xb);
    Yb = fmaf(t, XZ, Yb);
    Zb = fmaf(t, XY, Zb);
    drb -= fmaf(p111, XYZ, fmaf(sx, X2, fmaf(sy, Y2, sz * Z2)));
    X2b = fmaf(-dr, sx, X2b);
    Y2b = fmaf(-dr, sy, Y2b);
    Z2b = fmaf(-dr, sz, Z2b);
  }
  const float X2Y2 = X2 * Y2, X2Z2 = X2 * Z2, Y2Z2 = Y2 * Z2;
  float XYb, XZb, YZb;                   // adjoints of X2 Y2, X2 Z2, Y2 Z2
  {  // fourth order: Delta_220 = r X2 Y2 + dr/9 - (X2 + Y2)/3, Delta_211 = Y Z (r X2 - 1/3)
    const float r = fmaf(3.0f, dr, 2.0f);   // 3 rho - 1
    const float dr9 = dr * ninth;
    const float p220 = one(kap(2, 2, 0), fmaf(r, X2Y2, fmaf(X2 + Y2, -third, dr9)), 1);
    const float p202 = one(kap(2, 0, 2), fmaf(r, X2Z2, fmaf(X2 + Z2, -third, dr9)), 1);
    const float p022 = one(kap(0, 2, 2), fmaf(r, Y2Z2, fmaf(Y2 + Z2, -third, dr9)), 1);
    XYb = r * p220;
    XZb = r * p202;
    YZb = r * p022;
    const float wx = fmaf(r, X2, -third), wy = fmaf(r, Y2, -third), wz = fmaf(r, Z2, -third);
    const float p211 = one(kap(2, 1, 1), YZ * wx, 1), p121 = one(kap(1, 2, 1), XZ * wy, 1);
    const float p112 = one(kap(1, 1, 2), XY * wz, 1);
    const float tx = p211 * YZ, ty = p121 * XZ, tz = p112 * XY;
    const float ax = p211 * wx, ay = p121 * wy, az = p112 * wz;
    Xb = fmaf(ay, Z, fmaf(az, Y, Xb));
    Yb = fmaf(ax, Z, fmaf(az, X, Yb));
    Zb = fmaf(ax, Y, fmaf(ay, X, Zb));
    X2b = fmaf(r, tx, fmaf(-third, p220 + p202, X2b));
    Y2b = fmaf(r, ty, fmaf(-third, p220 + p022, Y2b));
    Z2b = fmaf(r, tz, fmaf(-third, p202 + p022, Z2b));
    const float rb = fmaf(p220, X2Y2, fmaf(p202, X2Z2, fmaf(p022, Y2Z2,
                     fmaf(tx, X2, fmaf(ty, Y2, tz * Z2)))));
    drb = fmaf(3.0f, rb, fmaf(ninth, p220 + p202 + p022, drb));
  }
  {  // fifth order: Delta_122 = X (o Y2 Z2 + 1/9 - dr/3 (Y2 + Z2))
    const float o = fmaf(-6.0f, dr, -5.0f);   // 1 - 6 rho
    const float dr3 = dr * third;
    const float syz = Y2 + Z2, sxz = X2 + Z2, sxy = X2 + Y2;
    const float ix = fmaf(o, Y2Z2, fmaf(-dr3, syz, ninth));
    const float iy = fmaf(o, X2Z2, fmaf(-dr3, sxz, ninth));
    const float iz = fmaf(o, X2Y2, fmaf(-dr3, sxy, ninth));
    const float p122 = one(kap(1, 2, 2), X * ix, 2), p212 = one(kap(2, 1, 2), Y * iy, 2);
    const float p221 = one(kap(2, 2, 1), Z * iz, 2);
    Xb = fmaf(p122, ix, Xb);
    Yb = fmaf(p212, iy, Yb);
    Zb = fmaf(p221, iz, Zb);
    const float hx = p122 * X, hy = p212 * Y, hz = p221 * Z;
    YZb = fmaf(o, hx, YZb);
    XZb = fmaf(o, hy, XZb);
    XYb = fmaf(o, hz, XYb);
    X2b = fmaf(-dr3, hy + hz, X2b);
    Y2b = fmaf(-dr3, hx + hz, Y2b);
    Z2b = fmaf(-dr3, hx + hy, Z2b);
    drb = fmaf(-6.0f, fmaf(hx, Y2Z2, fmaf(hy, X2Z2, hz * X2Y2)),
               fmaf(-third, fmaf(hx, syz, fmaf(hy, sxz, hz * sxy)), drb));
  }
  {  // sixth order: Delta_222 = m X2 Y2 Z2 + n (X2 Y2 + X2 Z2 + Y2 Z2) + dr/27 - (X2 + Y2 + Z2)/9
    const float rho = 1.0f + dr;
    const float m = fmaf(10.0f, rho, -1.0f), n = rho - third;
    const float p2 = X2Y2 + X2Z2 + Y2Z2, q = X2Y2 * Z2;
    const float dl = fmaf(m, q, fmaf(n, p2, fmaf(dr, 1.0f / 27.0f, -ninth * (X2 + Y2 + Z2))));
    const float p = one(kap(2, 2, 2), dl, 3);
    const float pn = p * n, pm = p * m, p9 = -ninth * p;
    drb = fmaf(p, fmaf(10.0f, q, p2 + 1.0f / 27.0f), drb);
    XYb += fmaf(pm, Z2, pn);
    XZb += pn;
    YZb += pn;
    X2b += p9;
    Y2b += p9;
    Z2b += fmaf(pm, X2Y2, p9);
  }
  X2b = fmaf(XYb, Y2, fmaf(XZb, Z2, X2b));
  Y2b = fmaf(XYb, X2, fmaf(YZb, Z2, Y2b));
  Z2b = fmaf(XZb, X2, fmaf(YZb, Y2, Z2b));
  bar[0] += drb;
  bar[1] += fmaf(2.0f * X, X2b, Xb);
  bar[2] += fmaf(2.0f * Y, Y2b, Yb);
  bar[3] += fmaf(2.0f * Z, Z2b, Zb);
}

}  // namespace lbm
