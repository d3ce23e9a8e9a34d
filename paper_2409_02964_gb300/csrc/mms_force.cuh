// mms_force.cuh -- GENERATED by gen_mms_force.py; do not edit by hand.
//
// Body force of Eq. (25) (constant density, pressure term dropped) for the
// spatiotemporal manufactured solution phi = phi0 + A sin(kx) sin(ky) cos(wt),
// phi u = grad psi + rot Psi (see the generator for the definitions), per unit rho0.
// Arguments: sx, cx = sin, cos of k x; sy, cy = sin, cos of k y; ct, st = cos, sin
// of w t. Evaluated from phi, q = phi u and their derivatives, u by the quotient rule.
// T is the arithmetic type (float, or ForceV, whose products join the sum they enter in
// one fused operation); it must provide products of T values, of a float and a T, sums of
// these, T + float, and mms_rcp(T).
#pragma once

namespace lbmv {

template <typename T>
__device__ __forceinline__ void mms_force(T sx, T cx, T sy, T cy, float ct, float st, float k, float w, float A,
                                          float U0, float phi0, float nu, T& fx, T& fy) {
    const float a = A * ct;
    const float b = -(A * w * st) / (2.0f * k);
    const float bt = -(A * w * w * ct) / (2.0f * k);
    const float n1 = nu * k;
    const float c1 = bt / k + (2.0f / 3.0f) * n1 * b;
    const float c2 = 2.0f * n1;
    const float m7 = -(7.0f / 3.0f) * n1;
    const float m1 = (1.0f / 3.0f) * n1;
    const T asx = a * sx;
    const T acx = a * cx;
    const T nasx = (-a) * sx;
    const T nacx = (-a) * cx;
    const T bsx = b * sx;
    const T bcx = b * cx;
    const T nbsx = (-b) * sx;
    const T usx = U0 * sx;
    const T ucx = U0 * cx;
    const T nusx = (-U0) * sx;
    const T nucx = (-U0) * cx;
    const T dsx = c1 * sx;
    const T dcx = c1 * cx;
    const T e1 = asx * sy;
    const T e2 = acx * cy;
    const T ph = asx * sy + phi0;
    const T npx = nacx * sy;
    const T npy = nasx * cy;
    const T qx = bcx * sy + usx * cy;
    const T qy = bsx * cy + nucx * sy;
    const T nbss = nbsx * sy;
    const T bcc = bcx * cy;
    const T qxx = ucx * cy + nbss;
    const T qyy = nucx * cy + nbss;
    const T qxy = nusx * sy + bcc;
    const T qyx = usx * sy + bcc;
    const T ip = mms_rcp(ph);
    const T ux = qx * ip;
    const T uy = qy * ip;
    const T uxx = (ux * npx + qxx) * ip;
    const T uxy = (ux * npy + qxy) * ip;
    const T uyx = (uy * npx + qyx) * ip;
    const T uyy = (uy * npy + qyy) * ip;
    const T dv = uxx + uyy;
    const T dc = dv + c2;
    const T hx = (-n1) * npx;
    const T hy = (-n1) * npy;
    const T gx = dcx * sy + ux * (m7 * e1 + qxx) + uy * (m1 * e2 + qxy) + qx * dc + hx * ((1.0f / 3.0f) * uxx + dv) + hy * ((-2.0f / 3.0f) * uyx + uxy);
    const T gy = dsx * cy + uy * (m7 * e1 + qyy) + ux * (m1 * e2 + qyx) + qy * dc + hy * ((1.0f / 3.0f) * uyy + dv) + hx * ((-2.0f / 3.0f) * uxy + uyx);
    fx = k * gx;
    fy = k * gy;
}

}  // namespace lbmv
