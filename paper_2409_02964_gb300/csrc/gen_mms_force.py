#!/usr/bin/env python3
"""Generate mms_force.cuh: the body force of Eq. (25) for the spatiotemporal
manufactured solution, evaluated inside the batched kernel.

Fields (lattice units, n x n periodic lattice, k = 2 pi / n, w = 2 pi / T):
    phi = phi0 + A sin(kx) sin(ky) cos(wt)
    q = phi u = grad psi + rot Psi,  psi = -(A w sin(wt) / (2 k^2)) sin(kx) sin(ky),
                                     Psi = (U0 / k) sin(kx) sin(ky)
so that d_t phi + div q = 0 with rho = rho0; the force is Eq. (25) with the pressure
term dropped (constant density):
    F / rho0 = d_t q + div(q u) - nu div(phi tau),  tau = grad u + grad u^T - (2/3) div u I.

The emitted code evaluates this in a structured way rather than as one expanded
rational expression: phi and q with their first and second derivatives are short
products of sin/cos of kx, ky (the arguments sx, cx, sy, cy) with step constants;
u = q / phi and its derivatives follow from the quotient rule with one reciprocal;
the force is then assembled from those. At generation time the structured result
is checked against the direct symbolic derivation (sympy) at random points.

Run from this directory:  python gen_mms_force.py  (needs sympy; the generated
header is committed, so building the library does not).
"""
import os
import random

import sympy as sp


def direct_force():
    """Eq. (25) by symbolic differentiation of the fields (the reference form)."""
    x, y, t = sp.symbols("x y t", real=True)
    k, w, A, U0, phi0, nu = sp.symbols("k w A U0 phi0 nu", positive=True)
    s_x, s_y, c_x, c_y = sp.sin(k * x), sp.sin(k * y), sp.cos(k * x), sp.cos(k * y)
    phi = phi0 + A * s_x * s_y * sp.cos(w * t)
    b = -(A * w / (2 * k)) * sp.sin(w * t)
    qx = b * c_x * s_y + U0 * s_x * c_y
    qy = b * s_x * c_y - U0 * c_x * s_y
    ux, uy = qx / phi, qy / phi
    div = sp.diff(ux, x) + sp.diff(uy, y)
    txx = 2 * sp.diff(ux, x) - sp.Rational(2, 3) * div
    tyy = 2 * sp.diff(uy, y) - sp.Rational(2, 3) * div
    txy = sp.diff(ux, y) + sp.diff(uy, x)
    Fx = sp.diff(qx, t) + sp.diff(qx * ux, x) + sp.diff(qx * uy, y) - nu * (sp.diff(phi * txx, x) + sp.diff(phi * txy, y))
    Fy = sp.diff(qy, t) + sp.diff(qy * ux, x) + sp.diff(qy * uy, y) - nu * (sp.diff(phi * txy, x) + sp.diff(phi * tyy, y))
    return (x, y, t, k, w, A, U0, phi0, nu), Fx, Fy


# The structured evaluation: (name, kind, expression text). kind "s" = float scalar
# (uniform per lattice and step), "v" = per-cell value of type T. Expressions use the
# inputs sx, cx, sy, cy (T), ct, st, k, w, A, U0, phi0, nu (float) and earlier names.
#
# Derivatives here are with respect to kx and ky (a factor k each, restored at the end).
# With phi tau_ij = d_j q_i + d_i q_j - u_i d_j phi - u_j d_i phi - (2/3)(div q - u . grad
# phi) delta_ij the divergence holds no second derivative of u:
#   div(phi tau)_x = lap q_x + (1/3) d_x div q - (7/3) u_x phi_xx - (1/3) u_y phi_xy
#                    - ((1/3) u_x,x + div u) phi_x - (u_x,y - (2/3) u_y,x) phi_y
# (phi_xx = phi_yy, lap q = -2 q, div q = -2 b sin sin), 53 packed operations a cell pair
# against 170. Every line is a sum of products, each one fused operation; the first group
# of "v" lines depends on the column only and is formed once per strip.
STEPS = [
    # step constants
    ("a", "s", "A * ct"),                        # phi = phi0 + a sx sy
    ("b", "s", "-(A * w * st) / (2 * k)"),       # q_x = b cx sy + U0 sx cy, q_y = b sx cy - U0 cx sy
    ("bt", "s", "-(A * w * w * ct) / (2 * k)"),  # d_t b
    ("n1", "s", "nu * k"),
    ("c1", "s", "bt / k + (2.0 / 3.0) * n1 * b"),
    ("c2", "s", "2 * n1"),
    ("m7", "s", "-(7.0 / 3.0) * n1"),
    ("m1", "s", "(1.0 / 3.0) * n1"),
    # of the column
    ("asx", "v", "a * sx"),
    ("acx", "v", "a * cx"),
    ("nasx", "v", "(-a) * sx"),
    ("nacx", "v", "(-a) * cx"),
    ("bsx", "v", "b * sx"),
    ("bcx", "v", "b * cx"),
    ("nbsx", "v", "(-b) * sx"),
    ("usx", "v", "U0 * sx"),
    ("ucx", "v", "U0 * cx"),
    ("nusx", "v", "(-U0) * sx"),
    ("nucx", "v", "(-U0) * cx"),
    ("dsx", "v", "c1 * sx"),
    ("dcx", "v", "c1 * cx"),
    # phi and its derivatives (npx = -phi_x, e1 = -phi_xx = -phi_yy, e2 = phi_xy)
    ("e1", "v", "asx * sy"),
    ("e2", "v", "acx * cy"),
    ("ph", "v", "asx * sy + phi0"),
    ("npx", "v", "nacx * sy"),
    ("npy", "v", "nasx * cy"),
    # q and its derivatives
    ("qx", "v", "bcx * sy + usx * cy"),
    ("qy", "v", "bsx * cy + nucx * sy"),
    ("nbss", "v", "nbsx * sy"),
    ("bcc", "v", "bcx * cy"),
    ("qxx", "v", "ucx * cy + nbss"),            # d_x q_x
    ("qyy", "v", "nucx * cy + nbss"),           # d_y q_y
    ("qxy", "v", "nusx * sy + bcc"),            # d_y q_x
    ("qyx", "v", "usx * sy + bcc"),             # d_x q_y
    # u = q / phi and its derivatives (quotient rule)
    ("ip", "v", "1 / ph"),
    ("ux", "v", "qx * ip"),
    ("uy", "v", "qy * ip"),
    ("uxx", "v", "(ux * npx + qxx) * ip"),
    ("uxy", "v", "(ux * npy + qxy) * ip"),
    ("uyx", "v", "(uy * npx + qyx) * ip"),
    ("uyy", "v", "(uy * npy + qyy) * ip"),
    ("dv", "v", "uxx + uyy"),
    ("dc", "v", "dv + c2"),
    ("hx", "v", "(-n1) * npx"),
    ("hy", "v", "(-n1) * npy"),
    # Eq. (25) without the pressure term, per unit rho0
    ("gx", "v", "dcx * sy + ux * (m7 * e1 + qxx) + uy * (m1 * e2 + qxy) + qx * dc"
                " + hx * ((1.0 / 3.0) * uxx + dv) + hy * ((-2.0 / 3.0) * uyx + uxy)"),
    ("gy", "v", "dsx * cy + uy * (m7 * e1 + qyy) + ux * (m1 * e2 + qyx) + qy * dc"
                " + hy * ((1.0 / 3.0) * uyy + dv) + hx * ((-2.0 / 3.0) * uxy + uyx)"),
    ("fx", "out", "k * gx"),
    ("fy", "out", "k * gy"),
]

INPUTS_V = ("sx", "cx", "sy", "cy")
INPUTS_S = ("ct", "st", "k", "w", "A", "U0", "phi0", "nu")


def check_against_direct(trials: int = 12) -> float:
    """Largest relative difference between the structured and the direct force."""
    syms, Fx, Fy = direct_force()
    x, y, t, k, w, A, U0, phi0, nu = syms
    rng = random.Random(2409)
    worst = 0.0
    for _ in range(trials):
        vals = {k: 2 * 3.141592653589793 / rng.choice([16, 32, 48, 64]), w: 2 * 3.141592653589793 / rng.uniform(200, 3000),
                A: rng.uniform(0.05, 0.3), U0: rng.uniform(0.0, 0.02), phi0: 0.7, nu: rng.uniform(0.02, 0.3),
                x: rng.uniform(0, 64), y: rng.uniform(0, 64), t: rng.uniform(0, 5000)}
        ref = [sp.N(F.subs(vals), 30) for F in (Fx, Fy)]
        env = {"sx": sp.sin(vals[k] * vals[x]), "cx": sp.cos(vals[k] * vals[x]), "sy": sp.sin(vals[k] * vals[y]),
               "cy": sp.cos(vals[k] * vals[y]), "ct": sp.cos(vals[w] * vals[t]), "st": sp.sin(vals[w] * vals[t]),
               "k": vals[k], "w": vals[w], "A": vals[A], "U0": vals[U0], "phi0": vals[phi0], "nu": vals[nu]}
        for name, _, expr in STEPS:
            env[name] = sp.N(sp.sympify(expr, locals=dict(env)), 30)
        scale = max(abs(r) for r in ref) or 1
        for got, want in zip((env["fx"], env["fy"]), ref):
            worst = max(worst, float(abs(got - want) / scale))
    return worst


def emit(expr: str, kind: str) -> str:
    """C++ text: numbers as float literals, 1 / T as mms_rcp(T)."""
    import re
    text = expr.replace("1 / ph", "mms_rcp(ph)")
    text = re.sub(r"(?<![\w.])(\d+\.\d+|\d+)(?![\w.])", lambda m: f"{float(m.group(1))!r}f", text)
    return text


def main() -> None:
    err = check_against_direct()
    assert err < 1e-12, f"structured force differs from the direct derivation by {err}"
    lines = []
    for name, kind, expr in STEPS:
        if kind == "s":
            lines.append(f"    const float {name} = {emit(expr, kind)};")
        elif kind == "v":
            lines.append(f"    const T {name} = {emit(expr, kind)};")
        else:
            lines.append(f"    {name} = {emit(expr, kind)};")
    body = "\n".join(lines)
    text = f'''// mms_force.cuh -- GENERATED by gen_mms_force.py; do not edit by hand.
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

namespace lbmv {{

template <typename T>
__device__ __forceinline__ void mms_force(T sx, T cx, T sy, T cy, float ct, float st, float k, float w, float A,
                                          float U0, float phi0, float nu, T& fx, T& fy) {{
{body}
}}

}}  // namespace lbmv
'''
    out = os.path.join(os.path.dirname(os.path.abspath(__file__)), "mms_force.cuh")
    with open(out, "w") as fh:
        fh.write(text)
    print(out, f"{len(STEPS)} steps, structured vs direct: {err:.1e}")


if __name__ == "__main__":
    main()
