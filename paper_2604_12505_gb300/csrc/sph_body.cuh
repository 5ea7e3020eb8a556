// sph_body.cuh -- the rigid body's update (Eq. 20, kick then drift) as one warp
// computes it: everything that does not depend on the step's fluid force
// prepared before it is known, the update itself one FP64 FMA per output.
// Shared by the body kernel of a step and the resident kernel.
#pragma once

#include "sph_common.cuh"

namespace sph {

// The value at position `lane` of the list (0 past its end): nested selects,
// so the lanes of a warp pick different values without diverging.
__device__ __forceinline__ double pick(int, int) { return 0.0; }
template <class... R>
__device__ __forceinline__ double pick(int lane, int i, double x, R... rest)
{
    return lane == i ? x : pick(lane, i + 1, rest...);
}

__device__ __forceinline__ double sel3(int i, double a, double b, double c) { return i == 0 ? a : (i == 1 ? b : c); }

// Output l of the update is A + B F, F the component `comp` of (F_x, F_y,
// T_b): 0..5 r', theta', rdot', thetadot'; 6, 7 r' - W (the origin of the next
// grid); in an evaluation 0..5 are F_b, T_b and the accelerations of Eq. 20.
// Outputs 8 and 9 are cos and sin of the new angle, the old pair rotated by
// dtheta = dt thetadot' = Ad + Bd T_b.
struct BodyPlan {
    double A, B, Ad, Bd, X, Yr;
    int comp;
};

__device__ __forceinline__ BodyPlan body_plan(const TankDev& T, int lane, int eval, bool body_fixed, double rx, double ry,
                                              double th, double vx, double vy, double w, double c, double sn, double ux,
                                              double uy, double tau)
{
    BodyPlan P;
    const double dt = T.dt_d, im = T.inv_m_body, iJ = T.inv_J_body;
    const int comp = lane % 3;  // F_x, F_y or T_b for lanes 0..7 (0, 1, 2, 0, 1, 2, 0, 1)
    const int k = lane < 8 ? lane : 0;
    P.comp = comp;
    if (eval) {
        const double u3 = sel3(comp, ux, uy, tau), i3 = comp == 2 ? iJ : im;
        P.A = k < 3 ? 0.0 : u3 * i3;
        P.B = k < 3 ? 1.0 : i3;
    } else if (body_fixed) {
        P.A = pick(k, 0, rx, ry, th, vx, vy, w, rx - T.W, ry - T.W);
        P.B = 0.0;
    } else {
        const double x0 = sel3(comp, rx, ry, th), v0 = sel3(comp, vx, vy, w);
        const double u3 = sel3(comp, ux, uy, tau), i3 = comp == 2 ? iJ : im;
        const double Av = v0 + dt * (u3 * i3), Bv = dt * i3;  // velocity
        const bool vel = (k >= 3 && k <= 5);
        P.A = vel ? Av : x0 + dt * Av - (k >= 6 ? T.W : 0.0);
        P.B = vel ? Bv : dt * Bv;
    }
    // (cos, sin) first brought back to unit norm (off the dependent chain)
    P.Ad = P.Bd = 0.0;
    if (!eval && !body_fixed) {
        P.Ad = dt * (w + dt * (tau * iJ));
        P.Bd = dt * dt * iJ;
        const double f = 1.5 - 0.5 * (c * c + sn * sn);
        c *= f;
        sn *= f;
    }
    P.X = lane == 9 ? sn : c;  // lane 8: cos', lane 9: sin'
    P.Yr = lane == 9 ? c : -sn;
    return P;
}

// Out of line: a step turns the body by less than a hundredth of a radian.
static __device__ __noinline__ double2 cos_sin(double d)
{
    double s, c;
    sincos(d, &s, &c);
    return make_double2(c, s);
}

__device__ __forceinline__ double body_apply(const BodyPlan& P, int lane, int eval, bool body_fixed, double Fx, double Fy,
                                             double Tq)
{
    double v = fma(P.B, sel3(P.comp, Fx, Fy, Tq), P.A);
    if (!eval && !body_fixed) {
        const double d = fma(P.Bd, Tq, P.Ad), d2 = d * d;
        double cd, sd;
        if (fabs(d) <= 1e-4) {  // first omitted terms d^4 / 24, d^5 / 120 below 1e-16 relative
            cd = fma(-0.5, d2, 1.0);
            sd = fma(d * d2, -1.0 / 6.0, d);
        } else if (fabs(d) <= 1e-2) {
            cd = 1.0 - d2 * (0.5 - d2 * (1.0 / 24.0 - d2 * (1.0 / 720.0)));
            sd = d * (1.0 - d2 * (1.0 / 6.0 - d2 * (1.0 / 120.0 - d2 * (1.0 / 5040.0))));
        } else {
            const double2 cs = cos_sin(d);
            cd = cs.x;
            sd = cs.y;
        }
        if (lane == 8 || lane == 9) v = fma(P.X, cd, P.Yr * sd);
    } else if (lane == 8 || lane == 9) {
        v = P.X;  // unchanged angle
    }
    return v;
}

}  // namespace sph
