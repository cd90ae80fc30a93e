// Fused time-step kernel of the axisymmetric thermal cascaded LB method
// (arXiv 1806.10241) for sm_103a, plus the field, diagnostic and
// import/export kernels.
//
// Data layout (per lattice, per buffer): 19 planes [q][z][pitch] of the
// storage type: f0..f8, g0..g4, h0..h4 in the velocity order of Eq. 10 and
// Eq. 28.  f and h are stored as deviations from the rest state (w_a rho0,
// w_a T0), g as is, all multiplied by `scale` (1 except for FP16).
//
// Kernels: the FP32 / 16-bit step on column pairs (lb_pair.cuh: one launch per
// step, rows marched by a warp; lb_tile.cuh: several steps per launch on tiles
// in shared memory) and the FP64 step (k_step64), which share the node update of
// lb_node.cuh, the pre-collision fields and the diagnostics (block_fields), and
// the exchange with the host.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <functional>
#include <queue>
#include <type_traits>
#include <vector>

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "../../include/lb.h"
#include "lb_internal.h"
#include "lb_rcp.cuh"

namespace lbk {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kMaxSmem = 227 * 1024;  // dynamic shared memory of a block
constexpr int kSmemPerSm = 228 * 1024;  // of an SM, 1 KB of it taken per block by the system

// ---- storage conversions ------------------------------------------------

template <typename S, typename C> struct Cvt;
template <> struct Cvt<double, double> {
    static __device__ __forceinline__ double cv(double x) { return x; }
    static __device__ __forceinline__ double ld(const double *p) { return *p; }
    static __device__ __forceinline__ void st(double *p, double v) { *p = v; }
};
template <> struct Cvt<float, float> {
    static __device__ __forceinline__ float cv(float x) { return x; }
    static __device__ __forceinline__ float ld(const float *p) { return *p; }
    static __device__ __forceinline__ void st(float *p, float v) { *p = v; }
};
template <> struct Cvt<__nv_bfloat16, float> {
    static __device__ __forceinline__ float cv(__nv_bfloat16 x) { return __bfloat162float(x); }
    static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void st(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};
template <> struct Cvt<__half, float> {
    static __device__ __forceinline__ float cv(__half x) { return __half2float(x); }
    static __device__ __forceinline__ float ld(const __half *p) { return __half2float(*p); }
    static __device__ __forceinline__ void st(__half *p, float v) { *p = __float2half_rn(v); }
};

// 1/x: the hardware reciprocal for FP32 (|error| <= 2 ulp, far inside the
// FP32 parity tolerances), a correctly rounded division for FP64
__device__ __forceinline__ float rcp(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }

// FP16 storage is scaled (deviations x 1024, away from the subnormal range);
// the other storage types are not, and skip the multiplications.
template <typename S> struct Scaled { static constexpr bool value = std::is_same<S, __half>::value; };

// ---- kernel parameters in the compute type --------------------------------

#include "lb_node.cuh"

template <typename C> struct KP {
    int nr, nz, pitch, xper;
    long long plane;
    double r0;
    C om3, om4, omhi, omg, omh;
    C nu, alpha, gbeta, T0, bfx, rho0;
    int planar, sign_lit, explicit_src;
    // sides 0..3; entry 4 the outer segment of a split top (a copy of the top
    // when the top is one segment): columns >= top_split of the top follow it
    int flow[5], swirl[5], heat[5];
    C uwx[5], uwy[5], omega[5], Tw[5];
    int top_split;
    C ramp0, ramp1;       // wall temperature ramp of entry 4: T_w(y) = ramp0 + ramp1 y
    C scale, inv_scale;
    C r0c, roc;           // inner and outer wall radii, rounded once
    // Lateral walls (sides 2 and 3), computed once in the kernel's precision
    // with the operations the per-row rules would do (pair kernels): latf, the
    // moving-wall terms of the populations entering from the wall (f2, f5, f6
    // at the inner side, f4, f7, f8 at the outer); (latgs, latgc) and
    // (laths, lathc), the sign and constant of the scalar rule of g and h,
    // x = s x_own + c; (gha, ghb), the ghost values a q + b of u_x, u_y,
    // u_theta and T for the central differences.
    C latf[2][3], latgs[2], latgc[2], laths[2], lathc[2], gha[2][4], ghb[2][4];
    const float *ytab;    // y[pitch] then 1/y[pitch] (pair kernels)
    NodeConst<typename std::conditional<std::is_same<C, float>::value, float2, C>::type> pc;
    // Nusselt and equivalent-conductivity scales per side (diagnostics)
    double nu_scale[4], keq_scale[4];
    int pinned;           // pinned_order
};

// A lattice whose geometric sources amplify disturbances (see update_pinned):
// a diffusivity above 3 radii of its innermost node.
bool pinned_order(const HostParams &h)
{
    return h.storage != ST_FP64 && !h.planar && std::max(h.nu, h.alpha) > 3.0 * (h.r0 + 0.5);
}

template <typename C> KP<C> make_kp(const HostParams &h)
{
    KP<C> k;
    k.nr = h.nr;
    k.nz = h.nz;
    k.pitch = h.pitch;
    k.plane = h.plane;
    k.xper = h.flow[0] == 2;
    k.r0 = h.r0;
    const double omn = 1.0 / (3.0 * h.nu + 0.5), oma = 1.0 / (3.0 * h.alpha + 0.5);
    k.om3 = (C)h.omega3;
    k.om4 = (C)omn;
    k.omhi = (C)h.omega_hi;
    k.omg = (C)omn;
    k.omh = (C)oma;
    k.nu = (C)h.nu;
    k.alpha = (C)h.alpha;
    k.gbeta = (C)h.g_beta;
    k.T0 = (C)h.T0;
    k.bfx = (C)h.body_fx;
    k.rho0 = (C)h.rho0;
    k.planar = h.planar;
    k.sign_lit = h.sign_literal;
    k.explicit_src = h.explicit_sources;
    k.pinned = pinned_order(h);
    for (int s = 0; s < 5; ++s) {
        k.flow[s] = h.flow[s];
        k.swirl[s] = h.swirl[s];
        k.heat[s] = h.heat[s];
        k.uwx[s] = (C)h.uwx[s];
        k.uwy[s] = (C)h.uwy[s];
        k.omega[s] = (C)h.omega[s];
        k.Tw[s] = (C)h.Tw[s];
    }
    k.top_split = h.top_split;
    {  // Sec. 3.6 surface temperature: linear in r from the top's T_w at the
       // split radius to the outer segment's T_w at the outer wall
        const double rs = h.r0 + h.top_split, ro = h.r0 + h.nr;
        const double slope = h.top_split > 0 ? (h.Tw[4] - h.Tw[1]) / (ro - rs) : 0.0;
        k.ramp0 = (C)(h.Tw[1] - slope * rs);
        k.ramp1 = (C)slope;
    }
    k.scale = (C)h.scale;
    k.inv_scale = (C)(1.0 / h.scale);
    k.r0c = (C)h.r0;
    k.roc = (C)(h.r0 + h.nr);
    for (int j = 0; j < 2; ++j) {
        const int sd = 2 + j;
        const C rw = k.rho0, ux = k.uwx[sd], uy = k.uwy[sd], radius = j == 0 ? k.r0c : k.roc;
        const C c9 = (C)(6.0 / 9.0), c36 = (C)(6.0 / 36.0), two = (C)2;
        if (j == 0) {  // Sec. 3.1 moving wall (R11) at the inner side
            k.latf[0][0] = rw * c9 * uy;
            k.latf[0][1] = rw * c36 * (ux + uy);
            k.latf[0][2] = rw * c36 * (-ux + uy);
        } else {
            k.latf[1][0] = rw * c9 * (-uy);
            k.latf[1][1] = rw * c36 * (-ux - uy);
            k.latf[1][2] = rw * c36 * (ux - uy);
        }
        // scalar rules (R12, R13): Dirichlet -x + (2/6) w, odd axis -x, else x
        const C psi_w = k.rho0 * k.omega[sd] * radius, t_w = k.Tw[sd] - k.T0;
        k.latgs[j] = (C)(k.swirl[sd] == 0 || k.swirl[sd] == 2 ? -1 : 1);
        k.latgc[j] = k.swirl[sd] == 0 ? (C)(2.0 / 6.0) * psi_w : (C)0;
        k.laths[j] = (C)(k.heat[sd] == 0 ? -1 : 1);
        k.lathc[j] = k.heat[sd] == 0 ? (C)(2.0 / 6.0) * t_w : (C)0;
        // ghosts (R7): wall 2 q_w - q, zero flux q, axis u_x, T even, u_y, u_theta odd
        const bool axis = k.flow[sd] == 1;
        k.gha[j][0] = (C)(axis ? 1 : -1);
        k.ghb[j][0] = axis ? (C)0 : two * ux;
        k.gha[j][1] = (C)-1;
        k.ghb[j][1] = axis ? (C)0 : two * uy;
        k.gha[j][2] = (C)(k.swirl[sd] == 0 || k.swirl[sd] == 2 ? -1 : 1);
        k.ghb[j][2] = k.swirl[sd] == 0 ? two * k.omega[sd] * radius : (C)0;
        k.gha[j][3] = (C)(k.heat[sd] == 0 ? -1 : 1);
        k.ghb[j][3] = k.heat[sd] == 0 ? two * k.Tw[sd] : (C)0;
    }
    k.ytab = h.ytab;
    {
        const C osc = (C)h.scale, om3 = k.om3, om4 = k.om4, omh = k.omhi, third = (C)1 / (C)3, ninth = (C)1 / (C)9;
        auto e = [](C v) {
            if constexpr (std::is_same<C, float>::value) return make_float2(v, v);
            else return v;
        };
        auto &c = k.pc;
        c.rho0 = e(k.rho0), c.T0 = e(k.T0), c.bfx = e(k.bfx), c.fb = e(k.rho0 * k.gbeta);
        c.nu = e(k.nu), c.nuh = e((C)0.5 * k.nu), c.alh = e((C)0.5 * k.alpha), c.k3 = e(k.rho0 * third);
        c.c3 = e(om3 * ((C)1 / (C)12) * osc), c.c4 = e(om4 * (C)0.25 * osc), c.nc4 = e(om4 * (C)-0.25 * osc);
        c.ch = e(omh * (C)0.25 * osc), c.nch = e(omh * (C)-0.25 * osc);
        c.cg = e(k.omg * (C)0.5 * osc), c.ct = e(k.omh * (C)0.5 * osc);
        c.m9 = e(ninth * osc), c.m6 = e((C)1 / (C)6 * osc), c.m5 = e((C)0.2 * osc);
        c.sg = e((C)(h.sign_literal ? -1 : 1)), c.os = e(osc), c.one = e((C)1), c.mone = e((C)-1);
    }
    // Nusselt normalisation (Sec. 3.2): lateral walls -R_w / (H dT), end
    // walls -(H / dT) * 2 / (R_o^2 - R_i^2); dT from the Dirichlet values.
    double tmin = 0, tmax = 0;
    int nd = 0;
    for (int s = 0; s < 5; ++s)
        if ((h.heat[s] == 0 || h.heat[s] == 4) && (s < 4 || h.top_split > 0)) {
            if (nd == 0 || h.Tw[s] < tmin) tmin = h.Tw[s];
            if (nd == 0 || h.Tw[s] > tmax) tmax = h.Tw[s];
            ++nd;
        }
    const double dT = (nd >= 2 && tmax > tmin) ? tmax - tmin : 1.0;
    const double H = h.nz, Ri = h.r0, Ro = h.r0 + h.nr;
    k.nu_scale[0] = k.nu_scale[1] = -(H / dT) * 2.0 / (Ro * Ro - Ri * Ri);
    k.nu_scale[2] = -Ri / (H * dT);
    k.nu_scale[3] = -Ro / (H * dT);
    // mean equivalent conductivity of a lateral wall of an annulus (Sec. 3.5):
    // ln(R_o / R_i) / (H dT) times the sum over z of -R_w dT/dr
    const double lg = Ri > 0.0 ? std::log(Ro / Ri) : 0.0;
    k.keq_scale[0] = k.keq_scale[1] = 0.0;
    k.keq_scale[2] = -Ri * lg / (H * dT);
    k.keq_scale[3] = -Ro * lg / (H * dT);
    return k;
}

// ---- per-row helpers -------------------------------------------------------

template <typename C> struct PM {  // macroscopic fields of the stored state
    C rd, ux, uy, ut, T;
};

template <typename S, typename C> __device__ __forceinline__ PM<C> moments(const C v[NQ], const KP<C> &k)
{
    // rho = rho0 + sum f_dev, j = sum f_dev e, psi = sum g, T = T0 + sum h_dev
    C rd = v[0] + v[1] + v[2] + v[3] + v[4] + v[5] + v[6] + v[7] + v[8];
    C jx = v[1] - v[3] + v[5] - v[6] - v[7] + v[8];
    C jy = v[2] - v[4] + v[5] + v[6] - v[7] - v[8];
    C ps = v[9] + v[10] + v[11] + v[12] + v[13];
    C td = v[14] + v[15] + v[16] + v[17] + v[18];
    if (Scaled<S>::value) {
        const C is = k.inv_scale;
        rd *= is;
        jx *= is;
        jy *= is;
        ps *= is;
        td *= is;
    }
    const C ir = rcp(k.rho0 + rd);
    PM<C> m;
    m.rd = rd;
    m.ux = jx * ir;
    m.uy = jy * ir;
    m.ut = ps * ir;
    m.T = k.T0 + td;
    return m;
}

template <typename S, typename C>
__device__ __forceinline__ void load_row(const S *__restrict__ src, const KP<C> &k, int row, int col,
                                         C v[NQ])
{
    const S *p = src + (long long)row * k.pitch + col;
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = Cvt<S, C>::ld(p + q * k.plane);
}

template <typename S, typename C>
__device__ __forceinline__ C own(const S *__restrict__ src, const KP<C> &k, int q, int row, int col)
{
    return Cvt<S, C>::ld(src + q * k.plane + (long long)row * k.pitch + col);
}

// psi on a rotating wall: rho0 * omega * radius (side 4: the top's outer segment)
template <typename C> __device__ __forceinline__ C wall_psi(const KP<C> &k, int side, C y)
{
    const C radius = (side <= 1 || side == 4) ? y : (side == 2 ? k.r0c : k.roc);
    return k.rho0 * k.omega[side] * radius;
}

// the entry of an end wall at column col: the top's outer segment (4) for
// columns >= top_split of a split top, else the side itself
template <typename C> __device__ __forceinline__ int end_seg(const KP<C> &k, int side, int col)
{
    return (side == 1 && k.top_split > 0 && col >= k.top_split) ? 4 : side;
}

// wall temperature of an end-wall entry at the column radius y (the ramp of
// Sec. 3.6 on entry 4 with heat type 4), and the entry's h rule with the ramp
// read as Dirichlet
template <typename C> __device__ __forceinline__ C end_T(const KP<C> &k, int seg, C y)
{
    return k.heat[seg] == 4 ? k.ramp0 + k.ramp1 * y : k.Tw[seg];
}
template <typename C> __device__ __forceinline__ int heat_rule(const KP<C> &k, int seg)
{
    return k.heat[seg] == 4 ? 0 : k.heat[seg];
}
// a side whose wall temperatures enter its Nusselt number (Sec. 3.2): a
// Dirichlet side, or a top any of whose segments holds a wall temperature
template <typename C> __device__ __forceinline__ bool wall_heated(const KP<C> &k, int sd)
{
    if (sd == 1 && k.top_split > 0) return k.heat[1] == 0 || k.heat[4] == 0 || k.heat[4] == 4;
    return k.heat[sd] == 0;
}

// Scalar boundary value for the population entering from a wall (Sec. 3):
// Dirichlet anti-bounce-back -x_own + 2 w s_w (w = 1/6, deviation form for h),
// Neumann / even axis bounce-back x_own, odd axis (psi) -x_own.
template <typename C>
__device__ __forceinline__ C scalar_bc(int bc, C own_v, C wall_dev_scaled, bool odd_axis)
{
    if (bc == 0) return -own_v + (C)(2.0 / 6.0) * wall_dev_scaled;
    if (bc == 2 && odd_axis) return -own_v;
    return own_v;
}

// ---- the node update -------------------------------------------------------

template <typename C> struct NodeOut {
    C f[9], g[5], h[5];
    C rho, ux, uy, ut, T;  // pre-collision fields
};

// Pulled (deviation, unscaled) values in fv/gv/hv; gradient inputs.
template <typename C>
__device__ __forceinline__ void update_node(const KP<C> &k, C y, C iy, C fv[9], C gv[5], C hv[5],
                                            C dxuy, C dyux, C dyuy, C dyut, C dyT, NodeOut<C> &o)
{
    // output moments, Eq. 18, 35, 47 (deviation form: rest parts cancel)
    const C rdo = fv[0] + fv[1] + fv[2] + fv[3] + fv[4] + fv[5] + fv[6] + fv[7] + fv[8];
    const C jxo = fv[1] - fv[3] + fv[5] - fv[6] - fv[7] + fv[8];
    const C jyo = fv[2] - fv[4] + fv[5] + fv[6] - fv[7] - fv[8];
    const C pso = gv[0] + gv[1] + gv[2] + gv[3] + gv[4];
    const C tdo = hv[0] + hv[1] + hv[2] + hv[3] + hv[4];

    // sources (Eq. 4a-4c, 5, 7, 9) at the pre-collision state, two sweeps.
    // Written per unit of the swept state (rd, j, psi, td): with mu = rho nu,
    //   F_x^A = -j_x u_y / y + rho nu (d_x u_y + d_y u_x) / y
    //   F_y^A = psi^2 / (rho y) - j_y u_y / y + rho 2 nu d_y u_y / y - 2 nu j_y / y^2
    //   S_psi = -2 u_y psi / y + rho nu d_y u_theta / y - nu psi / y^2
    //   S_phi = -u_y T / y + alpha d_y T / y
    // so the gradient factors are formed once per node.
    C rd = rdo, jx = jxo, jy = jyo, ps = pso, td = tdo;
    C MA = 0, Fx = 0, Fy = 0, Sps = 0, Sph = 0;
    const bool geo = !k.planar;
    const C Gx = geo ? k.nu * (dxuy + dyux) * iy : (C)0;
    const C Gy = geo ? (C)2 * k.nu * dyuy * iy : (C)0;
    const C Gw = geo ? k.nu * dyut * iy : (C)0;
    const C Gt = geo ? k.alpha * dyT * iy : (C)0;
    const C iy2nu = geo ? k.nu * iy * iy : (C)0;
    const C gy = geo ? iy : (C)0;
    const C Fb = k.rho0 * k.gbeta;
    const int sweeps = k.explicit_src ? 1 : 2;
    for (int sw = 0; sw < sweeps; ++sw) {
        const C r = k.rho0 + rd, ir = rcp(r);
        const C uyy = jy * ir * gy;  // u_y / y
        const C ph = k.T0 + td;
        const C FAx = -jx * uyy + r * Gx;
        const C FAy = (ps * ps - jy * jy) * ir * gy + r * Gy - (C)2 * jy * iy2nu;
        Sps = (C)-2 * uyy * ps + r * Gw - iy2nu * ps;
        Sph = -uyy * ph + Gt;
        Fx = FAx + Fb * td + k.bfx;
        Fy = FAy;
        jx = jxo + (C)0.5 * Fx;
        jy = jyo + (C)0.5 * Fy;
        ps = pso + (C)0.5 * Sps;
        td = tdo + (C)0.5 * Sph;
        // M^A = -j_y / y, from the newest momentum (from the output momentum
        // in the single-evaluation mode)
        MA = -(k.explicit_src ? jyo : jy) * gy;
        rd = rdo + (C)0.5 * MA;
    }
    const C r = k.rho0 + rd, ir = rcp(r);
    const C ux = jx * ir, uy = jy * ir;
    const C phi = k.T0 + td;
    o.rho = r;
    o.ux = ux;
    o.uy = uy;
    o.ut = ps * ir;
    o.T = phi;

    // D2Q9 cascaded collision, Eq. 17 (raw moments of the streamed f; the
    // rest-state parts rho0/3, rho0/9 written out)
    const C third = (C)(1.0 / 3.0);
    const C Dxx = fv[1] + fv[3] + fv[5] + fv[6] + fv[7] + fv[8];
    const C Dyy = fv[2] + fv[4] + fv[5] + fv[6] + fv[7] + fv[8];
    const C Dxy = fv[5] - fv[6] + fv[7] - fv[8];
    const C Dxxy = fv[5] + fv[6] - fv[7] - fv[8];
    const C Dxyy = fv[5] - fv[6] - fv[7] + fv[8];
    const C Dxxyy = fv[5] + fv[6] + fv[7] + fv[8];
    const C Kxx = k.rho0 * third + Dxx, Kyy = k.rho0 * third + Dyy;
    const C ux2 = ux * ux, uy2 = uy * uy, uxy = ux * uy;
    const C p3 = k.om3 * (C)(1.0 / 12.0) * ((C)(2.0 / 3.0) * rd + r * (ux2 + uy2) - (Dxx + Dyy));
    const C p4 = k.om4 * (C)0.25 * (r * (ux2 - uy2) - (Dxx - Dyy));
    const C p5 = k.om4 * (C)0.25 * (r * uxy - Dxy);
    const C q34p = (C)3 * p3 + p4, q34m = (C)3 * p3 - p4;
    const C p6 = k.omhi * (C)0.25 * ((C)2 * r * ux2 * uy + Dxxy - (C)2 * ux * Dxy - uy * Kxx)
                 - (C)0.5 * uy * q34p - (C)2 * ux * p5;
    const C p7 = k.omhi * (C)0.25 * ((C)2 * r * ux * uy2 + Dxyy - (C)2 * uy * Dxy - ux * Kyy)
                 - (C)0.5 * ux * q34m - (C)2 * uy * p5;
    const C p8 = k.omhi * (C)0.25 *
                     (rd * (C)(1.0 / 9.0) + (C)3 * r * ux2 * uy2 -
                      (Dxxyy - (C)2 * ux * Dxyy - (C)2 * uy * Dxxy + ux2 * Kyy + uy2 * Kxx + (C)4 * uxy * Dxy)) -
                 (C)2 * p3 - (C)0.5 * uy2 * q34p - (C)0.5 * ux2 * q34m - (C)4 * uxy * p5 - (C)2 * uy * p6 -
                 (C)2 * ux * p7;
    // source moments, Eq. 26
    const C p0 = MA * (C)(1.0 / 9.0), p1 = Fx * (C)(1.0 / 6.0), p2 = Fy * (C)(1.0 / 6.0);
    // back-transform, Eq. 27
    o.f[0] = fv[0] + (p0 - (C)4 * (p3 - p8));
    o.f[1] = fv[1] + (p0 + p1 - p3 + p4 + (C)2 * (p7 - p8));
    o.f[2] = fv[2] + (p0 + p2 - p3 - p4 + (C)2 * (p6 - p8));
    o.f[3] = fv[3] + (p0 - p1 - p3 + p4 - (C)2 * (p7 + p8));
    o.f[4] = fv[4] + (p0 - p2 - p3 - p4 - (C)2 * (p6 + p8));
    o.f[5] = fv[5] + (p0 + p1 + p2 + (C)2 * p3 + p5 - p6 - p7 + p8);
    o.f[6] = fv[6] + (p0 - p1 + p2 + (C)2 * p3 - p5 - p6 + p7 + p8);
    o.f[7] = fv[7] + (p0 - p1 - p2 + (C)2 * p3 + p5 + p6 + p7 + p8);
    o.f[8] = fv[8] + (p0 + p1 - p2 + (C)2 * p3 - p5 + p6 - p7 + p8);

    // D2Q5 cascaded collisions, Eq. 34 (psi) and Eq. 49 (T), with the sign
    // that makes the equilibrium a fixed point unless sign_lit is set
    const C sg = k.sign_lit ? (C)1 : (C)-1;
    const C uu = ux2 + uy2, ud = ux2 - uy2;
    {
        const C kx = gv[1] - gv[3], ky = gv[2] - gv[4];
        const C kxx = gv[1] + gv[3], kyy = gv[2] + gv[4];
        const C q1 = k.omg * (C)0.5 * (ps * ux - kx);
        const C q2 = k.omg * (C)0.5 * (ps * uy - ky);
        const C q3 = k.omhi * (C)0.25 * ((C)(2.0 / 3.0) * ps - (kxx + kyy) + (C)2 * (ux * kx + uy * ky) + sg * uu * ps)
                     + ux * q1 + uy * q2;
        const C q4 = k.omhi * (C)0.25 * (-(kxx - kyy) + (C)2 * (ux * kx - uy * ky) + sg * ud * ps) + ux * q1 - uy * q2;
        const C q0 = Sps * (C)0.2;  // Eq. 41
        // Eq. 42
        o.g[0] = gv[0] + (q0 - (C)4 * q3);
        o.g[1] = gv[1] + (q0 + q1 + q3 + q4);
        o.g[2] = gv[2] + (q0 + q2 + q3 - q4);
        o.g[3] = gv[3] + (q0 - q1 + q3 + q4);
        o.g[4] = gv[4] + (q0 - q2 + q3 - q4);
    }
    {
        const C kx = hv[1] - hv[3], ky = hv[2] - hv[4];
        const C Hxx = hv[1] + hv[3], Hyy = hv[2] + hv[4];
        const C r1 = k.omh * (C)0.5 * (phi * ux - kx);
        const C r2 = k.omh * (C)0.5 * (phi * uy - ky);
        const C r3 = k.omhi * (C)0.25 * ((C)(2.0 / 3.0) * td - (Hxx + Hyy) + (C)2 * (ux * kx + uy * ky) + sg * uu * phi)
                     + ux * r1 + uy * r2;
        const C r4 = k.omhi * (C)0.25 * (-(Hxx - Hyy) + (C)2 * (ux * kx - uy * ky) + sg * ud * phi) + ux * r1 - uy * r2;
        const C r0 = Sph * (C)0.2;  // Eq. 51
        // Eq. 52
        o.h[0] = hv[0] + (r0 - (C)4 * r3);
        o.h[1] = hv[1] + (r0 + r1 + r3 + r4);
        o.h[2] = hv[2] + (r0 + r2 + r3 - r4);
        o.h[3] = hv[3] + (r0 - r1 + r3 + r4);
        o.h[4] = hv[4] + (r0 - r2 + r3 - r4);
    }
}

// ---- scalar wall rules ----------------------------------------------------------

// Wall and axis rules (Sec. 3) on the pulled values of node (i, cl), in units
// of the storage scale sc; the own stored values are read from src.
template <typename S, typename C>
__device__ __forceinline__ void wall_rules1(const KP<C> &k, const S *__restrict__ src, int i, int cl, bool at_c0,
                                            bool at_cN, bool has_m, bool has_p, C y, C sc, C fv[9], C gv[5], C hv[5])
{
    const int nr = k.nr, nz = k.nz;
    // lateral boundaries (Sec. 3): the population entering from r < r0 or
    // r > r0 + nr is rebuilt from the node's own stored values
    {
        if (at_c0) {
            const int sd = 2;
            const C rw = k.rho0 * sc;
            if (k.flow[sd] == 1) {  // axis: mirror images
                fv[2] = own<S, C>(src, k, 4, i, 0);
                if (has_m) fv[5] = own<S, C>(src, k, 8, i > 0 ? i - 1 : nz - 1, 0);
                if (has_p) fv[6] = own<S, C>(src, k, 7, i + 1 < nz ? i + 1 : 0, 0);
            } else {  // wall: bounce-back + moving-wall term 6 w rho0 (e.u_w)
                const C ux_w = k.uwx[sd], uy_w = k.uwy[sd];
                fv[2] = own<S, C>(src, k, 4, i, 0) + rw * (C)(6.0 / 9.0) * uy_w;
                fv[5] = own<S, C>(src, k, 7, i, 0) + rw * (C)(6.0 / 36.0) * (ux_w + uy_w);
                fv[6] = own<S, C>(src, k, 8, i, 0) + rw * (C)(6.0 / 36.0) * (-ux_w + uy_w);
            }
            gv[2] = scalar_bc<C>(k.swirl[sd], own<S, C>(src, k, G0 + 4, i, 0), wall_psi<C>(k, sd, y) * sc, true);
            hv[2] = scalar_bc<C>(k.heat[sd], own<S, C>(src, k, H0 + 4, i, 0), (k.Tw[sd] - k.T0) * sc, false);
        }
        if (at_cN) {
            const int sd = 3;
            const C rw = k.rho0 * sc;
            const C ux_w = k.uwx[sd], uy_w = k.uwy[sd];
            fv[4] = own<S, C>(src, k, 2, i, nr - 1) + rw * (C)(6.0 / 9.0) * (-uy_w);
            fv[7] = own<S, C>(src, k, 5, i, nr - 1) + rw * (C)(6.0 / 36.0) * (-ux_w - uy_w);
            fv[8] = own<S, C>(src, k, 6, i, nr - 1) + rw * (C)(6.0 / 36.0) * (ux_w - uy_w);
            gv[4] = scalar_bc<C>(k.swirl[sd], own<S, C>(src, k, G0 + 2, i, nr - 1), wall_psi<C>(k, sd, y) * sc, true);
            hv[4] = scalar_bc<C>(k.heat[sd], own<S, C>(src, k, H0 + 2, i, nr - 1), (k.Tw[sd] - k.T0) * sc, false);
        }
    }
    // end walls (rows 0 and nz-1 unless periodic); they win in corners.  A
    // free surface (Sec. 3.6) reflects f specularly: the population that
    // left the neighbour column towards the wall, e_x reversed; at a corner
    // column the lateral side's rule for the node itself
    if (!has_m) {
        const int sd = end_seg(k, 0, cl);
        const C rw = k.rho0 * sc, ux_w = k.uwx[sd], uy_w = k.uwy[sd];
        if (k.flow[sd] == 3) {
            fv[1] = own<S, C>(src, k, 3, i, cl);
            fv[5] = at_c0 ? own<S, C>(src, k, 7, i, 0) +
                                (k.flow[2] == 1 ? (C)0 : rw * (C)(6.0 / 36.0) * (k.uwx[2] + k.uwy[2]))
                          : own<S, C>(src, k, 6, i, cl > 0 ? cl - 1 : 0);
            fv[8] = at_cN ? own<S, C>(src, k, 6, i, cl) + rw * (C)(6.0 / 36.0) * (k.uwx[3] - k.uwy[3])
                          : own<S, C>(src, k, 7, i, cl + 1 < nr ? cl + 1 : cl);
        } else {
            fv[1] = own<S, C>(src, k, 3, i, cl) + rw * (C)(6.0 / 9.0) * ux_w;
            fv[5] = own<S, C>(src, k, 7, i, cl) + rw * (C)(6.0 / 36.0) * (ux_w + uy_w);
            fv[8] = own<S, C>(src, k, 6, i, cl) + rw * (C)(6.0 / 36.0) * (ux_w - uy_w);
        }
        gv[1] = scalar_bc<C>(k.swirl[sd], own<S, C>(src, k, G0 + 3, i, cl), wall_psi<C>(k, sd, y) * sc, true);
        hv[1] = scalar_bc<C>(heat_rule(k, sd), own<S, C>(src, k, H0 + 3, i, cl), (end_T(k, sd, y) - k.T0) * sc,
                             false);
    }
    if (!has_p) {
        const int sd = end_seg(k, 1, cl);
        const C rw = k.rho0 * sc, ux_w = k.uwx[sd], uy_w = k.uwy[sd];
        if (k.flow[sd] == 3) {
            fv[3] = own<S, C>(src, k, 1, i, cl);
            fv[6] = at_c0 ? own<S, C>(src, k, 8, i, 0) +
                                (k.flow[2] == 1 ? (C)0 : rw * (C)(6.0 / 36.0) * (-k.uwx[2] + k.uwy[2]))
                          : own<S, C>(src, k, 5, i, cl > 0 ? cl - 1 : 0);
            fv[7] = at_cN ? own<S, C>(src, k, 5, i, cl) + rw * (C)(6.0 / 36.0) * (-k.uwx[3] - k.uwy[3])
                          : own<S, C>(src, k, 8, i, cl + 1 < nr ? cl + 1 : cl);
        } else {
            fv[3] = own<S, C>(src, k, 1, i, cl) + rw * (C)(6.0 / 9.0) * (-ux_w);
            fv[6] = own<S, C>(src, k, 8, i, cl) + rw * (C)(6.0 / 36.0) * (-ux_w + uy_w);
            fv[7] = own<S, C>(src, k, 5, i, cl) + rw * (C)(6.0 / 36.0) * (-ux_w - uy_w);
        }
        gv[3] = scalar_bc<C>(k.swirl[sd], own<S, C>(src, k, G0 + 1, i, cl), wall_psi<C>(k, sd, y) * sc, true);
        hv[3] = scalar_bc<C>(heat_rule(k, sd), own<S, C>(src, k, H0 + 1, i, cl), (end_T(k, sd, y) - k.T0) * sc,
                             false);
    }
}

#include "lb_pair.cuh"

// SplitMix64 finaliser of a step counter (the same function as step_salt on
// the host: a lattice draws the same rounding bits alone and in a batch)
__host__ __device__ __forceinline__ uint32_t salt_of(unsigned long long step)
{
    unsigned long long z = step + 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return (uint32_t)(z ^ (z >> 31));
}

// Programmatic dependent launch (sm_90+): the kernels of consecutive steps
// are launched with programmatic stream serialisation, so a step's blocks
// may start while the previous step's last blocks run.  Each block first
// allows the next launch to begin, then waits until every earlier grid of
// the stream has completed and its writes are visible, before it reads or
// writes any distribution.  Without the launch attribute both are no-ops.
__device__ __forceinline__ void grid_dependency_trigger()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void grid_dependency_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void grid_dependency_trigger_and_wait()
{
    grid_dependency_trigger();
    grid_dependency_wait();
}

// Waits on a flag in global memory: at most kFlagWaitLimit polls with a short
// sleep between them (about a second).
constexpr int kFlagWaitLimit = 1 << 20;

template <typename I> __device__ __forceinline__ I ld_acquire_gpu(const I *p)
{
    static_assert(sizeof(I) == 4, "32-bit flags");
    I v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
template <typename I> __device__ __forceinline__ void st_release_gpu(I *p, I v)
{
    static_assert(sizeof(I) == 4, "32-bit flags");
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

#include "lb_tile.cuh"

// FP64 step (the reference path of the other storages).  The FP64 pipe bounds
// it: an FP64 instruction occupies a scheduler's pipe for 64 cycles whatever
// the number of active lanes (76 with all four of an SM's busy; measured), so
// what counts is FP64 instructions per row of 32 columns -- 306 of the node
// update, 33 of a row's fields -- and schedulers in use.  A block takes `rows`
// rows of a 32-column window.  First its warps form the fields of the stored
// state of the rows and their neighbours, once per node, the two halo columns
// gathered into tasks of 16 rows each; then the warps update the rows.  With
// split = 2 a row goes to two warps, one storing f and the other g and h, each
// repeating the source terms (194 and 173 instead of 306 instructions): faster
// where the lattice has fewer rows of 32 columns than the device schedulers.
// The distributions are read where they lie (L1 / L2): loads, indices and
// rules other than arithmetic cost nothing beside the FP64 pipe.
// 41 x 41: 70.6 us per step before (30-column march, at least four rows per
// warp, terms not fused), 10.6 us now; 256 x 512: 220 us, 89.3 us.
constexpr int kFields64Cols = 34;  // 32 columns and the halo columns

// Wall rules of the FP64 step with their constants formed once on the host
// (entries 0..3 the sides, 4 the outer segment of a split top): the
// moving-wall terms of the three populations entering from the wall, and sign
// and constant of the scalar rules x = s x_own + c, the constants of end walls
// linear in the column radius (psi_w = rho0 omega y; the ramp): c0 + c1 y.
struct Walls64 {
    double f[5][3], gs[5], gc0[5], gc1[5], hs[5], hc0[5], hc1[5];
};

Walls64 make_walls64(const KP<double> &k)
{
    Walls64 w;
    for (int sd = 0; sd < 5; ++sd) {
        const double a = k.rho0 * (6.0 / 9.0), b = k.rho0 * (6.0 / 36.0), ux = k.uwx[sd], uy = k.uwy[sd];
        const bool end = sd != 2 && sd != 3, up = sd == 1 || sd == 4;
        const double f[4][3] = {{a * ux, b * (ux + uy), b * (ux - uy)},      // f1, f5, f8 at the bottom
                                {-a * ux, b * (-ux + uy), b * (-ux - uy)},   // f3, f6, f7 at the top
                                {a * uy, b * (ux + uy), b * (-ux + uy)},     // f2, f5, f6 at the inner side
                                {-a * uy, b * (-ux - uy), b * (ux - uy)}};   // f4, f7, f8 at the outer side
        for (int q = 0; q < 3; ++q) w.f[sd][q] = f[up ? 1 : sd][q];
        w.gs[sd] = k.swirl[sd] == 0 || k.swirl[sd] == 2 ? -1.0 : 1.0;
        const double psi = k.swirl[sd] == 0 ? (2.0 / 6.0) * (k.rho0 * k.omega[sd]) : 0.0;
        w.gc0[sd] = end ? 0.0 : psi * (sd == 2 ? k.r0c : k.roc);
        w.gc1[sd] = end ? psi : 0.0;
        const bool ramp = k.heat[sd] == 4;
        w.hs[sd] = k.heat[sd] == 0 || ramp ? -1.0 : 1.0;
        w.hc0[sd] = ramp ? (2.0 / 6.0) * (k.ramp0 - k.T0) : (k.heat[sd] == 0 ? (2.0 / 6.0) * (k.Tw[sd] - k.T0) : 0.0);
        w.hc1[sd] = ramp ? (2.0 / 6.0) * k.ramp1 : 0.0;
    }
    return w;
}

__global__ void __launch_bounds__(256) k_step64(const __grid_constant__ KP<double> k, const __grid_constant__ Walls64 w,
                                                const double *__restrict__ src, double *__restrict__ dst, int rows,
                                                int nwin, int split)
{
    extern __shared__ double fields64[];  // [rows + 2][u_x, u_y, u_theta, T][34]
    const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31, W = blockDim.x >> 5;
    const int c0 = (int)(blockIdx.x % nwin) * 32, s = (int)(blockIdx.x / nwin) * rows;
    const int nr = k.nr, nz = k.nz, n = min(rows, nz - s);
    const int c = c0 + lane, cl = min(c, nr - 1);
    const bool at_c0 = c == 0, at_cN = c == nr - 1, inner = c0 == 0, outer = c0 + 32 >= nr;
    // all of the column's own arithmetic before the wait for the last step
    const double y = k.r0 + cl + 0.5;
    const Geo<D1> geo = geo_of(k.pc, D1{k.planar ? 0.0 : rcp1(y)});
    grid_dependency_trigger_and_wait();

    // Fields of rows s - 1 .. s + n: all four of the block's rows, task by task;
    // of the halo columns c0 - 1 and c0 + 32, as (row, side) pairs; and u_y of
    // the rows below and above, one task.
    const int halo_tasks = (2 * n + 31) / 32;
    for (int t = warp; t < n + halo_tasks + 1; t += W) {
        const int h = lane + 32 * (t - n);
        const bool rim = t == n + halo_tasks, halo = !rim && t >= n;
        for (int q = 0; q < (rim ? 2 : 1); ++q) {
            const int r = rim ? q * (n + 1) : (halo ? (h >> 1) + 1 : t + 1);
            const int cc = halo ? ((h & 1) ? c0 + 32 : c0 - 1) : c;
            int i = s - 1 + r;
            if (k.xper) i = i < 0 ? i + nz : (i >= nz ? i - nz : i);
            if (r > n + 1 || (halo && r > n) || i < 0 || i >= nz || cc < 0 || cc >= nr) continue;
            double v[NQ];
            load_row<double, double>(src, k, i, cc, v);
            const double s13 = v[1] + v[3], s24 = v[2] + v[4], s5678 = (v[5] + v[7]) + (v[6] + v[8]);
            const double a57 = v[5] - v[7], a86 = v[8] - v[6];
            const double ir = rcp1(k.rho0 + ((v[0] + s13) + (s24 + s5678)));
            double *f = fields64 + (r * 4) * kFields64Cols + (cc - c0 + 1);
            f[kFields64Cols] = ((v[2] - v[4]) + (a57 - a86)) * ir;
            if (rim) continue;
            f[0] = ((v[1] - v[3]) + (a57 + a86)) * ir;
            f[2 * kFields64Cols] = ((v[9] + v[10]) + (v[11] + v[12]) + v[13]) * ir;
            f[3 * kFields64Cols] = k.T0 + ((v[14] + v[15]) + (v[16] + v[17]) + v[18]);
        }
    }
    __syncthreads();

    for (int t = warp; t < n * split; t += W) {
        const int r = t / split + 1, i = s + r - 1;
        const bool has_m = i > 0 || k.xper, has_p = i + 1 < nz || k.xper;
        // pulled values
        const int im = i > 0 ? i - 1 : nz - 1, ip = i + 1 < nz ? i + 1 : 0;
        const int jm = max(cl - 1, 0), jp = min(cl + 1, nr - 1);
        auto ld = [&](int q, int row, int col) { return src[q * k.plane + (long long)row * k.pitch + col]; };
        double fv[9] = {ld(0, i, cl),  ld(1, im, cl), ld(2, i, jm),  ld(3, ip, cl), ld(4, i, jp),
                        ld(5, im, jm), ld(6, ip, jm), ld(7, ip, jp), ld(8, im, jp)};
        double gv[5] = {ld(9, i, cl), ld(10, im, cl), ld(11, i, jm), ld(12, ip, cl), ld(13, i, jp)};
        double hv[5] = {ld(14, i, cl), ld(15, im, cl), ld(16, i, jm), ld(17, ip, cl), ld(18, i, jp)};
        // lateral walls and the axis (Sec. 3)
        if (inner && at_c0) {
            if (k.flow[2] == 1) {
                fv[2] = ld(4, i, 0);
                if (has_m) fv[5] = ld(8, im, 0);
                if (has_p) fv[6] = ld(7, ip, 0);
            } else {
                fv[2] = ld(4, i, 0) + w.f[2][0];
                fv[5] = ld(7, i, 0) + w.f[2][1];
                fv[6] = ld(8, i, 0) + w.f[2][2];
            }
            gv[2] = __fma_rn(w.gs[2], ld(13, i, 0), w.gc0[2]);
            hv[2] = __fma_rn(w.hs[2], ld(18, i, 0), w.hc0[2]);
        }
        if (outer && at_cN) {
            fv[4] = ld(2, i, cl) + w.f[3][0];
            fv[7] = ld(5, i, cl) + w.f[3][1];
            fv[8] = ld(6, i, cl) + w.f[3][2];
            gv[4] = __fma_rn(w.gs[3], ld(11, i, cl), w.gc0[3]);
            hv[4] = __fma_rn(w.hs[3], ld(16, i, cl), w.hc0[3]);
        }
        // end walls; they win in corners.  A free surface reflects f
        // specularly, at a corner column by the lateral side's rule
        if (!has_m) {
            const int sd = 0;
            if (k.flow[sd] == 3) {
                fv[1] = ld(3, i, cl);
                fv[5] = ld(6, i, jm);
                fv[8] = ld(7, i, jp);
                if (inner && at_c0) fv[5] = k.flow[2] == 1 ? ld(7, i, 0) : ld(7, i, 0) + w.f[2][1];
                if (outer && at_cN) fv[8] = ld(6, i, cl) + w.f[3][2];
            } else {
                fv[1] = ld(3, i, cl) + w.f[sd][0];
                fv[5] = ld(7, i, cl) + w.f[sd][1];
                fv[8] = ld(6, i, cl) + w.f[sd][2];
            }
            gv[1] = __fma_rn(w.gs[sd], ld(12, i, cl), w.gc1[sd] * y);
            hv[1] = __fma_rn(w.hs[sd], ld(17, i, cl), w.hc0[sd]);
        }
        if (!has_p) {
            const int sd = end_seg(k, 1, cl);
            if (k.flow[sd] == 3) {
                fv[3] = ld(1, i, cl);
                fv[6] = ld(5, i, jm);
                fv[7] = ld(8, i, jp);
                if (inner && at_c0) fv[6] = k.flow[2] == 1 ? ld(8, i, 0) : ld(8, i, 0) + w.f[2][2];
                if (outer && at_cN) fv[7] = ld(5, i, cl) + w.f[3][1];
            } else {
                fv[3] = ld(1, i, cl) + w.f[sd][0];
                fv[6] = ld(8, i, cl) + w.f[sd][1];
                fv[7] = ld(5, i, cl) + w.f[sd][2];
            }
            gv[3] = __fma_rn(w.gs[sd], ld(10, i, cl), w.gc1[sd] * y);
            hv[3] = __fma_rn(w.hs[sd], ld(15, i, cl), __fma_rn(w.hc1[sd], y, w.hc0[sd]));
        }

        // undivided central differences of the stored-state fields, with ghosts
        const double *f = fields64 + (r * 4) * kFields64Cols + (cl - c0 + 1);
        auto at = [&](int q, int dr, int dc) { return f[(dr * 4 + q) * kFields64Cols + dc]; };
        double l[4], rr[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            l[q] = at(q, 0, -1);
            rr[q] = at(q, 0, 1);
        }
        if (inner && at_c0)
#pragma unroll
            for (int q = 0; q < 4; ++q) l[q] = __fma_rn(k.gha[0][q], at(q, 0, 0), k.ghb[0][q]);
        if (outer && at_cN)
#pragma unroll
            for (int q = 0; q < 4; ++q) rr[q] = __fma_rn(k.gha[1][q], at(q, 0, 0), k.ghb[1][q]);
        double uy_m = at(1, -1, 0), uy_p = at(1, 1, 0);
        if (!has_m) uy_m = k.flow[0] == 3 ? at(1, 0, 0) : 2.0 * k.uwy[0] - at(1, 0, 0);
        if (!has_p) {
            const int st = end_seg(k, 1, cl);
            uy_p = k.flow[st] == 3 ? at(1, 0, 0) : 2.0 * k.uwy[st] - at(1, 0, 0);
        }

        D1 f1[9], g1[5], h1[5];
#pragma unroll
        for (int q = 0; q < 9; ++q) f1[q] = D1{fv[q]};
#pragma unroll
        for (int q = 0; q < 5; ++q) g1[q] = D1{gv[q]}, h1[q] = D1{hv[q]};
        NodeVals<D1> o;
        auto update = [&]() {
            update_node2<false>(k.pc, k.explicit_src, geo, f1, g1, h1, D1{uy_p - uy_m}, D1{rr[0] - l[0]},
                                D1{rr[1] - l[1]}, D1{rr[2] - l[2]}, D1{rr[3] - l[3]}, o);
        };
        double *p = dst + (long long)i * k.pitch + c;
        // each branch keeps only the arithmetic its planes need
        if (split == 1) {
            update();
            if (c < nr)
#pragma unroll
                for (int q = 0; q < NQ; ++q) p[q * k.plane] = o.v[q].v;
        } else if (t & 1) {
            update();
            if (c < nr)
#pragma unroll
                for (int q = 9; q < NQ; ++q) p[q * k.plane] = o.v[q].v;
        } else {
            update();
            if (c < nr)
#pragma unroll
                for (int q = 0; q < 9; ++q) p[q * k.plane] = o.v[q].v;
        }
    }
}

// Block of a step grid in traversal order: every other step (rev = 1) the
// blocks take the lattice from its last row segment back to its first.  A step
// then starts on the rows the previous step wrote last, which are still in
// the L2 (129 MB against the 319 MB of the 1024 x 2048 FP32 lattice); the
// results do not depend on the order.
__device__ __forceinline__ void step_block(int rev, int &bx, int &by)
{
    const unsigned nb = gridDim.x * gridDim.y, b0 = blockIdx.y * gridDim.x + blockIdx.x;
    const unsigned b = rev ? nb - 1u - b0 : b0;
    bx = (int)(b % gridDim.x);
    by = (int)(b / gridDim.x);
}

// FP32-compute step on column pairs (lb_pair.cuh): 64 aligned columns per warp
#ifndef LB_STEP2_MAXREG
#define LB_STEP2_MAXREG 232
#endif
template <typename S>
__global__ void __maxnreg__(LB_STEP2_MAXREG) k_step2(KP<float> k, const S *__restrict__ src, S *__restrict__ dst,
                                                     int seg_rows, int nwin2, uint32_t salt, int rev)
{
    int bx, by;
    step_block(rev, bx, by);
    const int warp = bx * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (warp >= nwin2) return;
    const int lane = threadIdx.x & 31;
    const int s = by * seg_rows;
    const int e = min(k.nz, s + seg_rows);
    const int A = warp * 64 + 2 * lane;
    const int Amax = (k.nr - 1) & ~1;
    int hcol = lane == 0 ? warp * 64 - 1 : warp * 64 + 64;
    hcol = hcol < 0 ? 0 : (hcol >= k.nr ? k.nr - 1 : hcol);
    RowDirect<S> rs{src, &k, A <= Amax ? A : Amax, hcol, (s > 0 || k.xper) ? s - 1 : s, k.nz, 0,
                    lane == 0 || lane == 31};
    grid_dependency_trigger_and_wait();
    march2<S>(k, src, dst, warp * 64, s, e, salt, rs);
}

// The same step with the rows of each warp fetched by TMA into a ring of
// shared-memory stages (one bulk tensor copy per row), so that a warp has
// up to kTmaStages rows in flight without holding them in registers.
template <typename S>
__global__ void __maxnreg__(LB_STEP2_MAXREG)
    k_step2_tma(KP<float> k, const __grid_constant__ CUtensorMap map, const S *__restrict__ src,
                S *__restrict__ dst, int seg_rows, int nwin2, uint32_t salt, int *status, int rev)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int wib = threadIdx.x >> 5;
    int bx, by;
    step_block(rev, bx, by);
    const int warp = bx * (blockDim.x >> 5) + wib;
    if (warp >= nwin2) return;
    const int lane = threadIdx.x & 31;
    const int s = by * seg_rows;
    const int e = min(k.nz, s + seg_rows);
    const bool has_m = s > 0 || k.xper, has_last = e < k.nz || k.xper;
    const int nrows = (e - s) + (has_m ? 1 : 0) + (has_last ? 1 : 0);
    const int per_warp = kTmaStages * TmaGeom<S>::stage_bytes + 128;  // keeps every ring 128-byte aligned
    unsigned char *ring = smem + per_warp * wib;
    RowTma<S> rs;
    rs.map = &map;
    rs.k = &k;
    rs.ring = ring;
    rs.ring_s = smem_u32(ring);
    rs.bar_s = smem_u32(ring + kTmaStages * TmaGeom<S>::stage_bytes);
    rs.first = has_m ? s - 1 : s;
    rs.nrows = nrows;
    rs.nz = k.nz;
    rs.taken = 0;
    rs.lane = lane;
    rs.x0 = warp * 64 - TmaGeom<S>::off;
    rs.status = status;
    grid_dependency_trigger_and_wait();
    rs.start();
    march2<S>(k, src, dst, warp * 64, s, e, salt, rs);
}

// The step with the rows resident in the TMA ring (march3): no row carried
// in registers.  kRingStages<S> stages of one row each per warp: rows i-1,
// i, i+1 of the step and one more in flight.
#ifndef LB_STEP3_MAXREG
#define LB_STEP3_MAXREG 168
#endif
template <typename S> constexpr int kRingStages = 4;
// march3 forms, as measured on GB300 (all give the same bits): the
// single-lattice FP32 step takes the separate interior form of the row update
// (+5 %; in 16-bit storage it cost 2-3 %) and every kernel reads the wall and
// axis values from the ring (the batched FP32 step on serving-size lattices,
// where nearly every warp holds a wall or the axis: +10 % over global loads).
template <typename S> constexpr bool kStepSplit = sizeof(S) == 4;

template <typename S>
__host__ __device__ size_t ring_smem_bytes(int wpb)
{
    return (size_t)wpb * (kRingStages<S> * TmaGeom<S>::stage_bytes + 128);
}

template <typename S, bool kPinned>
__global__ void __maxnreg__(LB_STEP3_MAXREG)
    k_step3_tma(KP<float> k, const __grid_constant__ CUtensorMap map, const S *__restrict__ src,
                S *__restrict__ dst, int seg_rows, int nwin2, uint32_t salt, int *status, int rev)
{
    constexpr int R = kRingStages<S>;
    extern __shared__ __align__(128) unsigned char smem[];
    const int wib = threadIdx.x >> 5;
    int bx, by;
    step_block(rev, bx, by);
    const int warp = bx * (blockDim.x >> 5) + wib;
    if (warp >= nwin2) return;
    const int s = by * seg_rows;
    const int e = min(k.nz, s + seg_rows);
    const bool has_m = s > 0 || k.xper, has_last = e < k.nz || k.xper;
    const int per_warp = R * TmaGeom<S>::stage_bytes + 128;  // keeps every ring 128-byte aligned
    unsigned char *ring = smem + per_warp * wib;
    RowRing<S, R> rs;
    rs.map = &map;
    rs.ring = ring;
    rs.ring_s = smem_u32(ring);
    rs.bar_s = smem_u32(ring + R * TmaGeom<S>::stage_bytes);
    rs.bar_stride = 8;
    rs.first = has_m ? s - 1 : s;
    rs.nrows = (e - s) + (has_m ? 1 : 0) + (has_last ? 1 : 0);
    rs.nz = k.nz;
    rs.x0 = warp * 64 - TmaGeom<S>::off;
    rs.lane = threadIdx.x & 31;
    rs.status = status;
    // programmatic dependent launch: let the next step's blocks become
    // resident now, and touch no distribution before the previous step is done
    grid_dependency_trigger_and_wait();
    rs.start();
    march3<S, R, kStepSplit<S>, true, kPinned>(k, src, dst, warp * 64, s, e, salt, rs);
}

// Stream function of the meridian flow (Sec. 3.6): dPsi/dy = -y u_x with
// Psi = 0 on the inner boundary y = r0, midpoint sums over whole cells, so
// psi[i][j] is Psi on the face y = r0 + j + 1 of row i.  One warp per row:
// an FP64 warp scan per 32 columns plus the carry; rowmax[i] = max |Psi|.
__global__ void __launch_bounds__(128) k_psi(const double *__restrict__ ux, double *__restrict__ psi,
                                             double *__restrict__ rowmax, int nrows, int nr, double r0)
{
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= nrows) return;
    const int lane = threadIdx.x & 31;
    double carry = 0.0, m = 0.0;
    for (int j0 = 0; j0 < nr; j0 += 32) {
        const int j = j0 + lane;
        double v = j < nr ? -(r0 + j + 0.5) * ux[(long long)row * nr + j] : 0.0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double w = __shfl_up_sync(FULL, v, o);
            if (lane >= o) v += w;
        }
        v += carry;
        if (j < nr) {
            if (psi) psi[(long long)row * nr + j] = v;
            m = fmax(m, fabs(v));
        }
        carry = __shfl_sync(FULL, v, 31);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(FULL, m, o));
    if (lane == 0) rowmax[row] = m;
}

// Pre-collision fields of the nodes of a block: 128 columns from c0, rows s ..
// s + n - 1, by 256 threads, a thread's nodes all in one column.  Eight rows at
// a time the block forms the macroscopic fields of the stored state of the rows
// and their neighbours in shared memory (F: ten rows, two of which stay for
// the next eight), then each thread its nodes.  stored(i, c, fields) sees every
// node's stored state once, node(i, c, out) its pre-collision state.  (A warp
// marching 32 rows of 30 columns on its own, as before, is a serial chain of
// 32 row updates; these are four nodes per thread and round, all independent: the
// diagnostics of 1024 x 2048 FP32 took 220 us and take 110.)
constexpr int kBlockCols = 128, kBlockChunk = 8, kBlockThreads = 256, kBlockPitch = kBlockCols + 2;
template <typename C> constexpr size_t kBlockSmem = (size_t)(kBlockChunk + 2) * 4 * kBlockPitch * sizeof(C);

template <typename S, typename C, typename Stored, typename Node>
__device__ __forceinline__ void block_fields(const KP<C> &k, const S *__restrict__ src, int c0, int s, int n, C *F,
                                             Stored stored, Node node)
{
    const int nr = k.nr, nz = k.nz;
    const int c = c0 + (int)(threadIdx.x % kBlockCols), half = threadIdx.x / kBlockCols;
    const bool at_c0 = c == 0, at_cN = c == nr - 1;
    const double yd = k.r0 + c + 0.5;
    const C y = (C)yd, iy = (C)(1.0 / yd);
    auto slot = [&](int rel) { return F + ((rel + 1) % (kBlockChunk + 2)) * 4 * kBlockPitch; };
    // the fields of row s + rel, column cc; rows and columns outside the lattice have none
    auto form = [&](int rel, int cc, bool own_node) {
        int i = s + rel;
        if (k.xper) i = i < 0 ? i + nz : (i >= nz ? i - nz : i);
        if (i < 0 || i >= nz || cc < 0 || cc >= nr) return;
        C v[NQ];
        load_row<S, C>(src, k, i, cc, v);
        const PM<C> m = moments<S, C>(v, k);
        C *f = slot(rel) + (cc - c0 + 1);
        f[0] = m.ux;
        f[kBlockPitch] = m.uy;
        f[2 * kBlockPitch] = m.ut;
        f[3 * kBlockPitch] = m.T;
        if (own_node) stored(i, cc, m);
    };
    for (int r0 = 0; r0 < n; r0 += kBlockChunk) {
        const int m = min(kBlockChunk, n - r0), first = r0 == 0 ? -1 : r0 + 1;
#pragma unroll 2
        for (int rel = first + half; rel <= r0 + m; rel += 2) form(rel, c, rel >= 0 && rel < n);
        if ((int)threadIdx.x < 2 * (r0 + m - first + 1))
            form(first + (int)(threadIdx.x >> 1), (threadIdx.x & 1) ? c0 + kBlockCols : c0 - 1, false);
        __syncthreads();
        if (c < nr)
            for (int rel = r0 + half; rel < r0 + m; rel += 2) {
                const int i = s + rel;
                const bool has_m = i > 0 || k.xper, has_p = i + 1 < nz || k.xper;
                const int im = i > 0 ? i - 1 : nz - 1, ip = i + 1 < nz ? i + 1 : 0;
                const int jm = max(c - 1, 0), jp = min(c + 1, nr - 1);
                auto ld = [&](int q, int row, int col) { return own<S, C>(src, k, q, row, col); };
                // pulled values (scaled storage units)
                C fv[9] = {ld(0, i, c),   ld(1, im, c),  ld(2, i, jm),  ld(3, ip, c), ld(4, i, jp),
                           ld(5, im, jm), ld(6, ip, jm), ld(7, ip, jp), ld(8, im, jp)};
                C gv[5] = {ld(9, i, c), ld(10, im, c), ld(11, i, jm), ld(12, ip, c), ld(13, i, jp)};
                C hv[5] = {ld(14, i, c), ld(15, im, c), ld(16, i, jm), ld(17, ip, c), ld(18, i, jp)};
                wall_rules1<S, C>(k, src, i, c, at_c0, at_cN, has_m, has_p, y, k.scale, fv, gv, hv);
                if (Scaled<S>::value) {
#pragma unroll
                    for (int q = 0; q < 9; ++q) fv[q] *= k.inv_scale;
#pragma unroll
                    for (int q = 0; q < 5; ++q) {
                        gv[q] *= k.inv_scale;
                        hv[q] *= k.inv_scale;
                    }
                }
                // central differences of the stored-state fields, with ghosts
                // (a free surface: no shear, u_y even across it)
                const C *f = slot(rel) + (c - c0 + 1), *fm = slot(rel - 1) + (c - c0 + 1), *fp = slot(rel + 1) + (c - c0 + 1);
                constexpr int P = kBlockPitch;
                const C uy = f[P];
                C uy_m = uy, uy_p = uy;
                if (has_m) uy_m = fm[P];
                else if (k.flow[end_seg(k, 0, c)] != 3) uy_m = (C)2 * k.uwy[end_seg(k, 0, c)] - uy;
                if (has_p) uy_p = fp[P];
                else if (k.flow[end_seg(k, 1, c)] != 3) uy_p = (C)2 * k.uwy[end_seg(k, 1, c)] - uy;
                C l[4], r[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    l[q] = f[q * P - 1];
                    r[q] = f[q * P + 1];
                }
                if (at_c0) {
                    const bool axis = k.flow[2] == 1;
                    l[0] = axis ? f[0] : (C)2 * k.uwx[2] - f[0];
                    l[1] = axis ? -uy : (C)2 * k.uwy[2] - uy;
                    const C ut = f[2 * P], T = f[3 * P];
                    l[2] = k.swirl[2] == 2 ? -ut : (k.swirl[2] == 0 ? (C)2 * k.omega[2] * (C)k.r0 - ut : ut);
                    l[3] = k.heat[2] == 0 ? (C)2 * k.Tw[2] - T : T;
                }
                if (at_cN) {
                    r[0] = (C)2 * k.uwx[3] - f[0];
                    r[1] = (C)2 * k.uwy[3] - uy;
                    const C ut = f[2 * P], T = f[3 * P];
                    r[2] = k.swirl[3] == 0 ? (C)2 * k.omega[3] * (C)(k.r0 + k.nr) - ut : ut;
                    r[3] = k.heat[3] == 0 ? (C)2 * k.Tw[3] - T : T;
                }
                NodeOut<C> o;
                update_node<C>(k, y, iy, fv, gv, hv, (C)0.5 * (uy_p - uy_m), (C)0.5 * (r[0] - l[0]),
                               (C)0.5 * (r[1] - l[1]), (C)0.5 * (r[2] - l[2]), (C)0.5 * (r[3] - l[3]), o);
                node(i, c, o);
            }
        __syncthreads();
    }
}

// Registers for four of these blocks on an SM, where an FP32 kernel has two by
// itself, as they wait for their loads: fields of 2048 x 2048 FP32 290 us in all
// as lb_stream_function took them, 267 with three, 251 so (238 storing u_x
// alone); diagnostics of 1024 x 2048 FP32 128, 122 and 110 us, of 64 annuli in one
// FP16 batch, whose kernel also takes the lattice's parameters from shared memory,
// 538, 464 and 445 us.
template <typename C> constexpr int kBlocksPerSm = std::is_same<C, float>::value ? 4 : 1;

// Pre-collision fields of rows [row0, row1) as doubles, out[5][row1 - row0][nr],
// or u_x alone (plane 1): a block per `rows` rows.
template <typename S, typename C>
__global__ void __launch_bounds__(kBlockThreads, kBlocksPerSm<C>)
    k_fields(const __grid_constant__ KP<C> k, const S *__restrict__ src, double *__restrict__ out, int row0, int row1,
             int nbx, int rows, int only_ux)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int s = row0 + (int)(blockIdx.x / nbx) * rows;
    const long long n = (long long)(row1 - row0) * k.nr;  // plane stride of the output chunk
    block_fields<S, C>(
        k, src, (int)(blockIdx.x % nbx) * kBlockCols, s, min(row1, s + rows) - s, reinterpret_cast<C *>(smem),
        [](int, int, const PM<C> &) {},
        [&](int i, int c, const NodeOut<C> &o) {
            double *p = out + (long long)(i - row0) * k.nr + c;
            p[n] = (double)o.ux;
            if (only_ux) return;
            p[0] = (double)o.rho;
            p[2 * n] = (double)o.uy;
            p[3 * n] = (double)o.ut;
            p[4 * n] = (double)o.T;
        });
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(FULL, v, o));
    return v;
}

// The largest |u|, of FP64 squares.  FP64 instructions are scarce (the pipe takes
// one per SM every 19 cycles, conversions included), so an FP32 thread keeps the
// velocity whose FP32 square is the largest and squares it in FP64 (where FP32
// squares are exact) at its end: 1024 x 2048 FP32 128 us, 140 with every node's
// square in FP64.  Two nodes whose FP32 squares do not tell which is larger, as
// these are within 2^-22 of the exact ones, or which lie near the ends of the
// range, are compared in FP64.
template <typename C> struct NodeMax {
    C x = 0, y = 0, top = 0;
    static __device__ __forceinline__ double square(C x, C y) { return (double)x * (double)x + (double)y * (double)y; }
    __device__ __forceinline__ void add(C ux, C uy)
    {
        if constexpr (std::is_same<C, double>::value) {
            top = fmax(top, square(ux, uy));
        } else {
            const C t = ux * ux + uy * uy;
            if ((t < 0.999999f * top && top > 1e-30f) || (ux == 0 && uy == 0)) return;
            if (!(t > 1.000001f * top && t > 1e-30f && t < 3e38f) && !(square(ux, uy) > square(x, y))) return;
            x = ux;
            y = uy;
            top = fminf(t, 3.4e38f);
        }
    }
    __device__ __forceinline__ double value() const
    {
        if constexpr (std::is_same<C, double>::value) return sqrt(top);
        else return sqrt(square(x, y));
    }
};

// Diagnostics of block (bx, by) of a grid gx blocks wide, seg_rows rows each:
// partial sums in a fixed order, and the temperatures next to the walls in
// strips: rows 0, 1, nz - 2, nz - 1 (4 x nr values), then columns 0, 1, nr - 2,
// nr - 1 (4 x nz).
template <typename S, typename C>
__device__ __forceinline__ void diag_block(const KP<C> &k, const S *__restrict__ src, double *__restrict__ partial,
                                           double *__restrict__ strips, int seg_rows, int bx, int by, int gx, C *F)
{
    constexpr int warps = kBlockThreads / 32;
    __shared__ double sh[warps][5];
    const int nr = k.nr, nz = k.nz, s = by * seg_rows;
    double rd = 0.0, T = 0.0;
    NodeMax<C> u;
    bool bad = false;
    block_fields<S, C>(
        k, src, bx * kBlockCols, s, min(nz, s + seg_rows) - s, F, [&](int, int, const PM<C> &m) { rd += (double)m.rd; },
        [&](int i, int c, const NodeOut<C> &o) {
            T += (double)o.T;
            u.add(o.ux, o.uy);
            bad |= !(isfinite(o.rho) && isfinite(o.ux) && isfinite(o.uy) && isfinite(o.ut) && isfinite(o.T)) ||
                   o.rho < (C)0.5 || o.rho > (C)1.5;
            double *cs = strips + 4LL * nr;
            if (i <= 1) strips[(long long)i * nr + c] = (double)o.T;
            if (i >= nz - 2) strips[(long long)(i - nz + 4) * nr + c] = (double)o.T;
            if (c <= 1) cs[(long long)c * nz + i] = (double)o.T;
            if (c >= nr - 2) cs[(long long)(c - nr + 4) * nz + i] = (double)o.T;
        });
    const double y = k.r0 + (bx * kBlockCols + (int)(threadIdx.x % kBlockCols)) + 0.5;
    double vals[5] = {rd, rd * y, T, u.value(), bad ? 1.0 : 0.0};
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 5; ++q) vals[q] = q >= 3 ? warp_max(vals[q]) : warp_sum(vals[q]);
    if (lane == 0)
        for (int q = 0; q < 5; ++q) sh[wib][q] = vals[q];
    __syncthreads();
    if (threadIdx.x < 5) {
        const int q = threadIdx.x;
        double r = sh[0][q];
        for (int w = 1; w < warps; ++w) r = q >= 3 ? fmax(r, sh[w][q]) : r + sh[w][q];
        partial[(by * gx + bx) * NSUM + (q == 4 ? 8 : q)] = r;
    }
}

template <typename S, typename C>
__global__ void __launch_bounds__(kBlockThreads, kBlocksPerSm<C>)
    k_diag(const __grid_constant__ KP<C> k, const S *__restrict__ src, double *__restrict__ partial,
           double *__restrict__ strips, int seg_rows, int gx)
{
    extern __shared__ __align__(128) unsigned char smem[];
    diag_block<S, C>(k, src, partial, strips, seg_rows, blockIdx.x % gx, blockIdx.x / gx, gx, reinterpret_cast<C *>(smem));
}

// A block's sum (or largest) of 256 values, a fixed tree (deterministic).
__device__ __forceinline__ double tree256(double v, bool mx)
{
    __shared__ double sh[256];
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            const double a = sh[threadIdx.x], b = sh[threadIdx.x + w];
            sh[threadIdx.x] = mx ? fmax(a, b) : a + b;
        }
        __syncthreads();
    }
    return sh[0];
}

// The last reductions of a diagnostics, one block of 256 threads each: tasks 0
// .. 3 the wall heat-flux sums of the sides, 4 .. 8 the sums over the blocks.
//
// Wall heat fluxes (Sec. 3.2) from the pre-collision T next to the walls
// (strips of diag_block): one-sided second-order derivative through the wall
// value, wall half a cell away, (-8 T_w + 9 T_1 - T_2) / 3 along the inward
// direction; end walls weighted by the radius.
constexpr int kDiagTasks = 9;
template <typename C>
__device__ __forceinline__ void diag_task(const KP<C> &k, int task, const double *__restrict__ partial, int nblocks,
                                          const double *__restrict__ strips, double *__restrict__ result)
{
    if (task >= 4) {
        const int q = task == 8 ? 8 : task - 4;
        const bool mx = q == 3 || q == 8;
        double r = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
            const double v = partial[b * NSUM + q];
            r = mx ? fmax(r, v) : r + v;
        }
        r = tree256(r, mx);
        if (threadIdx.x == 0) result[q] = r;
        return;
    }
    const int sd = task, nr = k.nr, nz = k.nz;
    const double *r0 = strips, *r1 = strips + nr, *r2 = strips + 2 * nr, *r3 = strips + 3 * nr;
    const double *c0 = strips + 4 * nr, *c1 = c0 + nz, *c2 = c0 + 2 * nz, *c3 = c0 + 3 * nz;
    double acc = 0;
    if (wall_heated(k, sd)) {
        const double Tw = (double)k.Tw[sd];
        if (sd == 2)
            for (int i = threadIdx.x; i < nz; i += blockDim.x) acc += (-8.0 * Tw + 9.0 * c0[i] - c1[i]) / 3.0;
        else if (sd == 3)
            for (int i = threadIdx.x; i < nz; i += blockDim.x) acc += (8.0 * Tw - 9.0 * c3[i] + c2[i]) / 3.0;
        else if (sd == 0)
            for (int j = threadIdx.x; j < nr; j += blockDim.x)
                acc += (k.r0 + j + 0.5) * (-8.0 * Tw + 9.0 * r0[j] - r1[j]) / 3.0;
        else  // the top: the columns whose segment holds a wall temperature, each with its own value
            for (int j = threadIdx.x; j < nr; j += blockDim.x) {
                const int sg = end_seg(k, 1, j);
                if (k.heat[sg] != 0 && k.heat[sg] != 4) continue;
                const double Tj = (double)end_T(k, sg, (C)(k.r0 + j + 0.5));
                acc += (k.r0 + j + 0.5) * (8.0 * Tj - 9.0 * r3[j] + r2[j]) / 3.0;
            }
    }
    acc = tree256(acc, false);
    if (threadIdx.x == 0) {
        result[4 + sd] = wall_heated(k, sd) ? acc * k.nu_scale[sd] : 0.0;
        if (sd >= 2) result[7 + sd] = k.heat[sd] == 0 ? acc * k.keq_scale[sd] : 0.0;  // 9, 10: k_eq
    }
}

template <typename C>
__global__ void __launch_bounds__(256) k_diag_final(const __grid_constant__ KP<C> k, const double *__restrict__ partial,
                                                    int nblocks, const double *__restrict__ strips,
                                                    double *__restrict__ result)
{
    diag_task<C>(k, blockIdx.x, partial, nblocks, strips, result);
}

// ---- initialisation and exchange ---------------------------------------------

__constant__ double c_w9[9] = {4.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36};
__constant__ double c_w5[5] = {1.0 / 3, 1.0 / 6, 1.0 / 6, 1.0 / 6, 1.0 / 6};

// Equilibria of given fields: the D2Q9 one with Maxwellian raw moments is a
// product of a factor per axis, 2/3 - u^2 for e = 0 and (1/3 + u^2 +- u) / 2 for
// e = +-1; the D2Q5 ones use the same factors.  Bound by the FP64 pipe (35
// instructions and 19 conversions per node; the term by term form had over
// 100), behind the copy of its fields from the host.
template <typename S>
__global__ void k_init_fields(HostParams h, const double *__restrict__ fields, S *__restrict__ dst, int row0,
                              int row1)
{
    using C = typename std::conditional<std::is_same<S, double>::value, double, float>::type;
    const C scale = (C)h.scale;
    const double w0 = -4.0 / 9 * h.rho0, w1 = -1.0 / 9 * h.rho0, w5 = -1.0 / 36 * h.rho0, t0 = -1.0 / 3 * h.T0,
                 t1 = -1.0 / 6 * h.T0;
    const long long nrow = row1 - row0;
    const long long n = nrow * h.nr;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int i = row0 + (int)(t / h.nr), j = (int)(t % h.nr);
        const double rho = fields[t], ux = fields[n + t], uy = fields[2 * n + t];
        const double ut = fields[3 * n + t], T = fields[4 * n + t];
        const double hx = 0.5 * ux, hy = 0.5 * uy;
        const double x0 = __fma_rn(-ux, ux, 2.0 / 3), mx = __fma_rn(hx, ux, 1.0 / 6), xp = mx + hx, xm = mx - hx;
        const double y0 = __fma_rn(-uy, uy, 2.0 / 3), my = __fma_rn(hy, uy, 1.0 / 6), yp = my + hy, ym = my - hy;
        const double r0 = rho * x0, rp = rho * xp, rm = rho * xm, c0 = __fma_rn(-uy, uy, x0 - 1.0 / 3), ps = rho * ut;
        const double v[NQ] = {__fma_rn(r0, y0, w0), __fma_rn(rp, y0, w1), __fma_rn(r0, yp, w1), __fma_rn(rm, y0, w1),
                              __fma_rn(r0, ym, w1), __fma_rn(rp, yp, w5), __fma_rn(rm, yp, w5), __fma_rn(rm, ym, w5),
                              __fma_rn(rp, ym, w5), ps * c0, ps * xp, ps * yp, ps * xm, ps * ym,
                              __fma_rn(T, c0, t0), __fma_rn(T, xp, t1), __fma_rn(T, yp, t1), __fma_rn(T, xm, t1),
                              __fma_rn(T, ym, t1)};
        S *p = dst + (long long)i * h.pitch + j;
#pragma unroll
        for (int q = 0; q < NQ; ++q) Cvt<S, C>::st(p + q * h.plane, Scaled<S>::value ? (C)v[q] * scale : (C)v[q]);
    }
}

template <typename S>
__global__ void k_export(HostParams h, const S *__restrict__ src, double *__restrict__ out, int row0, int row1)
{
    using C = typename std::conditional<std::is_same<S, double>::value, double, float>::type;
    const long long n = (long long)(row1 - row0) * h.nr;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int i = row0 + (int)(t / h.nr), j = (int)(t % h.nr);
        const S *p = src + (long long)i * h.pitch + j;
        for (int q = 0; q < NQ; ++q) {
            double rest = q < 9 ? c_w9[q] * h.rho0 : (q < 14 ? 0.0 : c_w5[q - 14] * h.T0);
            out[q * n + t] = (double)Cvt<S, C>::ld(p + q * h.plane) / h.scale + rest;
        }
    }
}

template <typename S>
__global__ void k_import(HostParams h, const double *__restrict__ in, S *__restrict__ dst, int row0, int row1)
{
    using C = typename std::conditional<std::is_same<S, double>::value, double, float>::type;
    const long long n = (long long)(row1 - row0) * h.nr;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const int i = row0 + (int)(t / h.nr), j = (int)(t % h.nr);
        S *p = dst + (long long)i * h.pitch + j;
        for (int q = 0; q < NQ; ++q) {
            double rest = q < 9 ? c_w9[q] * h.rho0 : (q < 14 ? 0.0 : c_w5[q - 14] * h.T0);
            Cvt<S, C>::st(p + q * h.plane, (C)((in[q * n + t] - rest) * h.scale));
        }
    }
}

// ---- batched step: many lattices, one launch per step ----------------------------

struct alignas(128) BatchDesc {
    unsigned char map[2][128];  // CUtensorMap of buf[0], buf[1] (64-byte aligned in the device array)
    unsigned char map64[2][128];  // the same with 64-column boxes (tiles)
    TileShape tiles;            // the lattice's tiles (automatic launch)
    KP<float> k;
    void *buf[2];
    int *status;               // the lattice's device status word
    unsigned long long step0;  // the lattice's step count when the batch was made
    int parity0;               // its current buffer then
    int nwin2, seg_rows, pad;
};

// The batch's step counter in device memory: the step at the start of the
// running CUDA graph replay.  A graph holds K launches that take steps
// counter + 0 .. counter + K - 1 and then a one-thread launch that adds K, so
// every replay is the same; launches outside a graph get their step as a
// parameter.
struct BatchCtl {
    unsigned long long counter;
    unsigned long long pad;
};

__global__ void k_batch_counter(BatchCtl *ctl, unsigned long long value, int add)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) ctl->counter = add ? ctl->counter + value : value;
}

// Instance of a work item: the last m < n with prefix[m] <= item (prefix is
// non-decreasing, prefix[0] = 0 <= item < prefix[n]).  Each round tests 32
// evenly spaced candidates of the remaining span with one load per lane and
// a ballot: one round for n <= 32, two for n <= 1024.
__device__ __forceinline__ int batch_instance(const int *__restrict__ prefix, int n, int item, int lane)
{
    int lo = 0, span = n;
    while (span > 1) {
        const int step = (span + 31) >> 5;
        const int m = lo + lane * step;
        const bool le = m < lo + span && prefix[m] <= item;
        const unsigned mask = __ballot_sync(FULL, le);  // bit 0 set: prefix[lo] <= item
        const int nlo = lo + (31 - __clz(mask)) * step;
        span = min(step, lo + span - nlo);
        lo = nlo;
    }
    return lo;
}

// Work items (instance, 64-column window, z-segment) are numbered by a prefix
// sum over the instances and dealt to the warps of a persistent grid.  The
// step is t0, plus the device counter when from_counter is set (inside a
// graph), so that every replay of a graph is the same.  Dynamic shared
// memory: one KP per warp.
template <typename S>
__global__ void __maxnreg__(LB_STEP2_MAXREG) k_batch(const BatchDesc *__restrict__ d, const int *__restrict__ prefix,
                                                     int n, int total, const BatchCtl *ctl, unsigned long long t0,
                                                     int from_counter)
{
    extern __shared__ __align__(128) unsigned char smem[];
    KP<float> *skp = reinterpret_cast<KP<float> *>(smem);
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    const unsigned long long t = t0 + (from_counter ? *(volatile const unsigned long long *)&ctl->counter : 0ULL);
    for (int item = blockIdx.x * wpb + wib; item < total; item += gridDim.x * wpb) {
        const int lo = batch_instance(prefix, n, item, lane);
        const BatchDesc *bd = d + lo;
        if (bd->k.pinned) continue;  // a launch of its own takes the pinned lattices
        __syncwarp();
        {
            const uint32_t *s = reinterpret_cast<const uint32_t *>(&bd->k);
            uint32_t *o = reinterpret_cast<uint32_t *>(&skp[wib]);
            for (int w = lane; w < (int)(sizeof(KP<float>) / 4); w += 32) o[w] = s[w];
        }
        __syncwarp();
        const KP<float> &k = skp[wib];
        const int local = item - prefix[lo];
        const int nw2 = bd->nwin2;
        const int w = local % nw2, sg = local / nw2;
        const int cur = (bd->parity0 + (int)(t & 1ULL)) & 1;
        const S *src = (const S *)bd->buf[cur];
        S *dst = (S *)bd->buf[cur ^ 1];
        const int seg = bd->seg_rows;
        const int s = sg * seg, e = min(k.nz, s + seg);
        const int A = w * 64 + 2 * lane, Amax = (k.nr - 1) & ~1;
        int hcol = lane == 0 ? w * 64 - 1 : w * 64 + 64;
        hcol = hcol < 0 ? 0 : (hcol >= k.nr ? k.nr - 1 : hcol);
        RowDirect<S> rs{src, &k, A <= Amax ? A : Amax, hcol, (s > 0 || k.xper) ? s - 1 : s, k.nz, 0,
                        lane == 0 || lane == 31};
        march2<S>(k, src, dst, w * 64, s, e, salt_of(bd->step0 + t), rs);
    }
}

// The batched step with the rows read in place from the TMA ring (march3):
// one warp per work item, tensor maps from the lattice's descriptor; the
// step as in k_batch.  Dynamic shared memory: the warps' rings (each a
// multiple of 128 bytes), then one KP per warp.  Each stage's mbarrier sits in
// the padding after the stage's box, which the copies never write, so that
// ten FP32 warps still fit on an SM (22,272 bytes per warp).
// R ring stages per warp: 4 by default (one more row in flight); 3 in the
// FP32 variant that fits 12 instead of 10 warps on an SM (16.9 instead of
// 22.3 KB of shared memory per warp), for batches too small to fill the GPU,
// whose step time is the latency of one wave of work items.
template <typename S, int R>
__host__ __device__ constexpr size_t batch3_ring_bytes()
{
    static_assert(TmaGeom<S>::stage_bytes - TmaGeom<S>::box_bytes >= 8 && TmaGeom<S>::box_bytes % 8 == 0,
                  "room for the stage's mbarrier after its box");
    return (size_t)R * TmaGeom<S>::stage_bytes;
}
template <typename S, int R = kRingStages<S>>
__host__ __device__ size_t batch3_smem_bytes(int wpb)
{
    return (size_t)wpb * (batch3_ring_bytes<S, R>() + sizeof(KP<float>));
}

template <typename S, int R, bool kPinned = false>
__global__ void __maxnreg__(LB_STEP3_MAXREG) k_batch3(const BatchDesc *__restrict__ d, const int *__restrict__ prefix,
                                                      int n, int total, const BatchCtl *ctl, unsigned long long t0,
                                                      int from_counter, int rev)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    unsigned char *ring = smem + batch3_ring_bytes<S, R>() * wib;
    KP<float> *skp = reinterpret_cast<KP<float> *>(smem + batch3_ring_bytes<S, R>() * wpb);
    // Programmatic dependent launch: the next step's blocks may become
    // resident now.  The instance lookup and the parameter copy read only
    // what no launch of the batch writes (the prefix sums, the descriptors),
    // so they overlap the previous launch's last blocks; the step counter and
    // the rows are read after the wait below.
    grid_dependency_trigger();
    const int item0 = blockIdx.x * wpb + wib;
    const int item = rev ? total - 1 - item0 : item0;  // every other step from the last item back
    if (item0 < total) {
        const int lo = batch_instance(prefix, n, item, lane);
        const BatchDesc *bd = d + lo;
        if ((bd->k.pinned != 0) != kPinned) return;  // a launch of its own takes the pinned lattices
        {
            const uint32_t *s = reinterpret_cast<const uint32_t *>(&bd->k);
            uint32_t *o = reinterpret_cast<uint32_t *>(&skp[wib]);
            for (int w = lane; w < (int)(sizeof(KP<float>) / 4); w += 32) o[w] = s[w];
        }
        __syncwarp();
        const KP<float> &k = skp[wib];
        const int local = item - prefix[lo];
        const int nw2 = bd->nwin2;
        const int w = local % nw2, sg = local / nw2;
        const int seg = bd->seg_rows;
        const int s = sg * seg, e = min(k.nz, s + seg);
        const bool has_m = s > 0 || k.xper, has_last = e < k.nz || k.xper;
        if (lane < 2)
            asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                             (unsigned long long)bd->map[lane])
                         : "memory");
        grid_dependency_wait();  // the previous launch is complete and its writes are visible
        const unsigned long long t =
            t0 + (from_counter ? *(volatile const unsigned long long *)&ctl->counter : 0ULL);
        const int cur = (bd->parity0 + (int)(t & 1ULL)) & 1;
        const CUtensorMap *map = reinterpret_cast<const CUtensorMap *>(bd->map[cur]);
        RowRing<S, R> rs;
        rs.map = map;
        rs.ring = ring;
        rs.ring_s = smem_u32(ring);
        rs.bar_s = smem_u32(ring + TmaGeom<S>::box_bytes);
        rs.bar_stride = TmaGeom<S>::stage_bytes;
        rs.first = has_m ? s - 1 : s;
        rs.nrows = (e - s) + (has_m ? 1 : 0) + (has_last ? 1 : 0);
        rs.nz = k.nz;
        rs.x0 = w * 64 - TmaGeom<S>::off;
        rs.lane = lane;
        rs.status = bd->status;
        rs.start();
        march3<S, R, false, true, kPinned>(k, (const S *)bd->buf[cur], (S *)bd->buf[cur ^ 1], w * 64, s, e,
                                           salt_of(bd->step0 + t), rs);
    }
}

// The batched step as one persistent launch for nsteps steps, for batches
// whose work items all fit on the device at once (a cooperative launch, one
// warp per item).  Instead of a launch boundary after each step, an item
// starts step j once the up-to-eight items around it (windows and z-segments
// +-1 in its lattice; segments wrap on a periodic lattice) have completed
// step j - 1: their halo rows and columns are then written (read after write)
// and no longer read from the buffer that step j overwrites (write after
// read).  done[item] counts the steps an item has completed in this launch,
// stored with release semantics after its writes; lanes 0..7 poll one
// neighbour each with acquire loads, at most kFlagWaitLimit times with a
// short sleep between polls (about a second), after which the lattice's
// status word gets LB_ERR_TIMEOUT and the warp leaves.
template <typename S, int R>
__global__ void __maxnreg__(LB_STEP3_MAXREG) k_batch3p(const BatchDesc *__restrict__ d, const int *__restrict__ prefix,
                                                       int n, int total, unsigned long long t0, int nsteps, int *done)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    unsigned char *ring = smem + batch3_ring_bytes<S, R>() * wib;
    KP<float> *skp = reinterpret_cast<KP<float> *>(smem + batch3_ring_bytes<S, R>() * wpb);
    const int item = blockIdx.x * wpb + wib;
    if (item >= total) return;
    const int lo = batch_instance(prefix, n, item, lane);
    const BatchDesc *bd = d + lo;
    if (bd->k.pinned) return;  // launches of their own take the pinned lattices
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&bd->k);
        uint32_t *o = reinterpret_cast<uint32_t *>(&skp[wib]);
        for (int q = lane; q < (int)(sizeof(KP<float>) / 4); q += 32) o[q] = src[q];
    }
    __syncwarp();
    const KP<float> &k = skp[wib];
    const int local = item - prefix[lo];
    const int nw2 = bd->nwin2;
    const int w = local % nw2, sg = local / nw2;
    const int seg = bd->seg_rows, nseg = (k.nz + seg - 1) / seg;
    const int s = sg * seg, e = min(k.nz, s + seg);
    const bool has_m = s > 0 || k.xper, has_last = e < k.nz || k.xper;
    // the neighbour item this lane watches (lanes 0..7), -1 for none
    int nb = -1;
    if (lane < 8) {
        const int c = lane < 4 ? lane : lane + 1;  // the 3 x 3 block without its centre
        const int dw = c % 3 - 1, dg = c / 3 - 1;
        const int w2 = w + dw;
        int g2 = sg + dg;
        if (k.xper) g2 = (g2 + nseg) % nseg;
        if (w2 >= 0 && w2 < nw2 && g2 >= 0 && g2 < nseg && g2 * nw2 + w2 != local) nb = prefix[lo] + g2 * nw2 + w2;
    }
    if (lane < 2)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((unsigned long long)bd->map[lane])
                     : "memory");
    RowRing<S, R> rs;
    rs.ring = ring;
    rs.ring_s = smem_u32(ring);
    rs.bar_s = smem_u32(ring + TmaGeom<S>::box_bytes);
    rs.bar_stride = TmaGeom<S>::stage_bytes;
    rs.first = has_m ? s - 1 : s;
    rs.nrows = (e - s) + (has_m ? 1 : 0) + (has_last ? 1 : 0);
    rs.nz = k.nz;
    rs.x0 = w * 64 - TmaGeom<S>::off;
    rs.lane = lane;
    rs.status = bd->status;
    for (int j = 0; j < nsteps; ++j) {
        if (j > 0) {
            bool ok = true;
            if (nb >= 0) {
                int it = 0;
                while (ld_acquire_gpu(done + nb) < j) {
                    if (++it > kFlagWaitLimit) {
                        ok = false;
                        break;
                    }
                    __nanosleep(100);
                }
            }
            if (!__all_sync(FULL, ok)) {
                if (lane == 0) atomicExch(bd->status, (int)LB_ERR_TIMEOUT);
                return;
            }
            // the neighbours' writes, acquired by the watching lanes, before this
            // warp's bulk-tensor reads; the ring stages read by the last step
            // before the copies that refill them
            __threadfence();
            asm volatile("fence.proxy.async.global;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        const unsigned long long t = t0 + (unsigned long long)j;
        const int cur = (bd->parity0 + (int)(t & 1ULL)) & 1;
        rs.map = reinterpret_cast<const CUtensorMap *>(bd->map[cur]);
        if (j == 0) rs.start();  // the barriers, once
        else rs.prime();
        march3<S, R, false, true>(k, (const S *)bd->buf[cur], (S *)bd->buf[cur ^ 1], w * 64, s, e,
                                  salt_of(bd->step0 + t), rs);
        if (*(volatile const int *)bd->status != 0) return;  // a ring wait ran out
        rs.advance();
        // publish: this item's writes, then its progress
        __threadfence();
        __syncwarp();
        if (lane == 0) st_release_gpu(done + item, j + 1);
    }
}

// Diagnostics of every lattice of a batch in two launches: the blocks of all the
// lattices' diagnostics grids in one grid, then the last reductions of every
// lattice.  Each lattice keeps the grid and summation order of its own
// diagnostics, so the results are bitwise those of lb_diagnostics.
struct BatchDiag {
    double *partial;         // the lattice's block partial sums
    int gx, gy, seg, pad;    // its diagnostics grid (diag_grid)
};

template <typename S>
__global__ void __launch_bounds__(kBlockThreads, kBlocksPerSm<float>)
    k_batch_diag(const BatchDesc *__restrict__ d, const BatchDiag *__restrict__ dd, const int *__restrict__ prefix, int n,
                 unsigned long long t)
{
    extern __shared__ __align__(128) unsigned char smem[];
    // the lattice of this block: the last m with prefix[m] <= blockIdx.x
    const int blk = blockIdx.x;
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= blk) lo = mid;
        else hi = mid;
    }
    const BatchDesc &bd = d[lo];
    const BatchDiag &g = dd[lo];
    __shared__ KP<float> sk;  // the lattice's parameters
    for (int w = threadIdx.x; w < (int)(sizeof(KP<float>) / 4); w += blockDim.x)
        reinterpret_cast<uint32_t *>(&sk)[w] = reinterpret_cast<const uint32_t *>(&bd.k)[w];
    __syncthreads();
    const int local = blk - prefix[lo];
    const int cur = (bd.parity0 + (int)(t & 1ULL)) & 1;  // the lattice's current buffer after t batch steps
    diag_block<S, float>(sk, (const S *)bd.buf[cur], g.partial, (double *)bd.buf[cur ^ 1], g.seg, local % g.gx,
                         local / g.gx, g.gx, reinterpret_cast<float *>(smem));
}

// out: one slot of slot_doubles per lattice, its NSUM sums and, 128 bytes in,
// the lattice's status word
__global__ void __launch_bounds__(256) k_batch_diag_final(const BatchDesc *__restrict__ d,
                                                          const BatchDiag *__restrict__ dd, double *__restrict__ out,
                                                          int slot_doubles, unsigned long long t)
{
    const int m = blockIdx.x / kDiagTasks, task = blockIdx.x % kDiagTasks;
    const BatchDesc &bd = d[m];
    const int cur = (bd.parity0 + (int)(t & 1ULL)) & 1;
    double *res = out + (size_t)m * slot_doubles;
    diag_task<float>(bd.k, task, dd[m].partial, dd[m].gx * dd[m].gy, (const double *)bd.buf[cur ^ 1], res);
    if (task == 0 && threadIdx.x == 0) *reinterpret_cast<int *>(res + 16) = *bd.status;
}

// T steps of every lattice of a batch on tiles or strips (lb_tile.cuh): the
// tiles of all lattices numbered by a prefix sum, one block each.  The pass
// takes the batch from step t on; `flip` says which buffer holds that state.
// Shared memory: the block's slots, then the lattice's parameters.  The plan is
// tile_plan's for the tiles of all lattices together.  With three
// batches on streams of their own, per step: 40 lattices of 64 to 128 columns
// in FP32 19.6 us in single steps, 15.2 us on strips of two steps; 64 annuli of
// 32 to 512 rows and columns in FP16 156 us with 4-row segments, 120 us in single
// steps, 105 us on strips of four (19.1 and 148 us for one batch alone, whose
// last wave nothing fills).  Bound as the single
// lattice's strips, and by the columns that a window of a narrow lattice leaves
// empty (a fifth of them in the first batch).
template <typename S, bool kStrip>
__global__ void __maxnreg__(kTileRegs<S>)
    k_batch_tiles(const BatchDesc *__restrict__ d, const int *__restrict__ prefix, int n, int total, int T,
                  unsigned long long t, int flip, int kp_off, int rev)
{
    extern __shared__ __align__(128) unsigned char smem[];
    grid_dependency_trigger();
    const int lane = threadIdx.x & 31;
    const int item = rev ? total - 1 - (int)blockIdx.x : (int)blockIdx.x;
    const int lo = batch_instance(prefix, n, item, lane);
    const BatchDesc *bd = d + lo;
    {
        const uint32_t *s = reinterpret_cast<const uint32_t *>(&bd->k);
        uint32_t *o = reinterpret_cast<uint32_t *>(smem + kp_off);
        for (int w = threadIdx.x; w < (int)(sizeof(KP<float>) / 4); w += blockDim.x) o[w] = s[w];
    }
    if (threadIdx.x < 2)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                         (unsigned long long)bd->map64[threadIdx.x])
                     : "memory");
    __syncthreads();
    const KP<float> &k = *reinterpret_cast<const KP<float> *>(smem + kp_off);
    const TileShape sh = bd->tiles;
    const int local = item - prefix[lo], cur = (bd->parity0 + flip) & 1;
    const CUtensorMap *map = reinterpret_cast<const CUtensorMap *>(bd->map64[cur]);
    S *dst = (S *)bd->buf[cur ^ 1];
    if constexpr (kStrip)
        strip_steps<S, sizeof(S) != 4>(k, map, dst, sh, T, local % sh.nw, local / sh.nw, bd->step0 + t, bd->status, smem);
    else tile_steps<S>(k, map, dst, sh, T, local % sh.nw, local / sh.nw, bd->step0 + t, bd->status, smem);
}

// Self-test of the bounded waits: one warp waits on an mbarrier that nothing
// arrives at, for `polls` polls of the same bounded wait the TMA rings use;
// the timeout must reach the status word as it does for a row that never
// arrives.  Nothing is in flight when the kernel ends.
__global__ void k_wait_selftest(int *status, int polls)
{
    __shared__ __align__(8) unsigned long long bar;
    const uint32_t b = smem_u32(&bar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    const bool ok = mbar_wait_bounded(b, 0u, polls);
    if (!__all_sync(FULL, ok) && threadIdx.x == 0) atomicExch(status, (int)LB_ERR_TIMEOUT);
}

int nwindows2(int nr) { return (nr + 63) / 64; }

// random bits of the stochastic rounding differ from step to step
uint32_t step_salt(unsigned long long step) { return salt_of(step); }

template <typename S>
size_t tma_smem_bytes(int wpb)
{
    return (size_t)wpb * (kTmaStages * TmaGeom<S>::stage_bytes + 128);
}

// The dynamic shared-memory limit of a kernel is a per-device attribute:
// set it once on every device that launches the kernel (devices 0..63;
// beyond that it is set at every launch).
template <typename K>
cudaError_t smem_limit_once(K kernel, int bytes, std::atomic<unsigned long long> &done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ULL << dev : 0ULL;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// Launch configuration with programmatic stream serialisation (see
// grid_dependency_trigger_and_wait)
void pdl_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, dim3 grid, dim3 block, size_t smem,
                cudaStream_t s)
{
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

int nwindows64(int nr) { return (nr + 31) / 32; }
constexpr int kMaxRows64 = 32;  // rows of a block of the FP64 step (its fields stay within 48 KB of shared memory)

// A row goes to two warps while a block has at most two rows.
int split64(int rows) { return rows <= 2 ? 2 : 1; }

// Estimated cycles of an FP64 step on blocks of `rows` rows: the FP64
// instructions of a block's busiest scheduler (tasks and items go round the
// four), 64 cycles each, 76 with all four busy, or the sum over the blocks of
// an SM where there are several.  Within 10 % of the measured times, less 2.6
// us per launch, on nine sizes from 20 x 84 to 1024 x 1024.
double cycles64(const HostParams &h, int rows, int sms)
{
    const int tasks = rows + (2 * rows + 31) / 32 + 1, items = rows * split64(rows);
    const double node = split64(rows) == 2 ? 194.0 : 306.0;
    const double alone = 33.0 * ((tasks + 3) / 4) + node * ((items + 3) / 4);
    const double all = (33.0 * tasks + node * items) / 4.0;
    const double per_sm = (double)nwindows64(h.nr) * ((h.nz + rows - 1) / rows) / sms;
    return std::max((items < 4 ? 64.0 : 76.0) * alone, 76.0 * all * (per_sm <= 3.0 ? std::ceil(per_sm) : per_sm + 0.3));
}

// SMs of the current device (152 on GB300; also the answer without a device)
int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess || sms <= 0) {
        cudaGetLastError();  // clear the error of a query without a device
        return 152;
    }
    return sms;
}

template <typename S, typename C>
cudaError_t step_t(const HostParams &h, const Launch &l, const void *src, void *dst, unsigned long long step,
                   const void *tmap, int *status, cudaStream_t s)
{
    const KP<C> k = make_kp<C>(h);
    const int wpb = l.warps_per_block;
    const int seg = l.seg_rows;
    if constexpr (std::is_same<C, double>::value) {
        const int nwin = nwindows64(h.nr), rows = std::min(seg, kMaxRows64);
        const long long blocks = (long long)nwin * ((h.nz + rows - 1) / rows);
        if (blocks > INT_MAX) return cudaErrorInvalidValue;
        // A lattice of at most three blocks per SM asks for the shared memory
        // with which just that many fit: the blocks of the next step, which
        // come early (programmatic dependent launch), would otherwise gather
        // on some SMs and leave others idle (70 x 96: 28 us per step, 11.7 us
        // with the limit; 14.4 us with plain launches)
        size_t smem = (size_t)(rows + 2) * 4 * kFields64Cols * sizeof(double);
        const int sms = sm_count(), per_sm = (int)std::min<long long>((blocks + sms - 1) / sms, 4);
        if (per_sm <= 3) smem = std::max(smem, (size_t)(kSmemPerSm / (per_sm + 1) - 1024 + 256));
        static std::atomic<unsigned long long> attr_set{0};
        cudaError_t e = smem_limit_once(k_step64, kMaxSmem, attr_set);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute pdl[1];
        pdl_config(cfg, pdl, dim3((unsigned)blocks), dim3(32 * wpb), smem, s);
        e = cudaLaunchKernelEx(&cfg, k_step64, k, make_walls64(k), (const double *)src, (double *)dst,
                                           rows, nwin, split64(rows));
        if (e != cudaSuccess) return e;
    } else {
        const int nwin2 = nwindows2(h.nr);
        dim3 grid((nwin2 + wpb - 1) / wpb, (h.nz + seg - 1) / seg);
        if (tmap && (l.use_tma == 2 || k.pinned)) {
            const size_t sm = ring_smem_bytes<S>(wpb);
            static std::atomic<unsigned long long> attr_set{0}, pinned_set{0};
            cudaError_t e = smem_limit_once(k_step3_tma<S, false>, (int)ring_smem_bytes<S>(8), attr_set);
            if (e == cudaSuccess) e = smem_limit_once(k_step3_tma<S, true>, (int)ring_smem_bytes<S>(8), pinned_set);
            if (e != cudaSuccess) return e;
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute pdl[1];
            pdl_config(cfg, pdl, grid, dim3(32 * wpb), sm, s);
            e = cudaLaunchKernelEx(&cfg, k.pinned ? k_step3_tma<S, true> : k_step3_tma<S, false>, k,
                                   *(const CUtensorMap *)tmap, (const S *)src, (S *)dst, seg, nwin2, step_salt(step),
                                   status, (int)(step & 1ULL));
            if (e != cudaSuccess) return e;
        } else if (tmap && l.use_tma) {
            const size_t sm = tma_smem_bytes<S>(wpb);
            static std::atomic<unsigned long long> attr_set{0};
            cudaError_t e = smem_limit_once(k_step2_tma<S>, (int)tma_smem_bytes<S>(8), attr_set);
            if (e != cudaSuccess) return e;
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute pdl[1];
            pdl_config(cfg, pdl, grid, dim3(32 * wpb), sm, s);
            e = cudaLaunchKernelEx(&cfg, k_step2_tma<S>, k, *(const CUtensorMap *)tmap, (const S *)src, (S *)dst,
                                   seg, nwin2, step_salt(step), status, (int)(step & 1ULL));
            if (e != cudaSuccess) return e;
        } else {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute pdl[1];
            pdl_config(cfg, pdl, grid, dim3(32 * wpb), 0, s);
            cudaError_t e = cudaLaunchKernelEx(&cfg, k_step2<S>, k, (const S *)src, (S *)dst, seg, nwin2,
                                               step_salt(step), (int)(step & 1ULL));
            if (e != cudaSuccess) return e;
        }
    }
    return cudaGetLastError();
}

template <typename S, typename C>
cudaError_t fields_t(const HostParams &h, const void *src, double *out, int row0, int row1, int only_ux, cudaStream_t s)
{
    const int nbx = (h.nr + kBlockCols - 1) / kBlockCols;
    // 16 rows, 8 on few blocks (1024 x 2048 FP64: 941 us as lb_stream_function takes
    // them, 977 with 8 throughout)
    int rows = 2 * kBlockChunk;
    auto blocks = [&]() { return (long long)nbx * ((row1 - row0 + rows - 1) / rows); };
    while (rows > kBlockChunk && blocks() < 4 * sm_count()) rows /= 2;
    if (blocks() > INT_MAX) return cudaErrorInvalidValue;
    k_fields<S, C><<<(unsigned)blocks(), kBlockThreads, kBlockSmem<C>, s>>>(make_kp<C>(h), (const S *)src, out, row0, row1,
                                                                            nbx, rows, only_ux);
    return cudaGetLastError();
}

// The two launches of a diagnostics: strips holds 4 (nr + nz) doubles.
template <typename S, typename C>
cudaError_t diag_t(const HostParams &h, const DiagGrid &g, const void *src, double *partial, double *strips,
                   double *result, cudaStream_t s)
{
    const KP<C> k = make_kp<C>(h);
    k_diag<S, C><<<g.gx * g.gy, kBlockThreads, kBlockSmem<C>, s>>>(k, (const S *)src, partial, strips, g.seg, g.gx);
    k_diag_final<C><<<kDiagTasks, 256, 0, s>>>(k, partial, g.gx * g.gy, strips, result);
    return cudaGetLastError();
}

int blocks_for(long long n) { return (int)std::min<long long>((n + 255) / 256, 4096); }

}  // namespace

size_t storage_bytes(int storage)
{
    switch (storage) {
        case ST_FP64: return 8;
        case ST_FP32: return 4;
        default: return 2;
    }
}

Launch default_launch(const HostParams &p)
{
    Launch l;
    if (p.storage == ST_FP64) {
        // the rows with the least estimated time (41 x 41: 1, 10.9 us per
        // step, 2 rows 11.5, 4 rows 15.4; 256 x 512: 4, 88.5 us, 3 rows 97, 8
        // rows 97.5); eight warps while blocks run one or a few to an SM
        const int sms = sm_count();
        l.seg_rows = 1;
        for (int rows : {2, 3, 4, 6, 8, 12, 16})
            if (cycles64(p, rows, sms) < cycles64(p, l.seg_rows, sms)) l.seg_rows = rows;
        l.warps_per_block = (long long)nwindows64(p.nr) * ((p.nz + l.seg_rows - 1) / l.seg_rows) <= 3 * sms ? 8 : 4;
        l.use_tma = 0;
        return l;
    }
    l.warps_per_block = 1;
    l.use_tma = 2;
    // 4-row segments in FP32, 6 in 16-bit storage (measured on the 1024 x 2048
    // lattice; short segments balance the last wave, and their halo rows are
    // re-read from L2); fewer rows when the lattice would otherwise leave SMs
    // idle
    const int nwin = nwindows2(p.nr);
    int seg = p.storage == ST_FP32 ? 4 : 6;
    const long long warps = (long long)nwin * ((p.nz + seg - 1) / seg);
    const long long want = 16LL * sm_count();  // about two waves of resident warps
    if (warps < want) {
        const long long segs = (want + nwin - 1) / nwin;
        seg = (int)((p.nz + segs - 1) / segs);
        if (seg < 4) seg = 4;
    }
    if ((p.nz + seg - 1) / seg > 65535) seg = (p.nz + 65534) / 65535;  // grid.y limit
    l.seg_rows = seg;
    return l;
}

#define DISPATCH(p, CALL)                                                   \
    switch ((p).storage) {                                                  \
        case ST_FP64: { using S = double; using C = double; return CALL; }   \
        case ST_FP32: { using S = float; using C = float; return CALL; }     \
        case ST_BF16: { using S = __nv_bfloat16; using C = float; return CALL; } \
        case ST_FP16: { using S = __half; using C = float; return CALL; }    \
        default: return cudaErrorInvalidValue;                              \
    }

cudaError_t launch_step(const HostParams &p, const Launch &l, const void *src, void *dst, unsigned long long step,
                        const void *tmap, int *status, cudaStream_t s)
{
    DISPATCH(p, (step_t<S, C>(p, l, src, dst, step, tmap, status, s)));
}

bool step_is_pinned(const HostParams &h) { return pinned_order(h); }

int ring_cols(int storage) { return 64 + 2 * (16 / (int)storage_bytes(storage)); }

// Tensor map of one distribution buffer for the TMA row fetches: a 3-D view
// [19 planes][nz rows][pitch columns], box of box_cols x 1 x 19
// (ring_cols(storage) for the row rings, 64 for the tiles).
cudaError_t make_tensor_map(const HostParams &p, void *buf, int box_cols, void *map_out)
{
    if (p.storage == ST_FP64) return cudaErrorInvalidValue;
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    const int es = (int)storage_bytes(p.storage);
    const CUtensorMapDataType dt = p.storage == ST_FP32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : p.storage == ST_FP16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                          : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    const cuuint64_t dims[3] = {(cuuint64_t)p.pitch, (cuuint64_t)p.nz, (cuuint64_t)NQ};
    const cuuint64_t strides[2] = {(cuuint64_t)p.pitch * es, (cuuint64_t)p.plane * es};
    const cuuint32_t box[3] = {(cuuint32_t)box_cols, 1u, (cuuint32_t)NQ};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    CUresult r = encode((CUtensorMap *)map_out, dt, 3, buf, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

namespace {

// The tiles of a lattice for passes of up to T steps: windows of 64 columns
// whose starts lie on 16-byte boundaries (TMA), so the column margin is T
// rounded up to 2 columns in FP32, 4 in 16-bit storage.
TileShape tile_shape(const HostParams &h, int T, int rows)
{
    TileShape sh;
    sh.rows = rows;
    sh.rm = T;
    sh.cm = h.storage == ST_FP32 ? (T + 1) / 2 * 2 : (T + 3) / 4 * 4;
    sh.rs = rows - 2 * T;
    sh.cs = 64 - 2 * sh.cm;
    sh.nw = h.nr <= 64 ? 1 : (h.nr - 64 + sh.cs - 1) / sh.cs + 1;
    return sh;
}

// Tiles along z, and in all.
int tiles_along(const HostParams &h, const TileShape &sh)
{
    if (h.flow[0] == 2) return (h.nz + sh.rs - 1) / sh.rs;
    return h.nz <= sh.rows ? 1 : (h.nz - sh.rows + sh.rs - 1) / sh.rs + 1;
}
long long tile_count(const HostParams &h, int T, int rows)
{
    const TileShape sh = tile_shape(h, T, rows);
    return (long long)sh.nw * tiles_along(h, sh);
}

int tile_slot_bytes(int storage)
{
    return storage == ST_FP32 ? TileGeom<float>::slot_bytes : TileGeom<__half>::slot_bytes;
}

int tile_slots(bool strip, int T, int rows, int warps) { return strip ? 2 * warps + 2 * T : rows + T - 1; }

constexpr int kBatchKpBytes = (int)((sizeof(KP<float>) + 127) / 128 * 128);

// Blocks of a pass that fit on an SM at once (shared memory with 1 KB of it per
// block for the system, registers).
int tiles_per_sm(int storage, int slots, int warps, bool batch)
{
    const int smem = slots * tile_slot_bytes(storage) + 128 + (batch ? kBatchKpBytes : 0);
    if (smem > kMaxSmem) return 0;
    const int regs = storage == ST_FP32 ? kTileRegs<float> : kTileRegs<__half>;
    return std::min(kSmemPerSm / (smem + 1024), 65536 / (regs * 32 * warps));
}

// The lattices that share a pass, and their tiles at a common tile height.
struct Lattices {
    const HostParams *const *h;
    int n, storage;
    long long tiles(int T, int rows) const
    {
        long long sum = 0;
        for (int m = 0; m < n; ++m) sum += tile_count(*h[m], T, rows);
        return sum;
    }
    int max_rows() const
    {
        int r = 0;
        for (int m = 0; m < n; ++m) r = std::max(r, h[m]->nz);
        return r;
    }
};

// The smallest tile, in rows, with which all tiles are resident at once, two
// or more to an SM; 0 when there is none.
int resident_tile_rows(const Lattices &ls, int T, int warps, int sms)
{
    for (int rows = 2 * T + 1;; ++rows) {
        const int per_sm = tiles_per_sm(ls.storage, tile_slots(false, T, rows, warps), warps, ls.n > 1);
        if (per_sm < 2) return 0;
        if (ls.tiles(T, rows) <= (long long)sms * per_sm) return rows;
    }
}

// The shortest strips, in rows, that make up at most `waves` waves of resident
// blocks; whole lattices where even those are more.
int strip_rows(const Lattices &ls, int T, int warps, int waves, int sms)
{
    const long long most = (long long)waves * sms * tiles_per_sm(ls.storage, tile_slots(true, T, 0, warps), warps, ls.n > 1);
    int lo = 2 * T + 1, hi = ls.max_rows() + 2 * T;
    while (lo < hi) {
        const int mid = lo + (hi - lo) / 2;
        if (ls.tiles(T, mid) <= most) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

template <typename S>
cudaError_t tile_t(const HostParams &h, const TileLaunch &l, const void *tmap, void *dst, unsigned long long step,
                   int *status, unsigned *begun, unsigned pass, cudaStream_t s)
{
    const KP<float> k = make_kp<float>(h);
    const int rev = (int)(pass & 1u);  // the block order alternates from pass to pass
    static std::atomic<unsigned long long> tile_set{0}, strip_set{0};
    cudaError_t e = smem_limit_once(k_tiles<S, false>, kMaxSmem, tile_set);
    if (e == cudaSuccess) e = smem_limit_once(k_tiles<S, true>, kMaxSmem, strip_set);
    if (e != cudaSuccess) return e;
    const TileShape sh = tile_shape(h, l.T, l.rows);
    const long long blocks = (long long)sh.nw * tiles_along(h, sh);
    const size_t smem = tile_smem_bytes<S>(tile_slots(l.strip, l.T, l.rows, l.warps));
    const bool two = l.strip && l.parts == 2 && blocks >= 2;
    for (int p = 0; p < l.parts; ++p) {
        const int q = rev ? l.parts - 1 - p : p;  // the parts in the order of their blocks
        const int first = (int)(blocks * q / l.parts), count = (int)(blocks * (q + 1) / l.parts) - first;
        if (count < 1) continue;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute pdl[1];
        pdl_config(cfg, pdl, dim3(count), dim3(32 * l.warps), smem, s);
        e = cudaLaunchKernelEx(&cfg, l.strip ? k_tiles<S, true> : k_tiles<S, false>, k, *(const CUtensorMap *)tmap,
                               (S *)dst, sh, l.T, first, step, status, rev, two ? 1 + p : 0, begun, pass);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

TileLaunch plan_tiles(const Lattices &ls, int T)
{
    const int sms = sm_count();
    const bool fp32 = ls.storage == ST_FP32;
    const int W = fp32 ? 6 : 8;
    TileLaunch l{T, 0, W, 0, 1};
    if (T == 0) {  // the best number of steps
        l.T = 3;
        l.rows = resident_tile_rows(ls, 3, W, sms);
        if (fp32 && (l.rows == 0 || l.rows > 9)) {
            l.T = 2;
            l.rows = resident_tile_rows(ls, 2, W, sms);
        }
        if (l.rows == 0) l.T = fp32 ? 2 : 4;
    } else {
        l.rows = resident_tile_rows(ls, T, W, sms);
    }
    if (l.rows) return l;
    l.strip = 1;
    l.rows = strip_rows(ls, l.T, W, 1, sms);
    if (l.rows > (fp32 ? 40 : 60)) {
        l.warps = 4;
        l.rows = strip_rows(ls, l.T, l.warps, 1, sms);
    }
    return l;
}

}  // namespace

// Which pass a lattice takes, from its size alone; times per step on one GB300
// over 24 sizes from 20 x 84 to 1024 x 2048, all tiles, strips, T and warps
// that fit (the chosen ones lie within 5 % of the best, 8 % at two sizes):
// - Resident tiles while the lattice fits, as small as that allows.  FP32: three
//   steps while the tiles are small (100 x 100: 2.45 us, two steps 2.58, four
//   2.79), two steps from ten rows on (180 x 360: 3.77 against 4.00 us).  In
//   16-bit storage, whose margins are 4 columns for up to four steps, three
//   (100 x 100: 2.89 us, two 2.99, four 3.03; 400 x 400: 5.90, 6.04, 5.98).
// - Strips beyond (512 x 512 FP32: 7.5 us, tiles 8.0).  FP32: two steps (1024 x
//   2048: 39.4 us as one launch; three 45.2, four 42.5; 512 x 1024: 12.5, 12.7,
//   12.8).  16-bit: four (1024 x 2048 FP16: 41.5 us; three 43.0, two 43.1; 512 x
//   1024: 12.2, 12.8, 12.8; all with cheaper rounding words, 44.6 and 13.4 now).
//   Six (eight) warps per block while the strips are short, four and one more
//   block per SM from 40 (60) rows on (512 x 1024 FP32: 12.5 against 13.1 us; 1024
//   x 2048: 42.4 against 39.4; two, three or five warps: 8-20 % slower).
// - FP32 strips of more than 64 rows go out as two launches, half of the strips
//   each, cut for two waves in all (k_tiles; 1024 x 2048: 40.6 us per step, as one
//   launch of two waves 41.2; 768 x 1536: 23.9, 24.3; 2048 x 2048: 76.1, 77.6).
TileLaunch tile_plan(const HostParams &h, int T)
{
    const HostParams *one = &h;
    const Lattices ls{&one, 1, h.storage};
    TileLaunch l = plan_tiles(ls, T);
    if (l.strip && h.storage == ST_FP32 && l.T == 2 && l.rows > 64) {
        l.parts = 2;
        l.rows = strip_rows(ls, l.T, l.warps, 2, sm_count());
    }
    return l;
}

// The lattice's tiles under a pass made for the whole batch: strips of equal
// length, no longer than the pass's.
static TileShape batch_tiles(const HostParams &h, const TileLaunch &l)
{
    TileShape sh = tile_shape(h, l.T, l.rows);
    const int nt = tiles_along(h, sh), rows = h.flow[0] == 2 ? h.nz : std::max(1, h.nz - 2 * l.T);
    return nt > 1 || h.flow[0] == 2 ? tile_shape(h, l.T, (rows + nt - 1) / nt + 2 * l.T) : sh;
}

// How much of the time of a pass on strips its resident blocks are busy, with
// the strips started in order as blocks end; a strip takes its rows and the
// filling of its ring.
static double strips_busy(const std::vector<const HostParams *> &hs, const TileLaunch &l, int sms)
{
    const long long resident =
        (long long)sms * tiles_per_sm(hs[0]->storage, tile_slots(true, l.T, 0, l.warps), l.warps, hs.size() > 1);
    std::priority_queue<double, std::vector<double>, std::greater<double>> ends;
    double work = 0.0, end = 0.0;
    for (const HostParams *h : hs) {
        const TileShape sh = batch_tiles(*h, l);
        const bool per = h->flow[0] == 2;
        for (int t = 0, nt = tiles_along(*h, sh); t < nt; ++t) {
            const int rows = per ? std::min(sh.rs, h->nz - t * sh.rs) + 2 * sh.rm : std::min(sh.rows, h->nz - t * sh.rs);
            for (int w = 0; w < sh.nw; ++w) {
                double at = rows + l.warps;
                work += at;
                if ((long long)ends.size() >= resident) {
                    at += ends.top();
                    ends.pop();
                }
                ends.push(at);
                end = std::max(end, at);
            }
        }
    }
    return work / (end * resident);
}

// The pass of a batch: tile_plan's for the tiles of all lattices together, but
// single steps (T = 1, work items of equal length) where a few tall lattices
// would keep the blocks waiting.  Per step, annuli of 32 to 512 columns and rows,
// one batch alone and one of three side by side, which fill each other's gaps:
// FP16, 128 of them (0.58 busy) 329 and 209 us on strips, 261 and 242 in single
// steps, 64 (0.73) 148 and 105, 135 and 120; FP32, 96 (0.53) 265 and 158, 228 and
// 215.  (One launch per step of 4-row items, before the strips: 324 and 316, 163
// and 156, 284 and 277.)
TileLaunch tile_plan_batch(const HostParams *const *h, int n)
{
    std::vector<const HostParams *> tiled;  // pinned lattices take launches of their own
    for (int m = 0; m < n; ++m)
        if (!pinned_order(*h[m])) tiled.push_back(h[m]);
    if (tiled.empty()) tiled.assign(h, h + n);
    TileLaunch l = plan_tiles(Lattices{tiled.data(), (int)tiled.size(), h[0]->storage}, 0);
    if (l.strip && strips_busy(tiled, l, sm_count()) < (h[0]->storage == ST_FP32 ? 0.5 : 0.6)) l.T = 1;
    return l;
}

cudaError_t launch_tile(const HostParams &p, const TileLaunch &l, const void *tmap, void *dst, unsigned long long step,
                        int *status, unsigned *begun, unsigned pass, cudaStream_t s)
{
    switch (p.storage) {
        case ST_FP32: return tile_t<float>(p, l, tmap, dst, step, status, begun, pass, s);
        case ST_BF16: return tile_t<__nv_bfloat16>(p, l, tmap, dst, step, status, begun, pass, s);
        case ST_FP16: return tile_t<__half>(p, l, tmap, dst, step, status, begun, pass, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_wait_selftest(int *status, int polls, cudaStream_t s)
{
    k_wait_selftest<<<1, 32, 0, s>>>(status, polls);
    return cudaGetLastError();
}

cudaError_t launch_psi(const double *ux, double *psi, double *rowmax, int nrows, int nr, double r0, cudaStream_t s)
{
    if (nrows < 1) return cudaSuccess;
    k_psi<<<(nrows + 3) / 4, 128, 0, s>>>(ux, psi, rowmax, nrows, nr, r0);
    return cudaGetLastError();
}

cudaError_t launch_fields(const HostParams &p, const void *src, double *out, int row0, int row1, bool only_ux,
                          cudaStream_t s)
{
    DISPATCH(p, (fields_t<S, C>(p, src, out, row0, row1, only_ux, s)));
}

// Blocks of 32 rows, fewer while there would be less than two blocks per SM,
// more where there would be more than max_blocks.
DiagGrid diag_grid(const HostParams &p, int max_blocks)
{
    DiagGrid g;
    g.gx = (p.nr + kBlockCols - 1) / kBlockCols;
    // 32 rows, down to 8 on a lattice of less than two blocks per SM, 4 where
    // even those are less than a quarter of the SMs (512 x 512 FP32: 8 rows 41 us,
    // 4 rows 54, 16 rows 43; 41 x 41 FP64: 65, 48, 97; 64 annuli in one batch: 8
    // rows 508 us, 4 rows 743, whose blocks form 6 rows of fields each); not on the
    // longest, whose sums have to fit beside their strips (lb_diagnostics_static)
    g.seg = 32;
    auto blocks = [&]() { return (long long)g.gx * ((p.nz + g.seg - 1) / g.seg); };
    while (p.nr + p.nz <= 16384 && ((g.seg > 8 && blocks() < 304) || (g.seg == 8 && blocks() < 38))) g.seg /= 2;
    if ((long long)g.gx * ((p.nz + g.seg - 1) / g.seg) > max_blocks) {
        const int segs = std::max(1, max_blocks / g.gx);
        g.seg = (p.nz + segs - 1) / segs;
    }
    g.gy = (p.nz + g.seg - 1) / g.seg;
    return g;
}

cudaError_t launch_diag(const HostParams &p, const void *src, double *partial, double *strips, double *result,
                        cudaStream_t s)
{
    const DiagGrid g = diag_grid(p, MAX_DIAG_BLOCKS);
    if ((long long)g.gx * g.gy > MAX_DIAG_BLOCKS) return cudaErrorInvalidValue;
    DISPATCH(p, (diag_t<S, C>(p, g, src, partial, strips, result, s)));
}

#define DISPATCH_S(p, CALL)                                         \
    switch ((p).storage) {                                          \
        case ST_FP64: { using S = double; CALL; break; }            \
        case ST_FP32: { using S = float; CALL; break; }             \
        case ST_BF16: { using S = __nv_bfloat16; CALL; break; }     \
        case ST_FP16: { using S = __half; CALL; break; }            \
        default: return cudaErrorInvalidValue;                      \
    }

cudaError_t launch_init_fields(const HostParams &p, const double *fields, void *dst, int row0, int row1,
                               cudaStream_t s)
{
    const int nb = blocks_for((long long)(row1 - row0) * p.nr);
    DISPATCH_S(p, (k_init_fields<S><<<nb, 256, 0, s>>>(p, fields, (S *)dst, row0, row1)));
    return cudaGetLastError();
}

cudaError_t launch_export(const HostParams &p, const void *src, double *out, int row0, int row1, cudaStream_t s)
{
    const int nb = blocks_for((long long)(row1 - row0) * p.nr);
    DISPATCH_S(p, (k_export<S><<<nb, 256, 0, s>>>(p, (const S *)src, out, row0, row1)));
    return cudaGetLastError();
}

cudaError_t launch_import(const HostParams &p, const double *in, void *dst, int row0, int row1, cudaStream_t s)
{
    const int nb = blocks_for((long long)(row1 - row0) * p.nr);
    DISPATCH_S(p, (k_import<S><<<nb, 256, 0, s>>>(p, in, (S *)dst, row0, row1)));
    return cudaGetLastError();
}

}  // namespace lbk

namespace lbk {

size_t batch_desc_bytes() { return sizeof(BatchDesc); }
size_t batch_ctl_bytes() { return sizeof(BatchCtl); }

int batch_tile_count(const HostParams &h, const TileLaunch &l)
{
    if (pinned_order(h)) return 0;
    const TileShape sh = batch_tiles(h, l);
    return sh.nw * tiles_along(h, sh);
}

int batch_items(const HostParams &h, int seg_rows)
{
    return nwindows2(h.nr) * ((h.nz + seg_rows - 1) / seg_rows);
}

cudaError_t batch_fill_desc(const HostParams &h, void *buf0, void *buf1, unsigned long long step0, int parity0,
                            int seg_rows, const TileLaunch &l, int *status, void *out)
{
    BatchDesc d;
    std::memset(&d, 0, sizeof(d));
    cudaError_t e = make_tensor_map(h, buf0, ring_cols(h.storage), d.map[0]);
    if (e == cudaSuccess) e = make_tensor_map(h, buf1, ring_cols(h.storage), d.map[1]);
    if (e == cudaSuccess) e = make_tensor_map(h, buf0, 64, d.map64[0]);
    if (e == cudaSuccess) e = make_tensor_map(h, buf1, 64, d.map64[1]);
    if (e != cudaSuccess) return e;
    d.k = make_kp<float>(h);
    d.buf[0] = buf0;
    d.buf[1] = buf1;
    d.status = status;
    d.step0 = step0;
    d.parity0 = parity0;
    d.nwin2 = nwindows2(h.nr);
    d.seg_rows = seg_rows;
    d.tiles = batch_tiles(h, l);
    std::memcpy(out, &d, sizeof(d));
    return cudaSuccess;
}

cudaError_t batch_prepare(int storage)
{
    switch (storage) {
        case ST_FP32: {
            cudaError_t e = cudaFuncSetAttribute(k_batch3<float, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)batch3_smem_bytes<float, 4>(8));
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_batch3p<float, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)batch3_smem_bytes<float, 3>(8));
            if (e != cudaSuccess) return e;
            return cudaFuncSetAttribute(k_batch3<float, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)batch3_smem_bytes<float, 3>(8));
        }
        case ST_FP16: {
            cudaError_t e = cudaFuncSetAttribute(k_batch3p<__half, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)batch3_smem_bytes<__half>(8));
            if (e != cudaSuccess) return e;
            return cudaFuncSetAttribute(k_batch3<__half, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)batch3_smem_bytes<__half>(8));
        }
        case ST_BF16: {
            cudaError_t e = cudaFuncSetAttribute(k_batch3p<__nv_bfloat16, 4>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)batch3_smem_bytes<__nv_bfloat16>(8));
            if (e != cudaSuccess) return e;
            return cudaFuncSetAttribute(k_batch3<__nv_bfloat16, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)batch3_smem_bytes<__nv_bfloat16>(8));
        }
        default: return cudaErrorInvalidValue;
    }
}

int batch_grid(int storage, int wpb)
{
    int dev = 0, sms = 152, per = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t sm = (size_t)wpb * sizeof(KP<float>);
    switch (storage) {
        case ST_FP32: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch<float>, 32 * wpb, sm); break;
        case ST_FP16: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch<__half>, 32 * wpb, sm); break;
        case ST_BF16: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch<__nv_bfloat16>, 32 * wpb, sm); break;
        default: per = 1;
    }
    return sms * (per > 0 ? per : 1);
}

cudaError_t batch_resident_warps(int storage, int row_fetch, int wpb, int *out)
{
    if (row_fetch == 1) {
        *out = batch_grid(storage, wpb) * wpb;
        return cudaSuccess;
    }
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = batch_prepare(storage);
    if (e != cudaSuccess) return e;
    if (row_fetch == 5) {
        switch (storage) {
            case ST_FP32:
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch3p<float, 3>, 32 * wpb,
                                                                  batch3_smem_bytes<float, 3>(wpb));
                break;
            case ST_FP16:
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch3p<__half, 4>, 32 * wpb,
                                                                  batch3_smem_bytes<__half>(wpb));
                break;
            case ST_BF16:
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch3p<__nv_bfloat16, 4>, 32 * wpb,
                                                                  batch3_smem_bytes<__nv_bfloat16>(wpb));
                break;
            default: return cudaErrorInvalidValue;
        }
        *out = sms * per * wpb;
        return e;
    }
    switch (storage) {
        case ST_FP32:
            if (row_fetch == 4)
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch3<float, 3>, 32 * wpb,
                                                                  batch3_smem_bytes<float, 3>(wpb));
            else
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch3<float, 4>, 32 * wpb,
                                                                  batch3_smem_bytes<float, 4>(wpb));
            break;
        case ST_FP16:
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch3<__half, 4>, 32 * wpb,
                                                              batch3_smem_bytes<__half>(wpb));
            break;
        case ST_BF16:
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch3<__nv_bfloat16, 4>, 32 * wpb,
                                                              batch3_smem_bytes<__nv_bfloat16>(wpb));
            break;
        default: return cudaErrorInvalidValue;
    }
    *out = sms * per * wpb;
    return e;
}

// One step of the pinned lattices of a batch, whatever its row fetch.
template <typename S>
static cudaError_t batch_pinned_t(const BatchDesc *d, const int *prefix, int n, int total, const BatchCtl *ctl, int wpb,
                                  unsigned long long t0, int from_counter, cudaStream_t s)
{
    static std::atomic<unsigned long long> attr_set{0};
    cudaError_t e = smem_limit_once(k_batch3<S, 4, true>, (int)batch3_smem_bytes<S, 4>(8), attr_set);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute pdl[1];
    pdl_config(cfg, pdl, dim3((total + wpb - 1) / wpb), dim3(32 * wpb), batch3_smem_bytes<S, 4>(wpb), s);
    return cudaLaunchKernelEx(&cfg, k_batch3<S, 4, true>, d, prefix, n, total, ctl, t0, from_counter, (int)(t0 & 1ULL));
}

cudaError_t launch_batch_pinned(int storage, const void *desc, const int *prefix, int n, int total, void *ctl, int wpb,
                                unsigned long long t0, int from_counter, cudaStream_t s)
{
    const BatchDesc *d = (const BatchDesc *)desc;
    const BatchCtl *c = (const BatchCtl *)ctl;
    switch (storage) {
        case ST_FP32: return batch_pinned_t<float>(d, prefix, n, total, c, wpb, t0, from_counter, s);
        case ST_FP16: return batch_pinned_t<__half>(d, prefix, n, total, c, wpb, t0, from_counter, s);
        case ST_BF16: return batch_pinned_t<__nv_bfloat16>(d, prefix, n, total, c, wpb, t0, from_counter, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_batch_persist(int storage, const void *desc, const int *prefix, int n, int total, int wpb,
                                 unsigned long long t0, int nsteps, int *done, cudaStream_t s)
{
    if (total < 1 || nsteps < 1) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(done, 0, (size_t)total * sizeof(int), s);
    if (e != cudaSuccess) return e;
    const BatchDesc *dd = (const BatchDesc *)desc;
    void *args[] = {(void *)&dd, (void *)&prefix, (void *)&n, (void *)&total, (void *)&t0, (void *)&nsteps,
                    (void *)&done};
    const dim3 grid((total + wpb - 1) / wpb), block(32 * wpb);
    switch (storage) {
        case ST_FP32:
            return cudaLaunchCooperativeKernel((const void *)k_batch3p<float, 3>, grid, block, args,
                                               batch3_smem_bytes<float, 3>(wpb), s);
        case ST_FP16:
            return cudaLaunchCooperativeKernel((const void *)k_batch3p<__half, 4>, grid, block, args,
                                               batch3_smem_bytes<__half>(wpb), s);
        case ST_BF16:
            return cudaLaunchCooperativeKernel((const void *)k_batch3p<__nv_bfloat16, 4>, grid, block, args,
                                               batch3_smem_bytes<__nv_bfloat16>(wpb), s);
        default: return cudaErrorInvalidValue;
    }
}

template <typename S>
static cudaError_t batch_tiles_t(const TileLaunch &l, int T, const BatchDesc *d, const int *prefix, int n, int total,
                                 unsigned long long t, int flip, cudaStream_t s)
{
    static std::atomic<unsigned long long> tile_set{0}, strip_set{0};
    cudaError_t e = smem_limit_once(k_batch_tiles<S, false>, kMaxSmem, tile_set);
    if (e == cudaSuccess) e = smem_limit_once(k_batch_tiles<S, true>, kMaxSmem, strip_set);
    if (e != cudaSuccess) return e;
    const int kp_off = (int)tile_smem_bytes<S>(tile_slots(l.strip, T, l.rows, l.warps));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute pdl[1];
    pdl_config(cfg, pdl, dim3(total), dim3(32 * l.warps), kp_off + sizeof(KP<float>), s);
    return cudaLaunchKernelEx(&cfg, l.strip ? k_batch_tiles<S, true> : k_batch_tiles<S, false>, d, prefix, n, total, T,
                              t, flip, kp_off, flip);
}

cudaError_t launch_batch_tiles(int storage, const TileLaunch &l, int T, const void *desc, const int *prefix, int n,
                               int total, unsigned long long t, int flip, cudaStream_t s)
{
    const BatchDesc *d = (const BatchDesc *)desc;
    switch (storage) {
        case ST_FP32: return batch_tiles_t<float>(l, T, d, prefix, n, total, t, flip, s);
        case ST_FP16: return batch_tiles_t<__half>(l, T, d, prefix, n, total, t, flip, s);
        case ST_BF16: return batch_tiles_t<__nv_bfloat16>(l, T, d, prefix, n, total, t, flip, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_batch_counter(void *ctl, unsigned long long value, int add, cudaStream_t s)
{
    k_batch_counter<<<1, 32, 0, s>>>((BatchCtl *)ctl, value, add);
    return cudaGetLastError();
}

cudaError_t launch_batch(int storage, int row_fetch, const void *desc, const int *prefix, int n, int total,
                         void *ctl, int wpb, int blocks, unsigned long long t0, int from_counter, cudaStream_t s)
{
    const int need = (total + wpb - 1) / wpb;
    if (need < 1) return cudaSuccess;
    const BatchDesc *dd = (const BatchDesc *)desc;
    const BatchCtl *cc = (const BatchCtl *)ctl;
    // the item order alternates with the step (inside a graph with the launch
    // index, t0 = j there): a step starts on the items the previous one wrote last
    const int rev = (int)(t0 & 1ULL);
    if (row_fetch == 3 || row_fetch == 4) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute pdl[1];
        switch (storage) {
            case ST_FP32:
                if (row_fetch == 4) {
                    pdl_config(cfg, pdl, dim3(need), dim3(32 * wpb), batch3_smem_bytes<float, 3>(wpb), s);
                    return cudaLaunchKernelEx(&cfg, k_batch3<float, 3>, dd, prefix, n, total, cc, t0, from_counter, rev);
                }
                pdl_config(cfg, pdl, dim3(need), dim3(32 * wpb), batch3_smem_bytes<float, 4>(wpb), s);
                return cudaLaunchKernelEx(&cfg, k_batch3<float, 4>, dd, prefix, n, total, cc, t0, from_counter, rev);
            case ST_FP16:
                pdl_config(cfg, pdl, dim3(need), dim3(32 * wpb), batch3_smem_bytes<__half>(wpb), s);
                return cudaLaunchKernelEx(&cfg, k_batch3<__half, 4>, dd, prefix, n, total, cc, t0, from_counter, rev);
            case ST_BF16:
                pdl_config(cfg, pdl, dim3(need), dim3(32 * wpb), batch3_smem_bytes<__nv_bfloat16>(wpb), s);
                return cudaLaunchKernelEx(&cfg, k_batch3<__nv_bfloat16, 4>, dd, prefix, n, total, cc, t0,
                                          from_counter, rev);
            default: return cudaErrorInvalidValue;
        }
    }
    const int grid = blocks < need ? blocks : need;
    const size_t sm = (size_t)wpb * sizeof(KP<float>);
    switch (storage) {
        case ST_FP32: k_batch<float><<<grid, 32 * wpb, sm, s>>>(dd, prefix, n, total, cc, t0, from_counter); break;
        case ST_FP16: k_batch<__half><<<grid, 32 * wpb, sm, s>>>(dd, prefix, n, total, cc, t0, from_counter); break;
        case ST_BF16:
            k_batch<__nv_bfloat16><<<grid, 32 * wpb, sm, s>>>(dd, prefix, n, total, cc, t0, from_counter);
            break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

size_t batch_diag_bytes() { return sizeof(BatchDiag); }

int batch_fill_diag(const HostParams &h, double *partial, void *out)
{
    const DiagGrid grid = diag_grid(h, MAX_DIAG_BLOCKS);
    BatchDiag g;
    std::memset(&g, 0, sizeof g);
    g.partial = partial;
    g.seg = grid.seg;
    g.gx = grid.gx;
    g.gy = grid.gy;
    std::memcpy(out, &g, sizeof g);
    const long long nb = (long long)g.gx * g.gy;
    return nb <= MAX_DIAG_BLOCKS ? (int)nb : -1;
}

cudaError_t launch_batch_diag(int storage, const void *desc, const void *bdiag, const int *bprefix, int n, int total,
                              unsigned long long t, double *out, int slot_doubles, cudaStream_t s)
{
    const BatchDesc *d = (const BatchDesc *)desc;
    const BatchDiag *dd = (const BatchDiag *)bdiag;
    switch (storage) {
        case ST_FP32: k_batch_diag<float><<<total, kBlockThreads, kBlockSmem<float>, s>>>(d, dd, bprefix, n, t); break;
        case ST_FP16: k_batch_diag<__half><<<total, kBlockThreads, kBlockSmem<float>, s>>>(d, dd, bprefix, n, t); break;
        case ST_BF16: k_batch_diag<__nv_bfloat16><<<total, kBlockThreads, kBlockSmem<float>, s>>>(d, dd, bprefix, n, t); break;
        default: return cudaErrorInvalidValue;
    }
    k_batch_diag_final<<<n * kDiagTasks, 256, 0, s>>>(d, dd, out, slot_doubles, t);
    return cudaGetLastError();
}

}  // namespace lbk

// ---- diagnostics without scratch memory from the caller ------------------------
//
// lb_diagnostics_static() evaluates the diagnostics of a state the caller
// holds in device memory, with no context and no scratch from the caller:
// its block partial sums and wall temperature strips live in the file-scope
// array below (1 MiB, allocated by the CUDA runtime when the module loads on
// a device and held by every device that loads the library until the process
// exits).  Host code must not pass the array's name to a kernel -- in host
// code it is only a stand-in for the symbol -- so every call looks up the
// device address of the array in the current device's context with
// cudaGetSymbolAddress.  The address is not cached: after cudaDeviceReset, or
// under another context on the same device, the module is loaded again at
// another address.

static __device__ __align__(256) double g_diag_scratch[1 << 17];

namespace lbk {
namespace {

constexpr size_t kScratchDoubles = (size_t)1 << 17;
constexpr int kScratchMaxBlocks = 2048;

cudaError_t scratch_address(double **out)
{
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_diag_scratch);
    if (e != cudaSuccess) return e;
    *out = (double *)p;
    return cudaSuccess;
}

}  // namespace
}  // namespace lbk

extern "C" lb_status lb_diagnostics_static(const lb_grid_desc *desc, const lb_params *p, const void *dev_state,
                                           int64_t step, void *cuda_stream, lb_diag *out)
{
    using namespace lbk;
    if (!desc || !p || !dev_state || !out) {
        set_global_error("lb_diagnostics_static: NULL argument");
        return LB_ERR_ARG;
    }
    HostParams h;
    std::memset(&h, 0, sizeof(h));
    char why[200];
    if (host_from_desc(desc, &h, why, sizeof(why)) != LB_OK || host_set_params(p, &h, why, sizeof(why)) != LB_OK) {
        char msg[256];
        snprintf(msg, sizeof(msg), "lb_diagnostics_static: %s", why);
        set_global_error(msg);
        return LB_ERR_ARG;
    }
    if (((uintptr_t)dev_state & 255) != 0) {
        set_global_error("lb_diagnostics_static: dev_state must be 256-byte aligned");
        return LB_ERR_ARG;
    }
    // The size is limited by blocks of 120 columns and 32 rows, taller ones
    // where these were more than kScratchMaxBlocks.  The grid is lb_diagnostics's
    // where its partial sums fit beside the strips, else one with no more blocks
    // than counted here.
    const long long bx = (h.nr + 119) / 120, by = (h.nz + 31) / 32;
    const long long cap = std::max(1LL, std::min(by, kScratchMaxBlocks / bx)), seg = (h.nz + cap - 1) / cap;
    const long long most = bx * ((h.nz + seg - 1) / seg);
    const size_t need = 16 + (size_t)most * NSUM + 4 * ((size_t)h.nr + (size_t)h.nz);
    auto doubles = [&](const DiagGrid &g) { return 16 + (size_t)g.gx * g.gy * NSUM + 4 * ((size_t)h.nr + (size_t)h.nz); };
    DiagGrid g = diag_grid(h, MAX_DIAG_BLOCKS);
    if (doubles(g) > kScratchDoubles) g = diag_grid(h, (int)most);
    const long long nb = (long long)g.gx * g.gy;
    if (most > kScratchMaxBlocks || need > kScratchDoubles) {
        char msg[200];
        snprintf(msg, sizeof(msg),
                 "lb_diagnostics_static: a %d x %d lattice needs %zu scratch doubles, the static array holds %zu "
                 "(nr + nz must stay below about 26600)",
                 h.nr, h.nz, need, kScratchDoubles);
        set_global_error(msg);
        return LB_ERR_ARG;
    }
    double *scratch = nullptr;
    cudaError_t e = scratch_address(&scratch);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (e == cudaSuccess) e = cudaMemsetAsync(scratch, 0, doubles(g) * sizeof(double), st);
    if (e == cudaSuccess) {
        double *partial = scratch + 16, *strips = partial + (size_t)nb * NSUM;
        switch (h.storage) {
            case ST_FP64: e = diag_t<double, double>(h, g, dev_state, partial, strips, scratch, st); break;
            case ST_FP32: e = diag_t<float, float>(h, g, dev_state, partial, strips, scratch, st); break;
            case ST_BF16: e = diag_t<__nv_bfloat16, float>(h, g, dev_state, partial, strips, scratch, st); break;
            default: e = diag_t<__half, float>(h, g, dev_state, partial, strips, scratch, st); break;
        }
    }
    double res[NSUM];
    if (e == cudaSuccess) e = cudaMemcpyAsync(res, scratch, sizeof(res), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        char msg[200];
        snprintf(msg, sizeof(msg), "lb_diagnostics_static: %s", cudaGetErrorString(e));
        set_global_error(msg);
        return LB_ERR_CUDA;
    }
    diag_from_sums(h, res, 0, step, out);
    return LB_OK;
}
