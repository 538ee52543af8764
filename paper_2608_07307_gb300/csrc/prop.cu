// prop.cu -- orbit propagation with the ray-traced SRP force in every stage
// (Sec. 3, Eqs. 1-3: y = (x, v), y' = (v, a_g + a_SRP), integrated with an
// explicit embedded Runge-Kutta 7(8) pair that evaluates the SRP acceleration
// several times per step).
//
// One step is a fixed sequence of kernels, captured once in a CUDA graph and
// relaunched: for each stage, k_prop_stage forms the stage state and the Sun
// direction in the body frame, the SRP evaluation pipeline runs for every
// trajectory, k_prop_accel forms the stage derivative; k_prop_control then
// accepts or rejects the step and picks the next step size.  All state lives
// on the device; the host only relaunches the graph and polls a done counter.
// Every kernel of a step runs a warp per trajectory on a copy of its state in
// shared memory.  An FP64 instruction holds this GPU's FP64 pipe for 64 cycles a
// warp whatever the number of active lanes (a dependent chain and four independent
// ones measured the same; a square root or a division takes 10 of them, atan2 45,
// pow 92), so what these kernels cost is the number of FP64 instructions their warp
// issues: components, norms and divisions are spread over the lanes, and one
// instruction serves all of them.  Each value is formed by the expression a single
// lane would use.  At the first stage of a step, lanes compute the Sun positions of
// all stages (their times are fixed with the step size).  Without ray tracing between
// the stages (a SPAD table or SRP off) the whole step is one kernel, k_prop_step,
// built from the same parts.
//
// Integrators: Fehlberg's 7(8) pair (13 stages, NASA TR R-287, 1968),
// propagating the 7th-order solution, error norm
// max_i |e_i| / (atol_i + rtol max(|y_i|, |y_new_i|)), next h = h clamp(0.9
// err^(-1/8), 0.2, 5); or classical RK4 with a fixed step.  Forces: central
// point mass, optional Earth J2 (z = pole) and the Sun as a third body from the
// low-precision solar coordinates of Montenbruck & Gill (Satellite Orbits,
// Sec. 3.3.2), SRP zero inside a cylindrical Earth shadow; attitude: the LVLH
// frame (z to nadir, y along minus the orbit normal) turned by a constant
// quaternion, or a fixed inertial quaternion.
#include <math.h>

#include "srp_internal.cuh"

namespace srp {

namespace {

constexpr double kMuEarth = 3.986004418e14;
constexpr double kREarth = 6378137.0;
constexpr double kJ2 = 1.08262668e-3;
constexpr double kMuSun = 1.32712440018e20;
constexpr double kAU = 1.495978707e11;
constexpr double kPi = 3.14159265358979323846;

// Fehlberg 7(8): nodes, stage weights (lower triangle), 7th / 8th order weights.
__constant__ double cC[13] = {0.0,       2.0 / 27.0, 1.0 / 9.0, 1.0 / 6.0, 5.0 / 12.0, 0.5, 5.0 / 6.0,
                              1.0 / 6.0, 2.0 / 3.0,  1.0 / 3.0, 1.0,       0.0,        1.0};
__constant__ double cA[13][12] = {
    {0},
    {2.0 / 27.0},
    {1.0 / 36.0, 1.0 / 12.0},
    {1.0 / 24.0, 0.0, 1.0 / 8.0},
    {5.0 / 12.0, 0.0, -25.0 / 16.0, 25.0 / 16.0},
    {1.0 / 20.0, 0.0, 0.0, 1.0 / 4.0, 1.0 / 5.0},
    {-25.0 / 108.0, 0.0, 0.0, 125.0 / 108.0, -65.0 / 27.0, 125.0 / 54.0},
    {31.0 / 300.0, 0.0, 0.0, 0.0, 61.0 / 225.0, -2.0 / 9.0, 13.0 / 900.0},
    {2.0, 0.0, 0.0, -53.0 / 6.0, 704.0 / 45.0, -107.0 / 9.0, 67.0 / 90.0, 3.0},
    {-91.0 / 108.0, 0.0, 0.0, 23.0 / 108.0, -976.0 / 135.0, 311.0 / 54.0, -19.0 / 60.0, 17.0 / 6.0, -1.0 / 12.0},
    {2383.0 / 4100.0, 0.0, 0.0, -341.0 / 164.0, 4496.0 / 1025.0, -301.0 / 82.0, 2133.0 / 4100.0, 45.0 / 82.0,
     45.0 / 164.0, 18.0 / 41.0},
    {3.0 / 205.0, 0.0, 0.0, 0.0, 0.0, -6.0 / 41.0, -3.0 / 205.0, -3.0 / 41.0, 3.0 / 41.0, 6.0 / 41.0, 0.0},
    {-1777.0 / 4100.0, 0.0, 0.0, -341.0 / 164.0, 4496.0 / 1025.0, -289.0 / 82.0, 2193.0 / 4100.0, 51.0 / 82.0,
     33.0 / 164.0, 12.0 / 41.0, 0.0, 1.0},
};
__constant__ double cB7[13] = {41.0 / 840.0, 0.0, 0.0, 0.0, 0.0, 34.0 / 105.0, 9.0 / 35.0, 9.0 / 35.0, 9.0 / 280.0,
                               9.0 / 280.0, 41.0 / 840.0, 0.0, 0.0};
__constant__ double cB8[13] = {0.0, 0.0, 0.0, 0.0, 0.0, 34.0 / 105.0, 9.0 / 35.0, 9.0 / 35.0, 9.0 / 280.0,
                               9.0 / 280.0, 0.0, 41.0 / 840.0, 41.0 / 840.0};
// classical RK4
__constant__ double cC4[4] = {0.0, 0.5, 0.5, 1.0};
__constant__ double cB4[4] = {1.0 / 6.0, 1.0 / 3.0, 1.0 / 3.0, 1.0 / 6.0};

__device__ void sun_pos(double mjd_tt, double *r)
{
    const double deg = kPi / 180.0;
    double T = (mjd_tt - 51544.5) / 36525.0;
    double M = fmod(357.5256 + 35999.049 * T, 360.0) * deg;
    // two FP64 sincos calls (slow on this GPU's FP64 pipe); the double angle by identity
    double sM, cM;
    sincos(M, &sM, &cM);
    const double s2M = 2.0 * sM * cM, c2M = (cM - sM) * (cM + sM);
    double lam = 282.94 * deg + M + (6892.0 * sM + 72.0 * s2M) * (deg / 3600.0);
    double rr = 149.619e9 - 2.499e9 * cM - 0.021e9 * c2M;
    const double ce = 0.9174820620768958, se = 0.3977771559141214;  // cos, sin of the obliquity 23.43929111 deg
    double sl, cl;
    sincos(lam, &sl, &cl);
    r[0] = rr * cl;
    r[1] = rr * sl * ce;
    r[2] = rr * sl * se;
}

// cfg (null: P's values for every trajectory): [n][8] central, attitude, q[4], mass, unused
__global__ void k_prop_init(PropState *S, int n, const double *y0, const double *t01, PropDev P, const double *cfg,
                            int *n_done)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    PropState &X = S[i];
    const double h0 = P.h0;
    if (cfg) {
        const double *c = cfg + 8 * (size_t)i;
        X.central = (int)c[0];
        X.attitude = (int)c[1];
        for (int k = 0; k < 4; k++) X.q[k] = c[2 + k];
        X.mass = c[6];
    } else {
        X.central = P.central;
        X.attitude = P.attitude;
        for (int k = 0; k < 4; k++) X.q[k] = P.q[k];
        X.mass = P.mass;
    }
    X.imass = 1.0 / X.mass;
    quat_matrix(X.q, X.Qm);
    for (int k = 0; k < 6; k++) X.y[k] = y0[6 * i + k];
    X.t = t01[2 * i];
    X.t1 = t01[2 * i + 1];
    X.h = h0;
    X.hs = h0;
    X.done = X.t1 <= X.t ? 1 : 0;
    X.status = 0;
    X.steps = X.rejects = X.evals = 0;
    X.nlog = 0;
    X.shadow = 0;
    for (int j = 0; j < 13; j++)
        for (int k = 0; k < 6; k++) X.k[j][k] = 0.0;
    if (X.done) atomicAdd(n_done, 1);
}

// Warps (trajectories) of a block: one to each of an SM's four FP64 pipes.
constexpr int kPropWarps = 4;

// A trajectory's warp: its state, and the operands that lanes hand to each other.
struct PropWarp {
    PropState X;
    double y[6], h[3], sv[3], rs[3];  // stage state, r x v, Sun from spacecraft, Sun (stage_body)
    double q[11];                     // the stage's quotients
    double zb[3], yb[3], xb[3], e[3]; // LVLH axes, Sun direction from the central body
    double sun[3], dist;              // body-frame Sun direction and distance (AU; negative: no SRP)
};

// The state's words in and out of shared memory: independent loads, one latency.
__device__ __forceinline__ void load_state(PropWarp &W, const PropState &G, int lane)
{
    static_assert(sizeof(PropState) % 8 == 0, "copied by 8-byte words");
    const double *src = reinterpret_cast<const double *>(&G);
    double *dst = reinterpret_cast<double *>(&W.X);
#pragma unroll
    for (int k = 0; k < (int)(sizeof(PropState) / 8); k += 32)
        if (k + lane < (int)(sizeof(PropState) / 8)) dst[k + lane] = src[k + lane];
    __syncwarp();
}
__device__ __forceinline__ void store_state(const PropWarp &W, PropState &G, int lane)
{
    __syncwarp();
    const double *src = reinterpret_cast<const double *>(&W.X);
    double *dst = reinterpret_cast<double *>(&G);
#pragma unroll
    for (int k = 0; k < (int)(sizeof(PropState) / 8); k += 32)
        if (k + lane < (int)(sizeof(PropState) / 8)) dst[k + lane] = src[k + lane];
}

__device__ __forceinline__ double shfl(double x, int lane) { return __shfl_sync(0xffffffffu, x, lane); }

// Stage state, gravity, attitude, Sun direction (body frame) and distance for
// the SRP call (negative to skip it: a finished or shadowed trajectory).  At the
// first stage of a step, once the step size is fixed, every stage time is known:
// lanes compute the Sun positions of all stages at once.
__device__ __forceinline__ void stage_body(PropWarp &W, int i, const PropDev &P, int stage, int lane)
{
    PropState &X = W.X;
    const int rk4 = P.method == 1;
    if (stage == 0) {
        if (lane == 0 && !X.done) {
            double h = X.h;
            if (P.n_replay > 0) {
                h = X.steps < P.n_replay ? P.h_replay[(size_t)i * P.n_replay + X.steps] : 0.0;
            } else if (X.t + h >= X.t1) {
                h = X.t1 - X.t;  // land exactly on t1
            }
            X.hs = h;
        }
        __syncwarp();
        if (lane < (rk4 ? 4 : 13) && X.central == 0) {
            const double ts = X.t + (rk4 ? cC4[lane] : cC[lane]) * X.hs;
            double rs[3];
            sun_pos(P.epoch_mjd_tt + ts / 86400.0, rs);
            for (int k = 0; k < 3; k++) X.rs_st[lane][k] = rs[k];
        }
        __syncwarp();
    }
    const int c3 = lane % 3;
    // lanes 0-5: the components of the stage state; lane 6: the stage time
    {
        double acc = 0.0, base = X.t;
        if (lane < 6) base = X.y[lane];
        if (lane == 6) acc = rk4 ? cC4[stage] : cC[stage];
        const int k = lane < 6 ? lane : 0;
        if (rk4) {
            if (stage > 0) {
                const double x = 0.5 * X.k[stage - 1][k] * (stage == 3 ? 2.0 : 1.0);
                if (lane < 6) acc = x;
            }
        } else {
            double s = 0.0;
            for (int j = 0; j < stage; j++) s += cA[stage][j] * X.k[j][k];
            if (lane < 6) acc = s;
        }
        const double x = base + X.hs * acc;
        if (lane < 6) W.y[lane] = X.ys[lane] = x;
        if (lane == 6) X.ts = x;
        if (lane < 3) W.rs[lane] = X.central == 0 ? X.rs_st[stage][lane] : 0.0;
    }
    __syncwarp();
    // lanes 0-2: r x v; the others: the Sun from the spacecraft (a product with one is exact)
    {
        const int k1 = c3 == 2 ? 0 : c3 + 1, k2 = c3 == 0 ? 2 : c3 - 1;
        const bool hv = lane < 3;
        const double p = hv ? W.y[k1] : W.rs[c3], q = hv ? W.y[3 + k2] : 1.0;
        const double r = hv ? W.y[k2] : W.y[c3], s = hv ? W.y[3 + k1] : 1.0;
        const double x = p * q - r * s;
        if (lane < 3) W.h[lane] = x;
        else if (lane < 6) W.sv[c3] = x;
    }
    __syncwarp();
    // norms: lane 0 |r|, 1 |r x v|, 2 Sun distance, 3 |Sun|
    double n2, n;
    {
        const int g = lane & 3;
        const double *v = g == 0 ? W.y : g == 1 ? W.h : g == 2 ? W.sv : W.rs;
        n2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        n = sqrt(n2);
    }
    const double r2 = shfl(n2, 0), r = shfl(n, 0), hn = shfl(n, 1), sd = shfl(n, 2), sn = shfl(n, 3);
    // every quotient of the stage in one division
    {
        const double m = lane == 9 ? sn : lane == 8 ? sd : r2;           // cubes: r2 r, |d|^3, |s|^3
        const double m2 = m * (lane == 9 ? sn : lane == 8 ? sd : r);
        const double m3 = m2 * (lane == 9 ? sn : sd);
        double num = 1.0, den = 1.0;
        const bool lvlh = X.attitude != 1, earth = X.central == 0;
        if (lane < 3) { num = W.sv[lane]; den = sd; }
        else if (lane == 3) { num = -1.0; den = lvlh ? r : 1.0; }
        else if (lane == 4) { num = -1.0; den = lvlh ? hn : 1.0; }
        else if (lane == 5) den = earth ? sn : 1.0;
        else if (lane == 6) den = m2;
        else if (lane == 7) den = r2;
        else if (lane == 8 || lane == 9) den = earth ? m3 : 1.0;
        else if (lane == 10) { num = sd; den = kAU; }
        const double x = num / den;
        if (lane < 11) W.q[lane] = x;
    }
    __syncwarp();
    // z_b = nadir, y_b = -orbit normal, e = Sun direction from the central body
    {
        const int g = lane / 3;
        const double x = (g == 0 ? W.y[c3] : g == 1 ? W.h[c3] : W.rs[c3]) * W.q[g == 0 ? 3 : g == 1 ? 4 : 5];
        if (lane < 9) (g == 0 ? W.zb : g == 1 ? W.yb : W.e)[c3] = x;
    }
    __syncwarp();
    // x_b = y_b x z_b, in lanes 0-2
    {
        const int k1 = c3 == 2 ? 0 : c3 + 1, k2 = c3 == 0 ? 2 : c3 - 1;
        const double x = W.yb[k1] * W.zb[k2] - W.yb[k2] * W.zb[k1];
        if (lane < 3) W.xb[lane] = x;
    }
    __syncwarp();
    // body -> inertial rotation, an element a lane: the quaternion's (inertial attitude) or
    // the LVLH frame (columns x_b, y_b, z_b) turned by it
    {
        const int l = lane < 9 ? lane : 0, a = l / 3, b = l % 3;
        const double x = W.xb[a] * X.Qm[b] + W.yb[a] * X.Qm[3 + b] + W.zb[a] * X.Qm[6 + b];
        if (lane < 9) X.R[lane] = X.attitude == 1 ? X.Qm[lane] : x;
    }
    // cylindrical Earth shadow
    int shadow = 0;
    if (X.central == 0) {
        const double pr = W.y[0] * W.e[0] + W.y[1] * W.e[1] + W.y[2] * W.e[2];
        const double q = W.y[c3] - pr * W.e[c3];
        const double q0 = shfl(q, 0), q1 = shfl(q, 1), q2 = shfl(q, 2);
        if (pr < 0.0 && q0 * q0 + q1 * q1 + q2 * q2 < kREarth * kREarth) shadow = 1;
    }
    // gravity, a component a lane: central body, Earth J2, the Sun as a third body
    {
        const double mu = X.central == 1 ? kMuSun : kMuEarth;
        const double ir3 = W.q[6], yk = W.y[c3];
        double a = -mu * yk * ir3;
        if (X.central == 0 && P.j2) {
            const double ir2 = W.q[7];
            const double z2 = W.y[2] * W.y[2] * ir2;
            const double f = -1.5 * kJ2 * kMuEarth * kREarth * kREarth * (ir3 * ir2);
            a += f * yk * ((c3 == 2 ? 3.0 : 1.0) - 5.0 * z2);
        }
        if (X.central == 0 && P.sun3) a += kMuSun * (W.sv[c3] * W.q[8] - W.rs[c3] * W.q[9]);
        if (lane < 3) X.grav[lane] = a;
    }
    __syncwarp();
    const double dir = X.R[c3] * W.q[0] + X.R[3 + c3] * W.q[1] + X.R[6 + c3] * W.q[2];
    if (lane < 3) {
        X.rsun[lane] = W.rs[lane];
        W.sun[lane] = dir;
    }
    if (lane == 0) {
        X.shadow = shadow;
        W.dist = (X.done || shadow || !P.srp) ? -1.0 : W.q[10];
    }
    __syncwarp();
}

// The stage's Sun direction and distance where the SRP call reads them.
__device__ __forceinline__ void store_sun(const PropWarp &W, int i, int lane, double *sun_dir, double *sun_dist)
{
    if (lane < 3) sun_dir[3 * i + lane] = W.sun[lane];
    if (lane == 3) sun_dist[i] = W.dist;
}

// What the acceleration of a stage reads of the SRP call: the traced force, or
// the Sun direction and distance a SPAD table is read at.
__device__ __forceinline__ void load_srp(PropWarp &W, int i, const PropDev &P, int lane, const double *force,
                                         const double *sun_dir, const double *sun_dist)
{
    if (!P.srp) return;
    if (P.spad.table) {
        if (lane < 3) W.sun[lane] = sun_dir[3 * i + lane];
        if (lane == 3) W.dist = sun_dist[i];
    } else if (lane < 3) {
        W.h[lane] = force[3 * i + lane];
    }
    __syncwarp();
}

__global__ void __launch_bounds__(32 * kPropWarps) k_prop_stage(PropState *S, int n, PropDev P, int stage,
                                                                double *sun_dir, double *sun_dist)
{
    pdl_enter();
    __shared__ PropWarp sh[kPropWarps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kPropWarps + w;
    if (i >= n) return;  // whole warps
    PropWarp &W = sh[w];
    load_state(W, S[i], lane);
    stage_body(W, i, P, stage, lane);
    store_sun(W, i, lane, sun_dir, sun_dist);
    store_state(W, S[i], lane);
}

// spad_lookup's force by a warp, component `lane` in lanes 0-2: both angles in one
// atan2, the quotients in one division.
__device__ __forceinline__ double spad_force_warp(const SpadDev &g, const double *s, double dist, int lane)
{
    if (dist < 0.0) return 0.0;
    const bool elev = lane == 1;
    const double hyp = hypot(s[0], s[1]);
    const double a = atan2(elev ? s[2] : s[1], elev ? hyp : s[0]) - (elev ? g.el0 : g.az0);
    const double u = a * (g.n_az * 0.15915494309189535);  // cells of 2 pi / n_az
    const double q = (lane == 2 ? 1.0 : elev ? a : u) / (lane == 2 ? dist * dist : elev ? g.d_el : (double)g.n_az);
    const SpadCell c = spad_cell(g, shfl(u, 0), shfl(q, 0), shfl(q, 1));
    return spad_value(c, lane % 3, shfl(q, 2));
}

// Stage derivative: gravity plus the SRP force (traced, in W.h, or the SPAD
// interpolant, Sec. 4.2, at this stage's body-frame Sun direction).
__device__ __forceinline__ void accel_body(PropWarp &W, const PropDev &P, int stage, int lane)
{
    PropState &X = W.X;
    const int c3 = lane % 3;
    double a = X.grav[c3];
    if (P.srp && !X.shadow) {
        if (P.spad.table) {
            const double f = spad_force_warp(P.spad, W.sun, W.dist, lane);
            if (lane < 3) W.h[lane] = f;
            __syncwarp();
        }
        a += (X.R[3 * c3] * W.h[0] + X.R[3 * c3 + 1] * W.h[1] + X.R[3 * c3 + 2] * W.h[2]) * X.imass;
    }
    if (lane < 3) X.k[stage][lane] = X.ys[3 + lane];
    else if (lane < 6) X.k[stage][lane] = a;
    if (lane == 0 && !X.done) X.evals++;
    __syncwarp();
}

__global__ void __launch_bounds__(32 * kPropWarps) k_prop_accel(PropState *S, int n, PropDev P, int stage,
                                                                const double *force, const double *sun_dir,
                                                                const double *sun_dist)
{
    pdl_enter();
    __shared__ PropWarp sh[kPropWarps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kPropWarps + w;
    if (i >= n) return;  // whole warps
    PropWarp &W = sh[w];
    load_srp(W, i, P, lane, force, sun_dir, sun_dist);
    load_state(W, S[i], lane);
    accel_body(W, P, stage, lane);
    store_state(W, S[i], lane);
}

// Step control: accept or reject, next step size, completion.  Lanes 0-5 hold a
// component of the state each; lane 0 decides.
__device__ __forceinline__ void control_body(PropWarp &W, int i, const PropDev &P, int lane, int *n_done, double *h_log,
                                             int64_t h_cap)
{
    PropState &X = W.X;
    if (X.done) return;  // uniform
    const double h = X.hs;
    const int k = lane < 6 ? lane : 0;
    if (P.n_replay > 0) {
        // replay: take the given step, 7th-order solution, no error control
        double s7 = 0.0;
        for (int j = 0; j < 13; j++) s7 += cB7[j] * X.k[j][k];
        const double yn = X.y[k] + h * s7;
        __syncwarp();
        if (lane < 6) X.y[k] = yn;
        if (lane == 0) {
            X.t += h;
            if (h_log && X.nlog < h_cap) h_log[(size_t)i * h_cap + X.nlog] = h;
            X.nlog++;
            X.steps++;
            if (X.steps >= P.n_replay) { X.done = 1; atomicAdd(n_done, 1); }
        }
        __syncwarp();
        return;
    }
    const bool last = X.t + X.h >= X.t1;
    bool accept = true;
    double yn;
    double fac = 1.0;
    if (P.method == 1) {
        double acc = 0.0;
        for (int j = 0; j < 4; j++) acc += cB4[j] * X.k[j][k];
        yn = X.y[k] + h * acc;
    } else {
        double s7 = 0.0, s8 = 0.0;
        for (int j = 0; j < 13; j++) { s7 += cB7[j] * X.k[j][k]; s8 += cB8[j] * X.k[j][k]; }
        yn = X.y[k] + h * s7;
        const double sc = (k < 3 ? P.atol_pos : P.atol_vel) + P.rtol * fmax(fabs(X.y[k]), fabs(yn));
        const double ek = fabs(h * (s7 - s8)) / sc;
        double e = 0.0;
        for (int j = 0; j < 6; j++) e = fmax(e, shfl(ek, j));
        fac = e == 0.0 ? 5.0 : fmin(5.0, fmax(0.2, 0.9 * pow(e, -1.0 / 8.0)));
        accept = e <= 1.0;
    }
    __syncwarp();
    if (accept && lane < 6) X.y[k] = yn;
    if (lane == 0) {
        if (accept) {
            // fixed steps snap onto t1 when they land within 1e-9 of a step of it
            X.t = (last || (P.method == 1 && X.t1 - (X.t + h) < 1e-9 * P.h0)) ? X.t1 : X.t + h;
            if (h_log && X.nlog < h_cap) h_log[(size_t)i * h_cap + X.nlog] = h;
            X.nlog++;
            X.steps++;
        } else {
            X.rejects++;
        }
        if (P.method == 0) {
            double hn = X.hs * fac;
            if (P.h_max > 0.0) hn = fmin(hn, P.h_max);
            if (X.t < X.t1 && hn < P.h_min) { X.status = SRP_ERR_STEP; X.done = 1; }
            X.h = hn;
        }
        if (X.t >= X.t1) X.done = 1;
        if (X.steps + X.rejects > P.max_steps && !X.done) { X.status = SRP_ERR_STEP; X.done = 1; }
        if (X.done) atomicAdd(n_done, 1);
    }
    __syncwarp();
}

__global__ void __launch_bounds__(32 * kPropWarps) k_prop_control(PropState *S, int n, PropDev P, int *n_done,
                                                                  double *h_log, int64_t h_cap)
{
    pdl_enter();
    __shared__ PropWarp sh[kPropWarps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kPropWarps + w;
    if (i >= n) return;  // whole warps
    PropWarp &W = sh[w];
    load_state(W, S[i], lane);
    control_body(W, i, P, lane, n_done, h_log, h_cap);
    store_state(W, S[i], lane);
}

// The stage derivative of `stage` and, in the same launch, the state of the
// next stage; after the last stage, step control and the first stage of the
// next step (which the captured step then starts from).
__global__ void __launch_bounds__(32 * kPropWarps) k_prop_next(PropState *S, int n, PropDev P, int stage,
                                                               const double *force, double *sun_dir, double *sun_dist,
                                                               int *n_done, double *h_log, int64_t h_cap)
{
    pdl_enter();
    __shared__ PropWarp sh[kPropWarps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kPropWarps + w;
    if (i >= n) return;  // whole warps
    PropWarp &W = sh[w];
    const int nst = P.method == 1 ? 4 : 13;
    load_srp(W, i, P, lane, force, sun_dir, sun_dist);
    load_state(W, S[i], lane);
    accel_body(W, P, stage, lane);
    const bool end = stage + 1 >= nst;
    if (end) control_body(W, i, P, lane, n_done, h_log, h_cap);
    stage_body(W, i, P, end ? 0 : stage + 1, lane);
    store_sun(W, i, lane, sun_dir, sun_dist);
    store_state(W, S[i], lane);
}

// A whole step in one launch when no ray-traced evaluation sits between the
// stages (SPAD table or SRP off): the stage, acceleration and control parts of
// the kernels above, in their order.
__global__ void __launch_bounds__(32 * kPropWarps) k_prop_step(PropState *S, int n, PropDev P, double *sun_dir,
                                                               double *sun_dist, int *n_done, double *h_log,
                                                               int64_t h_cap)
{
    pdl_enter();
    __shared__ PropWarp sh[kPropWarps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kPropWarps + w;
    if (i >= n) return;  // whole warps
    PropWarp &W = sh[w];
    load_state(W, S[i], lane);
    const int nst = P.method == 1 ? 4 : 13;
    for (int stage = 0; stage < nst; stage++) {
        stage_body(W, i, P, stage, lane);
        accel_body(W, P, stage, lane);
    }
    store_sun(W, i, lane, sun_dir, sun_dist);
    control_body(W, i, P, lane, n_done, h_log, h_cap);
    store_state(W, S[i], lane);
}


// ------------------------------------------------------------------ adjoint
// Discrete adjoint of the RK4 step y' = y + h sum_i b_i k_i, k_i = f(t_i, y_i),
// y_i = y + h a_{i,i-1} k_{i-1}: with lam the cotangent of y',
//   kbar_i = h b_i lam + h a_{i+1,i} ybar_{i+1},   ybar_i = (df/dy_i)^T kbar_i,
//   lam_before = lam + sum_i ybar_i,
// and the SRP part of df/dy_i, d f / d(parameters) through the frozen-hit
// adjoint of the evaluation (adjoint.cu).  Stages run 3, 2, 1, 0.

__device__ inline void save_ckpt(const PropState &X, double *b)
{
    b[0] = X.t;
    for (int k = 0; k < 6; k++) b[1 + k] = X.y[k];
}

__global__ void k_prop_ckpt(PropState *S, int n, double *buf, int save, double h0)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    PropState &X = S[i];
    double *b = buf + 7 * (size_t)i;
    if (save) {
        save_ckpt(X, b);
        return;
    }
    X.t = b[0];
    for (int k = 0; k < 6; k++) X.y[k] = b[1 + k];
    X.h = X.hs = h0;  // a fixed-step arc always proposes h0
    X.done = X.t >= X.t1 ? 1 : 0;
    X.status = 0;
}

__global__ void k_prop_record(const PropState *S, int n, const double *sun, const double *dist, const double *force,
                              StageRec *rec, double *rec_sun, double *rec_dist)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const PropState &X = S[i];
    StageRec &r = rec[i];
    for (int k = 0; k < 6; k++) r.ys[k] = X.ys[k];
    r.ts = X.ts;
    r.hs = X.hs;
    for (int k = 0; k < 9; k++) r.R[k] = X.R[k];
    for (int k = 0; k < 3; k++) r.rsun[k] = X.rsun[k];
    r.lit = dist[i] >= 0.0 ? 1 : 0;
    for (int k = 0; k < 3; k++) {
        r.F[k] = r.lit ? force[3 * i + k] : 0.0;
        rec_sun[3 * i + k] = sun[3 * i + k];
    }
    rec_dist[i] = dist[i];
}

// kbar of this stage, and the cotangent of the body-frame SRP force; a warp per
// trajectory, a component a lane
__global__ void __launch_bounds__(32) k_adj_prop_in(int n, PropDev P, int stage, const StageRec *rec, PropAdj *A,
                                                    double *g_force)
{
    pdl_enter();
    const int i = blockIdx.x, lane = threadIdx.x;
    const StageRec &r = rec[i];
    PropAdj &X = A[i];
    const double h = r.hs;
    const double anext = stage == 2 ? 1.0 : 0.5;  // a_{stage+1, stage}
    const int k = lane < 6 ? lane : 0, c3 = lane % 3;
    const double R0 = r.R[c3], R1 = r.R[3 + c3], R2 = r.R[6 + c3];
    const double kb = h * cB4[stage] * X.lam[k] + (stage < 3 ? h * anext * X.ybar[stage + 1][k] : 0.0);
    if (lane < 6) X.kbar[k] = kb;
    const double a0 = shfl(kb, 3), a1 = shfl(kb, 4), a2 = shfl(kb, 5);
    if (lane < 3) g_force[3 * i + lane] = r.lit ? (R0 * a0 + R1 * a1 + R2 * a2) / P.mass : 0.0;
}

// (df/dy)^T kbar at this stage: gravity, SRP through the Sun direction, distance
// and attitude; attitude quaternion cotangent.  Four warps a trajectory on the SM's
// four FP64 pipes (64 cycles an instruction and warp): central body and J2, the Sun's
// force and direction, the quaternion, the LVLH frame and the third body; components,
// matrix elements and quotients a lane each.  (One thread: 649 instructions in a row, 26 us.)
__global__ void __launch_bounds__(128) k_adj_prop_out(int n, PropDev P, int stage, const StageRec *rec, PropAdj *A,
                                                      const double *g_sun, const double *g_dist)
{
    pdl_enter();
    const int i = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31, c3 = lane % 3;
    const int k1 = c3 == 2 ? 0 : c3 + 1, k2 = c3 == 0 ? 2 : c3 - 1;
    const int l9 = lane < 9 ? lane : 0, a = l9 / 3, b = l9 % 3;
    const StageRec &r = rec[i];
    PropAdj &X = A[i];
    __shared__ double s_y[6], s_ab[3], s_rs[3], s_gs[3];
    __shared__ double s_grav[3], s_third[3], s_wb[3], s_Rb[9], s_Q[9], s_Qb[9], s_L[9], s_Lb[9], s_in[2], s_rv[6];
    if (threadIdx.x < 6) s_y[threadIdx.x] = r.ys[threadIdx.x];
    if (w == 1 && lane < 3) {
        s_ab[lane] = X.kbar[3 + lane];
        s_rs[lane] = r.rsun[lane];
        s_gs[lane] = r.lit ? g_sun[3 * i + lane] : 0.0;
    }
    const bool lit = r.lit, lvlh = P.attitude != 1;  // uniform over the block
    __syncthreads();
    const double *y = s_y, *ab = s_ab;
    double qn = 1.0, qk = 0.0;  // warp 2: the quaternion's norm, its normalised components in lanes 0-3
    if (w == 0) {
        // central body: J = -mu (I / r^3 - 3 r r^T / r^5), symmetric
        const double r2 = y[0] * y[0] + y[1] * y[1] + y[2] * y[2], rn = sqrt(r2);
        const double mu = P.central == 1 ? kMuSun : kMuEarth;
        const double ra = y[0] * ab[0] + y[1] * ab[1] + y[2] * ab[2];
        const double kJ = -1.5 * kJ2 * kMuEarth * kREarth * kREarth;
        const double q = (lane == 2 ? kJ : 1.0) / (lane == 2 ? r2 * r2 * rn : lane == 1 ? r2 : r2 * rn);
        const double ir3 = shfl(q, 0), ir2 = shfl(q, 1), f = shfl(q, 2);
        const double ir5 = ir3 / r2;
        double x = -mu * (ab[c3] * ir3 - 3.0 * y[c3] * ra * ir5);
        if (P.central == 0 && P.j2) {
            const double z2 = y[2] * y[2] * ir2;
            const double m = (c3 == 2 ? 3.0 : 1.0) - 5.0 * z2;
            const double g = y[c3] * m;
            const double fb = ab[0] * shfl(g, 0) + ab[1] * shfl(g, 1) + ab[2] * shfl(g, 2);
            const double z2b = -5.0 * f * ra;
            const double r2b = -z2b * y[2] * y[2] * (ir2 * ir2) + fb * (-2.5) * f * ir2;
            x += f * ab[c3] * m;
            x += c3 == 2 ? z2b * 2.0 * y[2] * ir2 : 0.0;
            x += 2.0 * r2b * y[c3];
        }
        if (lane < 3) s_grav[lane] = x;
    } else if (w == 1 && lit) {
        // a_SRP = R F / m, s_body = R^T s_hat, s_hat = w / |w|, w = r_sun - r, dist = |w| / AU
        const double wv = s_rs[c3] - y[c3];
        const double w0 = shfl(wv, 0), w1 = shfl(wv, 1), w2 = shfl(wv, 2);
        const double wn = sqrt(w0 * w0 + w1 * w1 + w2 * w2);
        const double q = 1.0 / (lane == 1 ? P.mass : wn);
        const double iwn = shfl(q, 0), im = shfl(q, 1);
        const double sc = wv * iwn;
        const double sh0 = shfl(sc, 0), sh1 = shfl(sc, 1), sh2 = shfl(sc, 2);
        const double *R = r.R;
        const double shb = R[3 * c3] * s_gs[0] + R[3 * c3 + 1] * s_gs[1] + R[3 * c3 + 2] * s_gs[2];
        const double sd = shfl(shb, 0) * sh0 + shfl(shb, 1) * sh1 + shfl(shb, 2) * sh2;
        const double wb = (shb - sd * sc) * iwn + g_dist[i] * sc * (1.0 / kAU);
        if (lane < 3) s_wb[lane] = wb;
        const double Rb = ab[a] * r.F[b] * im + (a == 0 ? sh0 : a == 1 ? sh1 : sh2) * s_gs[b];
        if (lane < 9) s_Rb[lane] = Rb;
    } else if (w == 2 && lit) {
        // the normalised quaternion and its rotation
        qn = sqrt(P.q[0] * P.q[0] + P.q[1] * P.q[1] + P.q[2] * P.q[2] + P.q[3] * P.q[3]);
        qk = P.q[lane & 3] / qn;
        const double qw = shfl(qk, 0), qx = shfl(qk, 1), qy = shfl(qk, 2), qz = shfl(qk, 3);
        // diagonal 1 - 2 (p p + q q), off it 2 (p q -+ w r)
        const double v[3] = {qx, qy, qz};
        const int o = a == b ? 0 : 3 - a - b;
        const double p1 = a == b ? v[a == 0 ? 1 : 0] : v[a], q1 = a == b ? p1 : v[b];
        const double p2 = a == b ? v[a == 2 ? 1 : 2] : ((b - a + 3) % 3 == 1 ? -qw : qw), q2 = a == b ? p2 : v[o];
        const double x = p1 * q1 + p2 * q2;
        if (lane < 9) s_Q[lane] = a == b ? 1.0 - 2.0 * x : 2.0 * x;
    } else if (w == 3) {
        if (lit && lvlh) {
            // columns of L: x_b = y_b x z_b, y_b = -h / |h|, h = r x v, z_b = -r / |r|
            const double hc = y[k1] * y[3 + k2] - y[k2] * y[3 + k1];
            const double h0 = shfl(hc, 0), h1 = shfl(hc, 1), h2 = shfl(hc, 2);
            const bool hv = lane & 1;
            const double m0 = hv ? h0 : y[0], m1 = hv ? h1 : y[1], m2 = hv ? h2 : y[2];
            const double q = -1.0 / sqrt(m0 * m0 + m1 * m1 + m2 * m2);
            const double irn = shfl(q, 0), ihn = shfl(q, 1);
            const double zb = y[c3] * irn, yb = hc * ihn;
            const double xb = shfl(yb, k1) * shfl(zb, k2) - shfl(yb, k2) * shfl(zb, k1);
            if (lane < 3) { s_L[3 * lane] = xb; s_L[3 * lane + 1] = yb; s_L[3 * lane + 2] = zb; }
            if (lane < 2) s_in[lane] = q;
        }
        if (P.central == 0 && P.sun3) {
            const double dc = s_rs[c3] - y[c3];
            const double d0 = shfl(dc, 0), d1 = shfl(dc, 1), d2c = shfl(dc, 2);
            const double d2 = d0 * d0 + d1 * d1 + d2c * d2c, dn = sqrt(d2);
            const double da = d0 * ab[0] + d1 * ab[1] + d2c * ab[2];
            const double id3 = 1.0 / (d2 * dn), id5 = id3 / d2;
            const double x = -kMuSun * (ab[c3] * id3 - 3.0 * dc * da * id5);
            if (lane < 3) s_third[lane] = x;
        }
    }
    __syncthreads();
    if (lit && lvlh) {
        // attitude: R = L(y) Q(q): Qb = L^T Rb, Lb = Rb Q^T
        if (w == 1) {
            const double z = s_Rb[3 * a] * s_Q[3 * b] + s_Rb[3 * a + 1] * s_Q[3 * b + 1] + s_Rb[3 * a + 2] * s_Q[3 * b + 2];
            if (lane < 9) s_Lb[lane] = z;
            __syncwarp();
            const double irn = -s_in[0], ihn = -s_in[1];
            const auto col = [&](const double *M, int row, int c) { return M[3 * row + c]; };
            const double ybb = s_Lb[3 * c3 + 1] + (col(s_L, k1, 2) * col(s_Lb, k2, 0) - col(s_L, k2, 2) * col(s_Lb, k1, 0));
            const double zbb = s_Lb[3 * c3 + 2] + (col(s_Lb, k1, 0) * col(s_L, k2, 1) - col(s_Lb, k2, 0) * col(s_L, k1, 1));
            const double hh = -s_L[3 * c3 + 1];  // h / |h|
            const double yd = shfl(ybb, 0) * shfl(hh, 0) + shfl(ybb, 1) * shfl(hh, 1) + shfl(ybb, 2) * shfl(hh, 2);
            const double hb = -(ybb - yd * hh) * ihn;
            const double hb1 = shfl(hb, k1), hb2 = shfl(hb, k2);
            const double rh = -s_L[3 * c3 + 2];  // r / |r|
            const double zd = shfl(zbb, 0) * shfl(rh, 0) + shfl(zbb, 1) * shfl(rh, 1) + shfl(zbb, 2) * shfl(rh, 2);
            const double rb = (y[3 + k1] * hb2 - y[3 + k2] * hb1) - (zbb - zd * rh) * irn;
            const double vb = hb1 * y[k2] - hb2 * y[k1];
            if (lane < 3) { s_rv[lane] = rb; s_rv[3 + lane] = vb; }
        } else if (w == 2) {
            const double x = s_L[a] * s_Rb[b] + s_L[3 + a] * s_Rb[3 + b] + s_L[6 + a] * s_Rb[6 + b];
            if (lane < 9) s_Qb[lane] = x;
        }
        __syncwarp();
    }
    if (w == 2 && lit) {
        // Q of the normalised quaternion, differentiated
        const double q0 = shfl(qk, 0), q1 = shfl(qk, 1), q2 = shfl(qk, 2), q3 = shfl(qk, 3);
        double g[4];
        quat_unit_vjp(q0, q1, q2, q3, lvlh ? s_Qb : s_Rb, g);
        const double gd = g[0] * q0 + g[1] * q1 + g[2] * q2 + g[3] * q3;
        const double gk = lane == 0 ? g[0] : lane == 1 ? g[1] : lane == 2 ? g[2] : g[3];
        const double x = (gk - gd * qk) / qn;
        if (lane < 4) X.qbar[lane] += x;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const bool pos = lane < 3;
        double x = pos ? s_grav[c3] : X.kbar[c3];  // x' = v
        if (pos && P.central == 0 && P.sun3) x += s_third[c3];
        if (pos && lit) x -= s_wb[c3];
        if (lit && lvlh) x += s_rv[lane];
        X.ybar[stage][lane] = x;
    }
}

// attitude quaternion cotangent summed over the trajectories, in order
__global__ void k_adj_prop_qsum(int n, const PropAdj *A, double *out)
{
    if (threadIdx.x >= 4) return;
    double x = 0.0;
    for (int i = 0; i < n; i++) x += A[i].qbar[threadIdx.x];
    out[threadIdx.x] = x;
}

__global__ void k_adj_prop_step(int n, PropAdj *A)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    PropAdj &X = A[i];
    for (int k = 0; k < 6; k++) X.lam[k] += X.ybar[0][k] + X.ybar[1][k] + X.ybar[2][k] + X.ybar[3][k];
}

}  // namespace

cudaError_t launch_prop_init(PropState *S, int n, const double *y0, const double *t01, const PropDev &P,
                             const double *cfg, int *n_done, cudaStream_t st)
{
    k_prop_init<<<(n + 63) / 64, 64, 0, st>>>(S, n, y0, t01, P, cfg, n_done);
    return cudaGetLastError();
}
cudaError_t launch_prop_stage(PropState *S, int n, const PropDev &P, int stage, double *sun_dir, double *sun_dist,
                              cudaStream_t st)
{
    return launch_chained(k_prop_stage, dim3((n + kPropWarps - 1) / kPropWarps), dim3(32 * kPropWarps), 0, st, S, n, P, stage, sun_dir, sun_dist);
}
cudaError_t launch_prop_accel(PropState *S, int n, const PropDev &P, int stage, const double *force, cudaStream_t st,
                              const double *sun_dir, const double *sun_dist)
{
    return launch_chained(k_prop_accel, dim3((n + kPropWarps - 1) / kPropWarps), dim3(32 * kPropWarps), 0, st, S, n, P, stage, force, sun_dir, sun_dist);
}
cudaError_t launch_prop_next(PropState *S, int n, const PropDev &P, int stage, const double *force, double *sun_dir,
                             double *sun_dist, int *n_done, double *h_log, int64_t h_cap, cudaStream_t st)
{
    return launch_chained(k_prop_next, dim3((n + kPropWarps - 1) / kPropWarps), dim3(32 * kPropWarps), 0, st, S, n, P, stage, force, sun_dir, sun_dist,
                          n_done, h_log, h_cap);
}
cudaError_t launch_prop_step(PropState *S, int n, const PropDev &P, double *sun_dir, double *sun_dist, int *n_done,
                             double *h_log, int64_t h_cap, cudaStream_t st)
{
    return launch_chained(k_prop_step, dim3((n + kPropWarps - 1) / kPropWarps), dim3(32 * kPropWarps), 0, st, S, n, P, sun_dir, sun_dist, n_done, h_log, h_cap);
}
cudaError_t launch_prop_control(PropState *S, int n, const PropDev &P, int *n_done, double *h_log, int64_t h_cap,
                                cudaStream_t st)
{
    return launch_chained(k_prop_control, dim3((n + kPropWarps - 1) / kPropWarps), dim3(32 * kPropWarps), 0, st, S, n, P, n_done, h_log, h_cap);
}

cudaError_t launch_prop_ckpt(PropState *S, int n, double *buf, bool save, double h0, cudaStream_t st)
{
    k_prop_ckpt<<<(n + 63) / 64, 64, 0, st>>>(S, n, buf, save ? 1 : 0, h0);
    return cudaGetLastError();
}
cudaError_t launch_prop_record(const PropState *S, int n, const double *sun, const double *dist, const double *force,
                               StageRec *rec, double *rec_sun, double *rec_dist, cudaStream_t st)
{
    k_prop_record<<<(n + 63) / 64, 64, 0, st>>>(S, n, sun, dist, force, rec, rec_sun, rec_dist);
    return cudaGetLastError();
}
cudaError_t launch_adj_prop_in(int n, const PropDev &P, int stage, const StageRec *rec, PropAdj *A, double *g_force,
                               cudaStream_t st)
{
    return launch_chained(k_adj_prop_in, dim3(n), dim3(32), 0, st, n, P, stage, rec, A, g_force);
}
cudaError_t launch_adj_prop_out(int n, const PropDev &P, int stage, const StageRec *rec, PropAdj *A,
                                const double *g_sun, const double *g_dist, cudaStream_t st)
{
    return launch_chained(k_adj_prop_out, dim3(n), dim3(128), 0, st, n, P, stage, rec, A, g_sun, g_dist);
}
cudaError_t launch_adj_prop_qsum(int n, const PropAdj *A, double *out, cudaStream_t st)
{
    k_adj_prop_qsum<<<1, 32, 0, st>>>(n, A, out);
    return cudaGetLastError();
}
cudaError_t launch_adj_prop_step(int n, PropAdj *A, cudaStream_t st)
{
    k_adj_prop_step<<<(n + 63) / 64, 64, 0, st>>>(n, A);
    return cudaGetLastError();
}

}  // namespace srp
