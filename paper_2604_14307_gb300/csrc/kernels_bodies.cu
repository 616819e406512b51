// Rigid-body and surface-site kernels (Sec. II.B and II.B.2 of arXiv 2604.14307).
//
// k_body_md     (the transfer's sum,) first velocity-Verlet half kick, drift of R,
//               and the Miller et al. NO_SQUISH free-rotor sequence 3-2-1-2-3 for
//               q and its conjugate momentum p = 2 q (x) (0, L_body), formed from
//               the stored space-frame L and converted back; four lanes per body.
//               Finishes the force pass where no two bodies share a box.
// k_body_centres the space-frame offsets Q c of every WCA centre, once per pose
//               (k_body_md writes them for shapes of one or two centres).
// k_body_force  core-shifted WCA (Eq. 1) between the centres of different
//               bodies of a replica, with torques, over Verlet neighbour lists
//               (FP32 bounding-sphere prefilter); eight lanes per body for
//               shapes of one or two centres, one warp per body otherwise;
//               the pair arithmetic in the form's precision (FP32 for P32),
//               forces and torques summed in FP64; optional second kick.
// k_vacf_sample per-body velocity autocorrelation sums (Sec. III.A).
// k_sites_pre   one CTA per body: site positions from the pose, Maxwell-
//               Boltzmann draws, per-body mean velocity and angular velocity of
//               the draws, thermalised site velocity of Eq. 7, binning of the
//               sites into the cell sums.
// k_sites_post  one CTA per body: site collision with the cell parameters,
//               segmented reduction of dP = sum m (v' - v) and
//               dL = sum d x m (v' - v) (Eqs. 3-4) into the body's momenta;
//               the sites are reset to rigid motion (Eq. 5) implicitly, since
//               the next step recomputes them from P and L.  The ANG instance
//               (angular-momentum-conserving variants) adds the cell's
//               rigid-rotation correction to the rule's velocity first.
// k_ang_sites   the sites' terms of the +a cell words, from the thermalised
//               and the rule's velocities (the latter recomputed with the POST
//               coupling's arithmetic).
// This file is compiled without fused multiply-add so that the FP64 body and
// site-position arithmetic rounds the same way as the oracle.
#include "solvent_device.cuh"

namespace mpcd {

// The kernels of the body chain (POST, body step, forces, PRE) follow one
// another on one stream and are short: each may start while the one before it
// still runs (programmatic dependent launch), and does up to chain_wait() what
// needs nothing of it - for PRE the thermal draws of all sites.  A kernel lets
// the next one start with chain_next(); the next one's chain_wait() returns
// when all of it has completed, and since every kernel of the chain waits,
// when everything before it has.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
static void launch(void (*kernel)(P...), bool chained, unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                   A... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = chained ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);   // the caller reads the launch status
}
// Not beside the passes that already fill what an early kernel would take: the
// MPCD-AT solvent pass (issue slots, registers: 221 bodies 59.3 us per step,
// 62.6 chained) and the FP64 forms (FP64 pipes: 113 bodies 310 and 319).  FP32
// SRD gains the launch gaps and the draws: one body 30.1 -> 27.5, 191 bodies
// unpipelined 310 -> 302, 453 bodies 102 -> 99-102.
static bool chain_pays(const StepArgs &a) { return a.precision == 1 && a.rule == 0; }

template <typename... P, typename... A>
static void launch_chained(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                           const StepArgs &a, A... args)
{
    launch(kernel, chain_pays(a), grid, block, smem, s, a, args...);
}

// a slab of a decomposed box owns the sites whose stored z lies in its range
// (bounds are integers: the comparison is exact in either precision)
template <typename Real>
__device__ __forceinline__ bool site_owned(const StepArgs &a, Real z)
{
    return !a.site_own || (z >= (Real)a.site_zlo && z < (Real)a.site_zhi);
}


// ------------------------------------------------------------- quaternions
// rotation matrix of a unit quaternion (w, x, y, z), body -> space
__device__ __forceinline__ void rotmat(const double q[4], double Q[9])
{
    double xx = q[1] * q[1], yy = q[2] * q[2], zz = q[3] * q[3];
    double xy = q[1] * q[2], xz = q[1] * q[3], yz = q[2] * q[3];
    double wx = q[0] * q[1], wy = q[0] * q[2], wz = q[0] * q[3];
    Q[0] = 1.0 - 2.0 * (yy + zz); Q[1] = 2.0 * (xy - wz);       Q[2] = 2.0 * (xz + wy);
    Q[3] = 2.0 * (xy + wz);       Q[4] = 1.0 - 2.0 * (xx + zz); Q[5] = 2.0 * (yz - wx);
    Q[6] = 2.0 * (xz - wy);       Q[7] = 2.0 * (yz + wx);       Q[8] = 1.0 - 2.0 * (xx + yy);
}
__device__ __forceinline__ void mv(const double Q[9], const double x[3], double o[3])
{
    for (int a = 0; a < 3; ++a) o[a] = (Q[3 * a] * x[0] + Q[3 * a + 1] * x[1]) + Q[3 * a + 2] * x[2];
}
__device__ __forceinline__ void mtv(const double Q[9], const double x[3], double o[3])
{
    for (int a = 0; a < 3; ++a) o[a] = (Q[a] * x[0] + Q[3 + a] * x[1]) + Q[6 + a] * x[2];
}

__device__ __forceinline__ float wrapf(float y, float L, int &bad)
{
    if (y >= L) y = y - L;
    else if (y < 0.0f) { y = y + L; if (y >= L) y = 0.0f; }
    bad |= !(y >= 0.0f && y < L);
    return y;
}

// ------------------------------------------------- bodies, lane parallel
// A warp-wide FP64 instruction takes 64 cycles of its SM sub-partition however
// many lanes it has (measured: 64.2 cycles with 1 to 32 active lanes, four
// warps on four sub-partitions at once), so the rigid-body arithmetic is
// bound by the number of FP64 instructions a warp executes one after another,
// not by its operations.  A body is therefore spread over four lanes: lane c
// holds component c of its quaternion and conjugate momentum and component c of
// its vectors (lane 3 repeats lane 0's vector work), each component is formed
// by the expression of the scalar form, in the same order, and components of
// the other lanes come by shuffles.  The body step of one body went from 27 to
// 12 us with the transfer's sum and the centres in the same launch (36 us in three).
__device__ __forceinline__ double lane4(double v, int c) { return __shfl_sync(0xffffffffu, v, c, 4); }
__device__ __forceinline__ float lane4(float v, int c) { return __shfl_sync(0xffffffffu, v, c, 4); }
__device__ __forceinline__ double flip(double v, bool neg)   // -v if neg, exactly
{
    return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}

// component c of the quaternion product (quat_mul); a, b: lane c's component
__device__ __forceinline__ double lane_qmul(double a, double b, int c)
{
    const double t0 = lane4(a, 0) * lane4(b, c), t1 = lane4(a, 1) * lane4(b, c ^ 1);
    const double t2 = lane4(a, 2) * lane4(b, c ^ 2), t3 = lane4(a, 3) * lane4(b, c ^ 3);
    return ((t0 + flip(t1, c == 0 || c == 2)) + flip(t2, c == 0 || c == 3)) + flip(t3, c < 2);
}
// (0, v) as a quaternion from vector component lanes, and back (lane 3: component 0)
__device__ __forceinline__ double lane_vec_to_quat(double v, int c)
{
    const double t = lane4(v, (c + 3) & 3);
    return c == 0 ? 0.0 : t;
}
__device__ __forceinline__ double lane_quat_to_vec(double t, int c) { return lane4(t, c == 3 ? 1 : c + 1); }

// row and column c of the rotation matrix (rotmat) of the quaternion q
struct LaneRot { double r[3], c[3]; };
__device__ __forceinline__ LaneRot lane_rot(double q, int c)
{
    const int i = c == 3 ? 0 : c, j = i == 2 ? 0 : i + 1, l = i == 0 ? 2 : i - 1;
    const double w = lane4(q, 0), qi = lane4(q, 1 + i), qj = lane4(q, 1 + j), ql = lane4(q, 1 + l);
    const double dii = 1.0 - 2.0 * (qj * qj + ql * ql);
    const double ij = qi * qj, il = qi * ql, wl = w * ql, wj = w * qj;
    const double rij = 2.0 * (ij - wl), ril = 2.0 * (il + wj), cji = 2.0 * (ij + wl), cli = 2.0 * (il - wj);
    LaneRot o;
    o.r[0] = i == 0 ? dii : (i == 1 ? ril : rij); o.c[0] = i == 0 ? dii : (i == 1 ? cli : cji);
    o.r[1] = i == 0 ? rij : (i == 1 ? dii : ril); o.c[1] = i == 0 ? cji : (i == 1 ? dii : cli);
    o.r[2] = i == 0 ? ril : (i == 1 ? rij : dii); o.c[2] = i == 0 ? cli : (i == 1 ? cji : dii);
    return o;
}
__device__ __forceinline__ double lane_dot(const double (&m)[3], double x)
{
    return (m[0] * lane4(x, 0) + m[1] * lane4(x, 1)) + m[2] * lane4(x, 2);
}
__device__ __forceinline__ double lane_mv(const LaneRot &Q, double x) { return lane_dot(Q.r, x); }
__device__ __forceinline__ double lane_mtv(const LaneRot &Q, double x) { return lane_dot(Q.c, x); }

__device__ __forceinline__ double lane_L_to_p(double q, const LaneRot &Q, double L, int c)
{
    return 2.0 * lane_qmul(q, lane_vec_to_quat(lane_mtv(Q, L), c), c);
}
__device__ __forceinline__ double lane_p_to_Lb(double q, double p, int c)   // vec(q* (x) p) / 2
{
    return 0.5 * lane_quat_to_vec(lane_qmul(flip(q, c != 0), p, c), c);
}
__device__ __forceinline__ double lane_torque_kick(double q, const LaneRot &Q, double T, double h, int c)
{
    return 2.0 * h * lane_qmul(q, lane_vec_to_quat(lane_mtv(Q, T), c), c);
}
// free rotation about body axis k (rotor); Ih its moment, r4 = RN(1 / (4 Ih)).
// No rotation about an axis without a moment: that is one body's matter, and the
// warp holds eight of any shape, so every lane takes part in the shuffles first.
__device__ __forceinline__ void lane_rotor(double &q, double &p, int k, double h, double Ih, double r4, int c)
{
    const bool neg = k == 1 ? (c == 0 || c == 3) : (k == 2 ? c < 2 : (c == 0 || c == 2));
    const double Pq = flip(lane4(q, c ^ k), neg), Pp = flip(lane4(p, c ^ k), neg);
    const double t = p * Pq;
    const double dot = ((lane4(t, 0) + lane4(t, 1)) + lane4(t, 2)) + lane4(t, 3);
    if (Ih == 0.0) return;
    const double zeta = div_by(dot, 4.0 * Ih, r4);
    double sn, cs;
    sincos(zeta * h, &sn, &cs);
    q = cs * q + sn * Pq;
    p = cs * p + sn * Pp;
}

// Forces done: external force, stored F and T, the second half kick (kick) and
// the pose record the site kernels read, in two parts that share nothing, so
// that different warps can take them.  Component c of every vector on lane c;
// store: this lane writes (lane 3 and repeated lanes do not).
__device__ __forceinline__ void lane_finish_linear(const StepArgs &a, int64_t i, const DevShape &sh, double R, double P,
                                                   double F, int kick, int k, bool store)
{
    F += a.fext[k];   // external force at the centre of mass (no torque)
    if (kick) P = P + 0.5 * a.dt * F;
    const double V = div_by(P, sh.M, sh.rM);
    if (!store) return;
    DevBody *o = a.bodies + i;
    o->F[k] = F;
    if (kick) o->P[k] = P;
    double *p64 = a.pose64 + i * POSE_W;
    float *p32 = a.pose32 + i * POSE_W;
    p64[9 + k] = R; p32[9 + k] = (float)R;
    p64[12 + k] = V; p32[12 + k] = (float)V;
}
__device__ __forceinline__ void lane_finish_angular(const StepArgs &a, int64_t i, const DevShape &sh, double q, double L,
                                                    double T, int kick, int c, bool store)
{
    const int k = c == 3 ? 0 : c;
    const LaneRot Q = lane_rot(q, c);
    if (kick) {
        double p = lane_L_to_p(q, Q, L, c);
        p += lane_torque_kick(q, Q, T, 0.5 * a.dt, c);
        L = lane_mv(Q, lane_p_to_Lb(q, p, c));
    }
    // omega = Q Ihat^-1 Q^T L (Eq. 5)
    const double Lb = lane_mtv(Q, L);
    const double wb = sh.Ihat[k] > 0.0 ? div_by(Lb, sh.Ihat[k], sh.rI[k]) : 0.0;
    const double W = lane_mv(Q, wb);
    if (!store) return;
    DevBody *o = a.bodies + i;
    o->T[k] = T;
    if (kick) o->Lm[k] = L;
    double *p64 = a.pose64 + i * POSE_W;
    float *p32 = a.pose32 + i * POSE_W;
    for (int m = 0; m < 3; ++m) { p64[3 * k + m] = Q.r[m]; p32[3 * k + m] = (float)Q.r[m]; }
    p64[15 + k] = W; p32[15 + k] = (float)W;
}

// --------------------------------------------------------------- body MD
// IMPULSE: first adds the transfer's per-warp partial sums (the work of
// k_body_impulse, for the step pipeline, where nothing stands between the two).
// LONE: every replica has one body at most, so no force acts between bodies and
// the force pass is finished here.  Also writes the space-frame WCA centres of
// shapes with one or two of them.
// Two warps take eight bodies: one their rotation, one their translation.
constexpr int MD_BODIES = 8;
template <typename Real, bool IMPULSE, bool LONE>
__global__ void __launch_bounds__(64) k_body_md(StepArgs a)
{
    const int g = (int)(blockIdx.x * MD_BODIES + ((threadIdx.x & 31) >> 2));
    const bool linear = threadIdx.x >= 32;
    const int c = threadIdx.x & 3, k = c == 3 ? 0 : c;
    const bool valid = g < a.n_bodies;
    const int i = valid ? g : a.n_bodies - 1;   // every lane takes part in the shuffles
    const bool store = valid && c < 3;
    DevBody *o = a.bodies + i;
    const DevShape &sh = a.shapes[o->shape];
    const DevReplica &r = a.reps[o->rep];
    const double dt = a.dt;
    // component k (3 + k) of the transfer, with IMPULSE
    const Real *in = reinterpret_cast<const Real *>(a.partial) + (int64_t)i * SITE_WARPS * 6 + (linear ? k : 3 + k);
    auto transfer = [&]() {
        double s = 0.0;
        for (int w = 0; w < SITE_WARPS; ++w) s += (double)in[w * 6];
        return s;
    };
    chain_next();
    if (!IMPULSE) chain_wait();
    // with IMPULSE the pass before is POST, which writes only the partial sums
    if (linear) {
        int bad = 0;
        double P = o->P[k], R = o->R[k];
        const double kickF = 0.5 * dt * o->F[k], D0 = o->D[k];
        const float4 p0 = a.bpos_build[i];
        const float h = 0.5f * r.L[k], bound = (float)sh.bound;
        if (IMPULSE) {
            chain_wait();
            P += transfer();
        }
        P += kickF;
        const double d = dt * div_by(P, sh.M, sh.rM);
        const double D = D0 + d;
        R = wrap_box(R + d, (double)r.L[k], bad);
        if (store) { o->R[k] = R; o->D[k] = D; }
        if (store && !LONE) o->P[k] = P;
        // neighbour lists stay valid while every body is within half the skin of
        // its position at the last build
        const float Rf = (float)R;
        float dx = Rf - (k == 0 ? p0.x : (k == 1 ? p0.y : p0.z));
        dx = dx > h ? dx - r.L[k] : (dx < -h ? dx + r.L[k] : dx);
        const float x2 = dx * dx;
        const float d2 = ((0.0f + lane4(x2, 0)) + lane4(x2, 1)) + lane4(x2, 2);
        const float4 at = make_float4(lane4(Rf, 0), lane4(Rf, 1), lane4(Rf, 2), bound);
        if (valid && c == 3) {
            a.bpos[i] = at;
            if (!LONE && d2 > 0.25f * NLIST_SKIN * NLIST_SKIN) atomicOr(a.nl_dirty, 1);
        }
        if (store && bad) atomicOr(a.d_err, ERR_POSITION);
        if (LONE) lane_finish_linear(a, i, sh, R, P, 0.0, 1, k, store);
        return;
    }
    double q = o->q[c], L = o->Lm[k];
    LaneRot Q = lane_rot(q, c);
    const double kickT = lane_torque_kick(q, Q, o->T[k], 0.5 * dt, c);
    if (IMPULSE) {
        chain_wait();
        L += transfer();
    }
    double p = lane_L_to_p(q, Q, L, c);
    p += kickT;
#pragma unroll 1
    for (int e = 0; e < 5; ++e) {   // axes 3, 2, 1, 2, 3
        const int ax = e < 3 ? 3 - e : e - 1;
        lane_rotor(q, p, ax, e == 2 ? dt : 0.5 * dt, sh.Ihat[ax - 1], sh.r4I[ax - 1], c);
    }
    const double qq = q * q;
    q /= sqrt(((lane4(qq, 0) + lane4(qq, 1)) + lane4(qq, 2)) + lane4(qq, 3));
    Q = lane_rot(q, c);
    L = lane_mv(Q, lane_p_to_Lb(q, p, c));
    if (store && !LONE) o->Lm[k] = L;
    if (valid) o->q[c] = q;
    if (a.max_cent <= 2)
        for (int e = 0; e < sh.n_cent; ++e) {
            const double *t = a.tcent + 3 * (sh.cent_begin + e);
            const double x = (Q.r[0] * t[0] + Q.r[1] * t[1]) + Q.r[2] * t[2];
            if (store) {
                a.cent64[3 * (o->cent_begin + e) + k] = x;
                reinterpret_cast<float *>(a.cent32 + o->cent_begin + e)[k] = (float)x;
            }
        }
    if (LONE) lane_finish_angular(a, i, sh, q, L, 0.0, 1, c, store);
}

__global__ void k_body_pos(StepArgs a)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n_bodies) return;
    const DevBody &b = a.bodies[i];
    a.bpos[i] = make_float4((float)b.R[0], (float)b.R[1], (float)b.R[2], (float)a.shapes[b.shape].bound);
}

template <typename Real>
static void body_md(const StepArgs &a, bool impulse, cudaStream_t s)
{
    const unsigned grid = (unsigned)((a.n_bodies + MD_BODIES - 1) / MD_BODIES);
    // Without solvent nothing stands between the step counter's advance and the
    // first body step of a call, which lets PRE start and read the counter
    // before anything has waited for it: a full dependency there.
    const bool chained = chain_pays(a) && (impulse || a.n_tiles > 0);
    if (a.lone_bodies) {
        if (impulse) launch(k_body_md<Real, true, true>, chained, grid, 64, 0, s, a);
        else launch(k_body_md<Real, false, true>, chained, grid, 64, 0, s, a);
    } else {
        if (impulse) launch(k_body_md<Real, true, false>, chained, grid, 64, 0, s, a);
        else launch(k_body_md<Real, false, false>, chained, grid, 64, 0, s, a);
    }
}

void launch_body_md(const StepArgs &a, bool impulse, cudaStream_t s)
{
    if (a.n_bodies == 0) return;
    if (a.precision == 1) body_md<float>(a, impulse, s);
    else body_md<double>(a, impulse, s);
}

// ------------------------------------------------------------ WCA forces
// Rotated WCA centres of every body, Q c in the space frame, once per pose (in
// FP64 and rounded to float), so that the pair loop below only adds offsets.
// One warp per body, one centre per lane: the rotation matrix is formed once
// for all of them (1120 bodies of up to 19 centres: 6.6 us, 19.6 with one
// thread per body).
__global__ void __launch_bounds__(128) k_body_centres(StepArgs a)
{
    const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (i >= a.n_bodies) return;
    const DevBody &b = a.bodies[i];
    const DevShape &sh = a.shapes[b.shape];
    chain_next();
    chain_wait();
    double Q[9];
    rotmat(b.q, Q);
    for (int c = threadIdx.x & 31; c < sh.n_cent; c += 32) {
        double d[3];
        mv(Q, a.tcent + 3 * (sh.cent_begin + c), d);
        const int64_t g = b.cent_begin + c;
        for (int k = 0; k < 3; ++k) a.cent64[3 * g + k] = d[k];
        a.cent32[g] = make_float4((float)d[0], (float)d[1], (float)d[2], 0.0f);
    }
}

template <typename Real> struct CentreOf;
template <> struct CentreOf<float> {
    __device__ static void get(const StepArgs &a, int64_t g, float c[3])
    {
        const float4 v = a.cent32[g];
        c[0] = v.x; c[1] = v.y; c[2] = v.z;
    }
};
template <> struct CentreOf<double> {
    __device__ static void get(const StepArgs &a, int64_t g, double c[3])
    {
        c[0] = a.cent64[3 * g]; c[1] = a.cent64[3 * g + 1]; c[2] = a.cent64[3 * g + 2];
    }
};

// WCA force (Eq. 1) between centre c_a of body i and centre c_c of body j; dR =
// R_i - R_j, formed in FP64 and rounded to the form's precision.  The
// centre-pair vector dR + (c_a - c_c) takes its own minimum image.  Real =
// float for the P32 form, double for the P64 form.  False beyond the cutoff.
template <typename Real>
__device__ __forceinline__ bool centre_force(Real dij, const Real (&dR)[3], const Real (&c_a)[3], const Real (&c_c)[3],
                                             const DevReplica &r, Real (&f)[3])
{
    const Real rc_extra = Real(1.122462048309373);   // 2^(1/6) sigma
    const Real delta = dij - Real(1), rcut = delta + rc_extra;
    Real dv[3];
    for (int k = 0; k < 3; ++k) {
        dv[k] = dR[k] + (c_a[k] - c_c[k]);
        const Real L = (Real)r.L[k], h = Real(0.5) * L;
        if (dv[k] > h) dv[k] -= L;
        else if (dv[k] < -h) dv[k] += L;
    }
    const Real rr = sqrt(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
    if (!(rr <= rcut)) return false;
    const Real sdl = Real(1) / (rr - delta);
    const Real s6 = sdl * sdl * sdl * sdl * sdl * sdl;
    const Real fm = Real(4) * (Real(12) * s6 * s6 - Real(6) * s6) / (rr - delta);
    for (int k = 0; k < 3; ++k) f[k] = fm * dv[k] / rr;
    return true;
}

__device__ __forceinline__ bool may_interact(const StepArgs &a, const float4 &pi, const float4 &pj,
                                             const DevReplica &r, float reach)
{
    const float hx = 0.5f * r.L[0], hy = 0.5f * r.L[1], hz = 0.5f * r.L[2];
    float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
    dx = dx > hx ? dx - r.L[0] : (dx < -hx ? dx + r.L[0] : dx);
    dy = dy > hy ? dy - r.L[1] : (dy < -hy ? dy + r.L[1] : dy);
    dz = dz > hz ? dz - r.L[2] : (dz < -hz ? dz + r.L[2] : dz);
    const float lim = pi.w + pj.w + reach;
    return dx * dx + dy * dy + dz * dz <= lim * lim;
}

// candidate neighbours of each body within the bounding spheres + cutoff + skin
__global__ void k_nlist_build(StepArgs a)
{
    chain_next();
    chain_wait();
    if (!*a.nl_dirty) return;
    const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= a.n_bodies) return;
    const DevBody &bi = a.bodies[i];
    const DevShape &si = a.shapes[bi.shape];
    const DevReplica r = a.reps[bi.rep];
    const float4 pi = a.bpos[i];
    const float reach = (float)(0.5 * (si.wca_d + a.max_wca_d) - 1.0 + 1.122462048309373) + NLIST_SKIN + 1e-2f;
    int count = 0;
    for (int64_t j0 = r.body_begin; j0 < r.body_end; j0 += 32) {
        const int64_t j = j0 + lane;
        bool hit = j < r.body_end && j != i && may_interact(a, pi, a.bpos[j], r, reach);
        unsigned m = __ballot_sync(0xffffffffu, hit);
        int slot = count + __popc(m & ((1u << lane) - 1u));
        if (hit && slot < NLIST_MAX) a.nlist[(int64_t)i * NLIST_MAX + slot] = (int32_t)j;
        count += __popc(m);
    }
    if (lane == 0) {
        a.ncount[i] = count <= NLIST_MAX ? count : -1;
        a.bpos_build[i] = pi;
    }
}

// Shapes of one or two centres (spheres, dumbbells): eight lanes per body.
// The lanes take the body's candidates eight at a time, one candidate each;
// the forces of those in reach are then added in candidate order, component k
// on lane k, so the sums are those of a serial loop.  Rebuilds the body's
// candidate list first when the lists are out of date (the flag is cleared by
// the next site PRE pass).  One thread per body, in turn over its candidates,
// took 7.5 us for a body without any and 11-16 us at 221 bodies (with the list
// pass and the centres in launches of their own); now 5.5 and 9.5 us in all.
template <typename Real, int MAXC>
__global__ void __launch_bounds__(128) k_body_force(StepArgs a, int kick)
{
    constexpr int NP = MAXC * MAXC;
    __shared__ double sF[16][3], sT[16][3];   // the CTA's 16 bodies
    const unsigned full = 0xffffffffu;
    const int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    const int sub = threadIdx.x & 7, gsh = threadIdx.x & 24;   // lane of the body, its first lane in the warp
    const int k = (sub & 3) == 3 ? 0 : sub & 3, k1 = k == 2 ? 0 : k + 1, k2 = k == 0 ? 2 : k - 1;
    const bool valid = g < a.n_bodies;
    const int64_t i = valid ? g : a.n_bodies - 1;   // every lane takes part in the votes and shuffles
    const DevBody &bi = a.bodies[i];
    const DevShape &si = a.shapes[bi.shape];
    const DevReplica r = a.reps[bi.rep];
    const float cut = (float)(0.5 * (si.wca_d + a.max_wca_d) - 1.0 + 1.122462048309373);
    chain_wait();
    chain_next();
    // (loads that do not wait for one another)
    const int dirty = *a.nl_dirty;
    const float4 pi = a.bpos[i];
    const int32_t near0 = a.nlist[i * NLIST_MAX + sub];   // the first candidates, if the list holds
    int n = a.ncount[i];
    if (dirty) {
        // candidates within the bounding spheres + cutoff + skin, ascending
        const float reach = cut + NLIST_SKIN + 1e-2f;
        n = 0;
        constexpr int U = 4;   // position loads in flight per lane
        for (int64_t j0 = r.body_begin; __any_sync(full, j0 < r.body_end); j0 += 8 * U) {
            float4 pj[U];
#pragma unroll
            for (int u = 0; u < U; ++u) pj[u] = a.bpos[min(j0 + 8 * u + sub, r.body_end - 1)];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t j = j0 + 8 * u + sub;
                const bool hit = j < r.body_end && j != i && may_interact(a, pi, pj[u], r, reach);
                const unsigned m = (__ballot_sync(full, hit) >> gsh) & 0xffu;
                const int slot = n + __popc(m & ((1u << sub) - 1u));
                if (valid && hit && slot < NLIST_MAX) a.nlist[i * NLIST_MAX + slot] = (int32_t)j;
                n += __popc(m);
            }
        }
        n = n <= NLIST_MAX ? n : -1;
        if (valid && sub == 0) {
            a.ncount[i] = n;
            a.bpos_build[i] = pi;
        }
        __syncwarp();   // the list is read by the body's other lanes
    }
    const bool listed = n >= 0 && n <= NLIST_MAX;
    const int64_t total = !valid ? 0 : (listed ? n : r.body_end - r.body_begin);
    double F = 0.0, T = 0.0;
    for (int64_t e0 = 0; __any_sync(full, e0 < total); e0 += 8) {
        const int64_t e = e0 + sub;
        bool on = e < total;
        int64_t j = i;
        if (on) {
            j = !listed ? r.body_begin + e : (e0 == 0 && !dirty ? near0 : a.nlist[i * NLIST_MAX + e]);
            on = j >= r.body_begin && j < r.body_end;
            if (!listed) on = on && j != i && may_interact(a, pi, a.bpos[j], r, cut + 1e-2f);
        }
        Real f[NP][3];
        unsigned near[NP], some = 0;
        {
            const DevBody &bj = a.bodies[on ? j : i];
            const DevShape &sj = a.shapes[bj.shape];
            const Real dij = Real(0.5 * (si.wca_d + sj.wca_d));
            Real dR[3];
            for (int m = 0; m < 3; ++m) dR[m] = (Real)(bi.R[m] - bj.R[m]);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const int ca = p / MAXC, cc = p % MAXC;
                bool hit = on && ca < si.n_cent && cc < sj.n_cent;
                if (hit) {
                    Real ci[3], cj[3];
                    CentreOf<Real>::get(a, bi.cent_begin + ca, ci);
                    CentreOf<Real>::get(a, bj.cent_begin + cc, cj);
                    hit = centre_force<Real>(dij, dR, ci, cj, r, f[p]);
                }
                near[p] = (__ballot_sync(full, hit) >> gsh) & 0xffu;
                some |= near[p];
            }
        }
        while (__any_sync(full, some != 0)) {   // the body's candidates in reach, in order
            const int src = some ? __ffs(some) - 1 : 0;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                Real t[3];
                for (int m = 0; m < 3; ++m) t[m] = __shfl_sync(full, f[p][m], src, 8);
                if (some && (near[p] >> src & 1u)) {
                    Real ci[3];
                    CentreOf<Real>::get(a, bi.cent_begin + p / MAXC, ci);
                    const double f1 = (double)(k == 0 ? t[1] : (k == 1 ? t[2] : t[0]));
                    const double f2 = (double)(k == 0 ? t[2] : (k == 1 ? t[0] : t[1]));
                    F += (double)(k == 0 ? t[0] : (k == 1 ? t[1] : t[2]));
                    T += (double)ci[k1] * f2 - (double)ci[k2] * f1;
                }
            }
            some &= some - 1;
        }
    }
    if (sub < 3) {
        sF[threadIdx.x >> 3][k] = F;
        sT[threadIdx.x >> 3][k] = T;
    }
    __syncthreads();
    // four lanes per body: two warps for the angular part, two for the linear one
    const int m = (threadIdx.x & 63) >> 2, cm = threadIdx.x & 3, km = cm == 3 ? 0 : cm;
    const int64_t gm = (int64_t)blockIdx.x * 16 + m, im = min(gm, (int64_t)a.n_bodies - 1);
    const DevBody &bm = a.bodies[im];
    const DevShape &sm = a.shapes[bm.shape];
    const bool store = gm < a.n_bodies && cm < 3;
    if (threadIdx.x < 64)
        lane_finish_angular(a, im, sm, bm.q[cm], bm.Lm[km], sT[m][km], kick, cm, store);
    else
        lane_finish_linear(a, im, sm, bm.R[km], bm.P[km], sF[m][km], kick, km, store);
}

// One warp per body (shapes with many centres, e.g. rods): triple t = ((candidate
// e) n_centres + own centre) max_centres + its centre belongs to lane t mod 32,
// each lane sums its triples in order, and a fixed shuffle tree adds the lanes,
// so the result depends only on the candidate list.  A row of triples (candidate,
// own centre) is left out when the own centre is further from the candidate than
// its bounding sphere and the cutoff reach, which adds nothing: the lanes test 32
// rows at a time, and one row at a time is summed (rods see most bodies of a box
// as candidates, but few of their own centres lie near each).  What belongs to a candidate
// - R_i - R_j and the mean diameter, formed in FP64, and where its centres lie -
// is formed once and kept in shared memory: nine FP64 instructions per triple and
// the loads one behind the other were most of the pass (1120 bodies of up to 19
// centres: 200 us, 147 with R_i - R_j kept, 95 with all, 40 with rows left out).
constexpr int WARP_BODIES = 4;   // bodies (warps) per CTA
template <typename Real>
__global__ void __launch_bounds__(32 * WARP_BODIES) k_body_force_warp(StepArgs a, int kick)
{
    __shared__ Real sdR[WARP_BODIES][NLIST_MAX][3], sdij[WARP_BODIES][NLIST_MAX];
    __shared__ int64_t scent[WARP_BODIES][NLIST_MAX];
    __shared__ float sreach[WARP_BODIES][NLIST_MAX];   // squared, of a row
    __shared__ int sncent[WARP_BODIES][NLIST_MAX];
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (i >= a.n_bodies) return;   // uniform over the warp
    const DevBody &bi = a.bodies[i];
    const DevShape &si = a.shapes[bi.shape];
    const DevReplica r = a.reps[bi.rep];
    chain_wait();
    chain_next();
    double F[3] = {0, 0, 0}, T[3] = {0, 0, 0};
    const int64_t cent_i = bi.cent_begin;
    auto pair = [&](const Real (&dR)[3], Real dij, int64_t cent_j, int ca, int cc) {
        Real ci[3], cj[3], f[3];
        CentreOf<Real>::get(a, cent_i + ca, ci);
        CentreOf<Real>::get(a, cent_j + cc, cj);
        if (!centre_force<Real>(dij, dR, ci, cj, r, f)) return;
        for (int k = 0; k < 3; ++k) F[k] += (double)f[k];
        T[0] += (double)ci[1] * (double)f[2] - (double)ci[2] * (double)f[1];
        T[1] += (double)ci[2] * (double)f[0] - (double)ci[0] * (double)f[2];
        T[2] += (double)ci[0] * (double)f[1] - (double)ci[1] * (double)f[0];
    };
    const int n = a.ncount[i];
    const int nci = si.n_cent, maxc = max(a.max_cent, 1);
    if (n >= 0 && n <= NLIST_MAX) {
        for (int e = lane; e < n; e += 32) {
            const int64_t j = a.nlist[i * NLIST_MAX + e];
            const bool on = j >= r.body_begin && j < r.body_end;
            const DevBody &bj = a.bodies[on ? j : i];
            const DevShape &sj = a.shapes[bj.shape];
            for (int k = 0; k < 3; ++k) sdR[wid][e][k] = (Real)(bi.R[k] - bj.R[k]);
            sdij[wid][e] = Real(0.5 * (si.wca_d + sj.wca_d));
            scent[wid][e] = bj.cent_begin;
            sncent[wid][e] = on ? sj.n_cent : 0;
            const float reach = (float)(sj.bound + 0.5 * (si.wca_d + sj.wca_d) - 1.0 + 1.122462048309373) + 1e-2f;
            sreach[wid][e] = on ? reach * reach : -1.0f;
        }
        __syncwarp();
        const float L[3] = {(float)r.L[0], (float)r.L[1], (float)r.L[2]};
        for (int r0 = 0; r0 < n * nci; r0 += 32) {
            const int row = r0 + lane, e = row / nci, ca = row - e * nci;
            bool near = row < n * nci;
            if (near) {
                Real ci[3];
                CentreOf<Real>::get(a, cent_i + ca, ci);
                float d2 = 0.0f;
                for (int k = 0; k < 3; ++k) {   // the nearest image: no image of the pair is closer
                    float d = (float)sdR[wid][e][k] + (float)ci[k];
                    d -= L[k] * rintf(d / L[k]);
                    d2 += d * d;
                }
                near = d2 <= sreach[wid][e];
            }
            for (unsigned left = __ballot_sync(0xffffffffu, near); left; left &= left - 1) {
                const int src = __ffs(left) - 1;
                const int en = __shfl_sync(0xffffffffu, e, src), cn = __shfl_sync(0xffffffffu, ca, src);
                const unsigned t0 = (unsigned)(r0 + src) * (unsigned)maxc;   // its low bits name the lanes
                for (int c0 = 0; c0 < maxc; c0 += 32) {
                    const int cc = c0 + (int)(((unsigned)lane - t0 - (unsigned)c0) & 31u);
                    if (cc < sncent[wid][en]) pair(sdR[wid][en], sdij[wid][en], scent[wid][en], cn, cc);
                }
            }
        }
    } else {
        // the list overflowed: every body of the replica, prefiltered
        const float4 pi = a.bpos[i];
        const float reach = (float)(0.5 * (si.wca_d + a.max_wca_d) - 1.0 + 1.122462048309373) + 1e-2f;
        for (int64_t j = r.body_begin + lane; j < r.body_end; j += 32) {
            if (j == i || !may_interact(a, pi, a.bpos[j], r, reach)) continue;
            const DevBody &bj = a.bodies[j];
            const DevShape &sj = a.shapes[bj.shape];
            Real dR[3];
            for (int k = 0; k < 3; ++k) dR[k] = (Real)(bi.R[k] - bj.R[k]);
            const Real dij = Real(0.5 * (si.wca_d + sj.wca_d));
            for (int ca = 0; ca < nci; ++ca)
                for (int cc = 0; cc < sj.n_cent; ++cc) pair(dR, dij, bj.cent_begin, ca, cc);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            F[k] += __shfl_down_sync(0xffffffffu, F[k], o);
            T[k] += __shfl_down_sync(0xffffffffu, T[k], o);
        }
    const int c = lane & 3, k = c == 3 ? 0 : c;
    double Fk = 0.0, Tk = 0.0;
    for (int m = 0; m < 3; ++m) {   // lane 0's sums, component k to lane k
        const double f = __shfl_sync(0xffffffffu, F[m], 0), t = __shfl_sync(0xffffffffu, T[m], 0);
        if (m == k) { Fk = f; Tk = t; }
    }
    lane_finish_linear(a, i, si, bi.R[k], bi.P[k], Fk, kick, k, lane < 3);
    lane_finish_angular(a, i, si, bi.q[c], bi.Lm[k], Tk, kick, c, lane < 3);
    if (i == 0 && lane == 0) *a.nl_dirty = 0;   // the lists used by this step are fresh
}

void launch_body_force(const StepArgs &a, int kick, cudaStream_t s)
{
    if (a.n_bodies == 0) return;
    if (kick && a.lone_bodies) return;   // finished by k_body_md
    const unsigned warps = (unsigned)((a.n_bodies + WARP_BODIES - 1) / WARP_BODIES);
    if (!kick) k_body_pos<<<(a.n_bodies + 127) / 128, 128, 0, s>>>(a);
    if (!kick || a.max_cent > 2) launch_chained(k_body_centres, warps, 32 * WARP_BODIES, 0, s, a);
    if (a.max_cent <= 2) {   // spheres, dumbbells: eight lanes per body
        const unsigned grid = (unsigned)((a.n_bodies + 15) / 16);
        if (a.precision == 1) {
            if (a.max_cent <= 1) launch_chained(k_body_force<float, 1>, grid, 128, 0, s, a, kick);
            else launch_chained(k_body_force<float, 2>, grid, 128, 0, s, a, kick);
        } else {
            if (a.max_cent <= 1) launch_chained(k_body_force<double, 1>, grid, 128, 0, s, a, kick);
            else launch_chained(k_body_force<double, 2>, grid, 128, 0, s, a, kick);
        }
    } else {                 // many centres: one warp per body
        launch_chained(k_nlist_build, warps, 32 * WARP_BODIES, 0, s, a);
        if (a.precision == 1) launch_chained(k_body_force_warp<float>, warps, 32 * WARP_BODIES, 0, s, a, kick);
        else launch_chained(k_body_force_warp<double>, warps, 32 * WARP_BODIES, 0, s, a, kick);
    }
}

// ---------------------------------------------------------------- sites
// Site geometry of the two forms.  P32: d = Qf bf in float (three products,
// two adds), r = fl32(R) + d; P64: d = Q b in double.  Both wrapped into [0, L).
template <typename Real> struct Pose {
    Real Q[9], R[3];
};
__device__ __forceinline__ void site_geom(const StepArgs &a, int64_t t, const Pose<float> &P, const DevReplica &r,
                                          float d[3], float x[3], int &bad)
{
    const float *b = a.tbf + 3 * t;
    for (int k = 0; k < 3; ++k) {
        const float t0 = __fmul_rn(P.Q[3 * k], b[0]);
        const float t1 = __fmul_rn(P.Q[3 * k + 1], b[1]);
        const float t2 = __fmul_rn(P.Q[3 * k + 2], b[2]);
        d[k] = __fadd_rn(__fadd_rn(t0, t1), t2);
        x[k] = wrapf(__fadd_rn(P.R[k], d[k]), (float)r.L[k], bad);
    }
}
__device__ __forceinline__ void site_geom(const StepArgs &a, int64_t t, const Pose<double> &P, const DevReplica &r,
                                          double d[3], double x[3], int &bad)
{
    mv(P.Q, a.tb + 3 * t, d);
    for (int k = 0; k < 3; ++k) x[k] = wrap_box(P.R[k] + d[k], (double)r.L[k], bad);
}
__device__ __forceinline__ const float *pose_ptr(const StepArgs &a, int b, float) { return a.pose32 + (int64_t)b * POSE_W; }
__device__ __forceinline__ const double *pose_ptr(const StepArgs &a, int b, double) { return a.pose64 + (int64_t)b * POSE_W; }

template <typename Real> __device__ __forceinline__ Real site_mass(const StepArgs &a, int64_t t);
template <> __device__ __forceinline__ float site_mass<float>(const StepArgs &a, int64_t) { return a.m_site_f; }
template <> __device__ __forceinline__ double site_mass<double>(const StepArgs &a, int64_t t) { return a.tm[t]; }
// sqrt(kT / m) of a site, formed once on the host (both operations round
// correctly there and here; per site they cost 23 FP64 instructions)
template <typename Real> __device__ __forceinline__ Real site_scale(const StepArgs &a, int64_t t);
template <> __device__ __forceinline__ float site_scale<float>(const StepArgs &a, int64_t) { return a.site_sc_f; }
template <> __device__ __forceinline__ double site_scale<double>(const StepArgs &a, int64_t t) { return a.tsc[t]; }
template <typename Real> __device__ __forceinline__ Real cos_alpha(const StepArgs &a);
template <> __device__ __forceinline__ float cos_alpha<float>(const StepArgs &a) { return a.cos_af; }
template <> __device__ __forceinline__ double cos_alpha<double>(const StepArgs &a) { return a.cos_a; }
template <typename Real> __device__ __forceinline__ Real sin_alpha(const StepArgs &a);
template <> __device__ __forceinline__ float sin_alpha<float>(const StepArgs &a) { return a.sin_af; }
template <> __device__ __forceinline__ double sin_alpha<double>(const StepArgs &a) { return a.sin_a; }

// The sites' sums in the form's precision have one order, whatever the CTA:
// SITE_THREADS running sums, the j-th over the sites j, j + SITE_THREADS, ... in
// turn, then a shuffle tree over each 32 of them, then the SITE_WARPS results.
// With K lanes for each running sum (a CTA of K x SITE_THREADS threads) a lane
// takes every K-th of its sites, and the terms of the K lanes are added in site
// order on all of them, so K changes the latency but no bit of the result.
// Lane layout: 32 / K sums per warp, lane = part * (32 / K) + sum.
template <int K> struct SiteLane {
    static constexpr int SUMS = 32 / K;
    int j, part;
    __device__ SiteLane()
    {
        const int lane = threadIdx.x & 31;
        part = lane / SUMS;
        j = (int)(threadIdx.x >> 5) * SUMS + lane % SUMS;
    }
    // the s-th site of this lane
    __device__ int site(int s) const { return j + SITE_THREADS * (K * s + part); }
    // acc += the parts' terms in site order (zero for a part past the last site)
    template <typename Real> __device__ void add(Real (&acc)[6], const Real (&t)[6]) const
    {
#pragma unroll
        for (int p = 0; p < K; ++p)
#pragma unroll
            for (int k = 0; k < 6; ++k)
                acc[k] += K == 1 ? t[k] : __shfl_sync(0xffffffffu, t[k], p * SUMS + (int)(threadIdx.x & 31) % SUMS);
    }
};

// the shuffle trees: out[w][k] = the sum of component k over the running sums
// 32 w .. 32 w + 31 (shared memory; a CTA barrier must follow before it is read)
template <typename Real, int K>
__device__ __forceinline__ void site_trees(const SiteLane<K> &sl, Real (&acc)[6], Real (*out)[6])
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if constexpr (K == 1) {
        for (int k = 0; k < 6; ++k)
            for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], o);
        if (lane == 0)
            for (int k = 0; k < 6; ++k) out[wid][k] = acc[k];
    } else {
        __shared__ Real sum[6][SITE_THREADS];
        if (sl.part == 0)
            for (int k = 0; k < 6; ++k) sum[k][sl.j] = acc[k];
        __syncthreads();
        for (int e = wid; e < 6 * SITE_WARPS; e += K * SITE_WARPS) {
            const int k = e / SITE_WARPS, w = e % SITE_WARPS;
            Real v = sum[k][32 * w + lane];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) out[w][k] = v;
        }
    }
}

// FP64 form: the sites' contributions to the double sum arrays
__device__ __forceinline__ void add_sums64(const StepArgs &a, int64_t c, double m, const double v[3],
                                           const double xi[3])
{
    double *S = reinterpret_cast<double *>(a.sums);
    const int64_t C = a.n_cells;
    atomicAdd(S + c, 1.0);
    atomicAdd(S + C + c, m);
    for (int k = 0; k < 3; ++k) atomicAdd(S + (2 + k) * C + c, m * v[k]);
    if (a.rule == 0) atomicAdd(S + 5 * C + c, m * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]));
    else for (int k = 0; k < 3; ++k) atomicAdd(S + (5 + k) * C + c, m * xi[k]);
}

template <typename Real> __device__ __forceinline__ void load_cell(const StepArgs &a, int64_t c, Real p[8]);
template <> __device__ __forceinline__ void load_cell<float>(const StepArgs &a, int64_t c, float p[8])
{
    const float4 *r = reinterpret_cast<const float4 *>(a.params) + 2 * c;
    float4 x = r[0], y = r[1];
    p[0] = x.x; p[1] = x.y; p[2] = x.z; p[3] = x.w; p[4] = y.x; p[5] = y.y; p[6] = y.z; p[7] = 0.f;
}
template <> __device__ __forceinline__ void load_cell<double>(const StepArgs &a, int64_t c, double p[8])
{
    const double2 *r = reinterpret_cast<const double2 *>(a.params) + 4 * c;
    for (int k = 0; k < 4; ++k) { double2 t = r[k]; p[2 * k] = t.x; p[2 * k + 1] = t.y; }
}

// PRE coupling: site poses, thermal draws, Eq. 7, binning of the sites.
// Arithmetic in the form's precision only (the pose record carries the FP64
// body quantities already reduced to it).
// FP32 site kernels are held to 64 registers (8 CTAs of 128 threads per SM)
// so that they fit beside the solvent pass they overlap with.
// The draws and cells of a thread's sites wait in registers (N of them) for the
// sums they go into; in shared memory they left room for one CTA beside the
// three of the staged solvent pass (N = 0: shapes of more sites, in shared
// memory).  K lanes per running sum shorten the pass when there are few bodies.
template <typename Real> struct SiteMinBlocks { static constexpr int n = sizeof(Real) == 4 ? 8 : 1; };
template <typename Real, int K> struct SiteBlocks {
    static constexpr int n = SiteMinBlocks<Real>::n >= K ? SiteMinBlocks<Real>::n / K : 1;
};

template <typename Real, int K, int N>
__global__ void __launch_bounds__(K * SITE_THREADS, SiteBlocks<Real, K>::n) k_sites_pre(StepArgs a)
{
    extern __shared__ unsigned char smem_raw[];
    Real *svt = reinterpret_cast<Real *>(smem_raw);          // N = 0: [n_sites][3] thermal draws
    __shared__ Real sPose[POSE_W], sdV[3], sdW[3];
    __shared__ Real scratch[SITE_WARPS][6];
    __shared__ int sS[3];
    const DevBody &B = a.bodies[blockIdx.x];
    const int shape = B.shape, rep = B.rep;
    const int64_t site_begin = B.site_begin;
    const DevShape &sh = a.shapes[shape];
    const DevReplica r = a.reps[rep];
    const int64_t step = current_step(a);
    const int n = sh.n_sites;
    const SiteLane<K> sl;
    const int passes = N > 0 ? N : (n + K * SITE_THREADS - 1) / (K * SITE_THREADS);
    constexpr int NR = N > 0 ? N : 1;
    constexpr bool KEEP = sizeof(Real) == 8 && N > 0;   // FP64: the offsets too (formed again in FP32)
    Real vt[NR][3], off[NR][3];
    int cells[NR];
    bool own[NR];
    int bad = 0;
    Real acc[6] = {0, 0, 0, 0, 0, 0};
    auto draw_site = [&](int s) {   // the s-th site of the lane: thermal draw
        const int j = sl.site(s);
        Real w[3] = {0, 0, 0};
        if (j < n && !a.naive) {
            normals3(draw(r, step, (uint32_t)(r.site_id_base + (site_begin + j - r.site_begin)), TAG_SITE, 0u), w);
            const Real sc = site_scale<Real>(a, sh.site_begin + j);
            for (int k = 0; k < 3; ++k) w[k] = sc * w[k];
        }
        for (int k = 0; k < 3; ++k) {
            if (N > 0) vt[N > 0 ? s : 0][k] = w[k];
            else if (j < n) svt[3 * j + k] = w[k];
        }
    };
    if constexpr (N > 0) {
#pragma unroll
        for (int s = 0; s < N; ++s) draw_site(s);
    } else {
        for (int s = 0; s < passes; ++s) draw_site(s);
    }
    if (threadIdx.x == 32) grid_shift(r, step, sS);
    chain_wait();
    // the force pass of this pose is done: its neighbour lists are fresh
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.nl_dirty = 0;
    if (threadIdx.x < POSE_W) sPose[threadIdx.x] = pose_ptr(a, blockIdx.x, Real(0))[threadIdx.x];
    __syncthreads();
    Pose<Real> P;
    for (int k = 0; k < 9; ++k) P.Q[k] = sPose[k];
    for (int k = 0; k < 3; ++k) P.R[k] = sPose[9 + k];
    auto sum_site = [&](int s) {    // cell, terms of the body's sums
        const int j = sl.site(s);
        Real t[6] = {0, 0, 0, 0, 0, 0};
        int c = 0;
        if (j < n) {
            const int64_t ts = sh.site_begin + j, g = site_begin + j;
            Real d[3], x[3];
            site_geom(a, ts, P, r, d, x, bad);
            c = cell_axis(x[0], sS[0], r.L[0]) +
                r.L[0] * (cell_axis(x[1], sS[1], r.L[1]) + r.L[1] * cell_axis(x[2], sS[2], r.L[2]));
            a.site_cell[g] = c;
            if (KEEP) {
                for (int k = 0; k < 3; ++k) off[N > 0 ? s : 0][k] = d[k];
                own[N > 0 ? s : 0] = site_owned(a, x[2]);
            }
            if (!a.naive) {
                const Real m = site_mass<Real>(a, ts);
                for (int k = 0; k < 3; ++k) t[k] = m * (N > 0 ? vt[N > 0 ? s : 0][k] : svt[3 * j + k]);
                t[3] = d[1] * t[2] - d[2] * t[1];
                t[4] = d[2] * t[0] - d[0] * t[2];
                t[5] = d[0] * t[1] - d[1] * t[0];
            }
        }
        cells[N > 0 ? s : 0] = c;
        sl.add(acc, t);
    };
    if constexpr (N > 0) {
#pragma unroll
        for (int s = 0; s < N; ++s) sum_site(s);
    } else {
        for (int s = 0; s < passes; ++s) sum_site(s);
    }
    site_trees<Real, K>(sl, acc, scratch);
    __syncthreads();
    if (threadIdx.x < 32) {   // component k on lane k
        const int k = threadIdx.x < 3 ? threadIdx.x : 0;
        Real sp = 0, sL = 0, Vt = 0, Wt = 0;
        for (int w = 0; w < SITE_WARPS; ++w) {
            sp += scratch[w][k];
            sL += scratch[w][3 + k];
        }
        if (!a.naive) {
            // V~ = sum m v~ / M, omega~ = Q Ihat^-1 Q^T L~
            Vt = sp / (Real)sh.M;
            const Real L0 = __shfl_sync(0xffffffffu, sL, 0), L1 = __shfl_sync(0xffffffffu, sL, 1);
            const Real L2 = __shfl_sync(0xffffffffu, sL, 2);
            const Real lb = (sPose[k] * L0 + sPose[3 + k] * L1) + sPose[6 + k] * L2;
            const Real wb = sh.Ihat[k] > 0.0 ? lb / (Real)sh.Ihat[k] : Real(0);
            const Real w0 = __shfl_sync(0xffffffffu, wb, 0), w1 = __shfl_sync(0xffffffffu, wb, 1);
            const Real w2 = __shfl_sync(0xffffffffu, wb, 2);
            Wt = (sPose[3 * k] * w0 + sPose[3 * k + 1] * w1) + sPose[3 * k + 2] * w2;
        }
        if (threadIdx.x < 3) {
            sdV[k] = sPose[12 + k] - Vt;
            sdW[k] = sPose[15 + k] - Wt;
        }
    }
    __syncthreads();
    const Real dV[3] = {sdV[0], sdV[1], sdV[2]}, dW[3] = {sdW[0], sdW[1], sdW[2]};
    Real *SV = reinterpret_cast<Real *>(a.site_v);
    const int64_t NS = a.n_sites;
    auto bin_site = [&](int s) {    // Eq. 7 velocity, cell sums
        const int j = sl.site(s);
        if (j >= n) return;
        const int64_t ts = sh.site_begin + j, g = site_begin + j;
        Real d[3], v[3], xi[3] = {0, 0, 0};
        bool mine;   // a slab bins only the sites in its z range
        if (KEEP) {
            for (int k = 0; k < 3; ++k) d[k] = off[N > 0 ? s : 0][k];
            mine = own[N > 0 ? s : 0];
        } else {
            Real x[3];
            site_geom(a, ts, P, r, d, x, bad);
            mine = site_owned(a, x[2]);
        }
        v[0] = dV[0] + (dW[1] * d[2] - dW[2] * d[1]);
        v[1] = dV[1] + (dW[2] * d[0] - dW[0] * d[2]);
        v[2] = dV[2] + (dW[0] * d[1] - dW[1] * d[0]);
        if (!a.naive)
            for (int k = 0; k < 3; ++k) v[k] += N > 0 ? vt[N > 0 ? s : 0][k] : svt[3 * j + k];
        for (int k = 0; k < 3; ++k) SV[k * NS + g] = v[k];
        const Real m = site_mass<Real>(a, ts);
        if (a.rule == 1) {
            normals3(draw(r, step, (uint32_t)(r.site_id_base + (g - r.site_begin)), TAG_AT, 0u), xi);
            const Real sc = site_scale<Real>(a, ts);
            for (int k = 0; k < 3; ++k) xi[k] *= sc;
            if (Real *XI = reinterpret_cast<Real *>(a.site_xi))   // kept for POST
                for (int k = 0; k < 3; ++k) XI[k * NS + g] = xi[k];
        }
        const int cell = r.cell_base + (N > 0 ? cells[N > 0 ? s : 0] : a.site_cell[g]);
        if (!mine) return;
        if constexpr (sizeof(Real) == 4) {
            long long w[MAX_WORDS32];
            unsigned long long *S = reinterpret_cast<unsigned long long *>(a.sums);
            if (a.rule == 0) {
                record_terms<0>(m, v[0], v[1], v[2], xi, true, w);
                for (int k = 0; k < Words32<0>::n; ++k) atomicAdd(S + k * a.n_cells + cell, (unsigned long long)w[k]);
            } else {
                record_terms<1>(m, v[0], v[1], v[2], xi, true, w);
                for (int k = 0; k < Words32<1>::n; ++k) atomicAdd(S + k * a.n_cells + cell, (unsigned long long)w[k]);
            }
        } else {
            add_sums64(a, cell, m, v, xi);
        }
    };
    if constexpr (N > 0) {
#pragma unroll
        for (int s = 0; s < N; ++s) bin_site(s);
    } else {
        for (int s = 0; s < passes; ++s) bin_site(s);
    }
    if (bad) atomicOr(a.d_err, ERR_POSITION);
}

// POST coupling: site collision and the per-warp partial sums of the
// momentum dP = sum m (v' - v) and angular momentum dL = sum d x m (v' - v)
// transferred to the body (Eqs. 3-4); k_body_impulse adds them in FP64.
// the collision rule for one site: v -> vn with the parameters p of its cell; KEPT: the
// MPCD-AT draws of the PRE pass are read, else drawn again (the FP64 form with
// both in one kernel took 158 registers instead of 116)
template <typename Real, bool KEPT>
__device__ __forceinline__ void site_rule(const StepArgs &a, const DevReplica &r, int64_t step, int64_t ts, int64_t g,
                                          const Real (&v)[3], const Real (&p)[8], Real (&vn)[3])
{
    vn[0] = v[0]; vn[1] = v[1]; vn[2] = v[2];
    if (p[3] >= Real(0)) {
        const Real ca = cos_alpha<Real>(a), sa = sin_alpha<Real>(a);
        if (a.rule == 0) {
            const Real w[3] = {v[0] - p[0], v[1] - p[1], v[2] - p[2]};
            const Real nd = p[4] * w[0] + p[5] * w[1] + p[6] * w[2];
            const Real cx = p[5] * w[2] - p[6] * w[1], cy = p[6] * w[0] - p[4] * w[2];
            const Real cz = p[4] * w[1] - p[5] * w[0];
            const Real tt = nd * (Real(1) - ca);
            vn[0] = p[0] + p[3] * (w[0] * ca + cx * sa + p[4] * tt);
            vn[1] = p[1] + p[3] * (w[1] * ca + cy * sa + p[5] * tt);
            vn[2] = p[2] + p[3] * (w[2] * ca + cz * sa + p[6] * tt);
        } else {
            Real xi[3];
            if constexpr (KEPT) {
                const Real *XI = reinterpret_cast<const Real *>(a.site_xi);
                for (int k = 0; k < 3; ++k) xi[k] = XI[k * a.n_sites + g];
            } else {
                normals3(draw(r, step, (uint32_t)(r.site_id_base + (g - r.site_begin)), TAG_AT, 0u), xi);
                const Real sc = site_scale<Real>(a, ts);
                for (int k = 0; k < 3; ++k) xi[k] *= sc;
            }
            for (int k = 0; k < 3; ++k) vn[k] = p[k] + xi[k] - p[4 + k];
        }
    }
}

// lattice offset of a stored site position inside its shifted cell (+a variants)
template <typename Real>
__device__ __forceinline__ void site_lattice_q(const Real (&x)[3], const int (&S)[3], int (&Q)[3])
{
    for (int k = 0; k < 3; ++k) Q[k] = ang_lattice_q(x[k], S[k]);
}

// POST coupling; ANG: with the +a correction of the site's cell applied to the
// rule's velocity before the momentum change is taken
template <typename Real, bool ANG, bool KEPT, int K>
__global__ void __launch_bounds__(K * SITE_THREADS, SiteBlocks<Real, K>::n) k_sites_post(StepArgs a)
{
    __shared__ Real sPose[POSE_W];
    __shared__ Real scratch[SITE_WARPS][6];
    __shared__ int sS[3];   // ANG: grid shift
    const DevBody &B = a.bodies[blockIdx.x];
    const int64_t site_begin = B.site_begin;
    const DevShape &sh = a.shapes[B.shape];
    const DevReplica r = a.reps[B.rep];
    const int64_t step = current_step(a);
    chain_next();
    if (ANG && threadIdx.x == 32) grid_shift(r, step, sS);
    if (threadIdx.x < POSE_W) sPose[threadIdx.x] = pose_ptr(a, blockIdx.x, Real(0))[threadIdx.x];
    __syncthreads();
    Pose<Real> P;
    for (int k = 0; k < 9; ++k) P.Q[k] = sPose[k];
    for (int k = 0; k < 3; ++k) P.R[k] = sPose[9 + k];
    const Real *SV = reinterpret_cast<const Real *>(a.site_v);
    const int64_t NS = a.n_sites;
    const int n = sh.n_sites;
    const SiteLane<K> sl;
    int bad = 0;
    Real acc[6] = {0, 0, 0, 0, 0, 0};
    // uniform trip count: the lanes of a running sum exchange their terms
    for (int s = 0; K * SITE_THREADS * s < n; ++s) {
        const int j = sl.site(s);
        Real dt6[6] = {0, 0, 0, 0, 0, 0};
        if (j < n) {
            const int64_t t = sh.site_begin + j, g = site_begin + j;
            const int64_t cell = (int64_t)r.cell_base + a.site_cell[g];
            const Real v[3] = {SV[g], SV[NS + g], SV[2 * NS + g]};
            Real d[3], x[3];
            site_geom(a, t, P, r, d, x, bad);
            Real vn[3];
            Real p[8];
            load_cell<Real>(a, cell, p);
            const Real m = site_mass<Real>(a, t);
            site_rule<Real, KEPT>(a, r, step, t, g, v, p, vn);
            if constexpr (ANG) {
                const Real xs[3] = {x[0], x[1], x[2]};
                int Q[3];
                site_lattice_q(xs, sS, Q);
                ang_correct(reinterpret_cast<const AngParams<Real> *>(a.ang_params)[cell], Q, vn);
            }
            if (site_owned(a, x[2])) {   // a slab transfers only its own sites
                const Real dp[3] = {m * (vn[0] - v[0]), m * (vn[1] - v[1]), m * (vn[2] - v[2])};
                dt6[0] = dp[0];
                dt6[1] = dp[1];
                dt6[2] = dp[2];
                dt6[3] = d[1] * dp[2] - d[2] * dp[1];
                dt6[4] = d[2] * dp[0] - d[0] * dp[2];
                dt6[5] = d[0] * dp[1] - d[1] * dp[0];
            }
        }
        sl.add(acc, dt6);
    }
    site_trees<Real, K>(sl, acc, scratch);
    __syncthreads();
    if (threadIdx.x < SITE_WARPS * 6)
        (reinterpret_cast<Real *>(a.partial) + (int64_t)blockIdx.x * SITE_WARPS * 6)[threadIdx.x] =
            scratch[threadIdx.x / 6][threadIdx.x % 6];
    if (bad) atomicOr(a.d_err, ERR_POSITION);
}

// impulse P += dP, L += dL accumulated in FP64 from the per-warp partials
template <typename Real>
__global__ void k_body_impulse(StepArgs a)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n_bodies) return;
    const Real *in = reinterpret_cast<const Real *>(a.partial) + (int64_t)i * SITE_WARPS * 6;
    double s[6] = {0, 0, 0, 0, 0, 0};
    for (int w = 0; w < SITE_WARPS; ++w)
        for (int k = 0; k < 6; ++k) s[k] += (double)in[w * 6 + k];
    DevBody *o = a.bodies + i;
    for (int k = 0; k < 3; ++k) {
        o->P[k] += s[k];
        o->Lm[k] += s[3 + k];
    }
}

constexpr int SITES_KEPT = 6 * SITE_THREADS;   // most sites of a shape whose draws stay in registers

// Two lanes per running sum up to eight bodies per SM, one beyond: with few
// bodies the passes are as long as one CTA takes (221 bodies of 642 sites: PRE
// 18.5 -> 14.7, POST 13.8 -> 9.9 us; 1120 bodies of up to 2000: a step 552 ->
// 542), with many the wider CTA finds less room beside the solvent pass (8952
// bodies: a step 1766 us with one lane, 1783 with two).
static int site_lanes(const StepArgs &a, int num_sms) { return a.n_bodies <= 8 * num_sms ? 2 : 1; }

// Dynamic shared memory that a kernel is allowed (allow_shared_memory).
template <typename... P>
static size_t shared_room(void (*kernel)(P...))
{
    cudaFuncAttributes at{};
    return cudaFuncGetAttributes(&at, kernel) == cudaSuccess ? (size_t)at.maxDynamicSharedSizeBytes : 0;
}
// All that a CTA can have beside the kernel's own static arrays: the same for every
// context, so that none lowers what another one needs.
template <typename... P>
static cudaError_t allow_shared_memory(void (*kernel)(P...))
{
    int dev = 0, most = 0;
    cudaFuncAttributes at{};
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, kernel);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)at.sharedSizeBytes);
}

template <typename Real, int K>
static void sites_pre(const StepArgs &a, int max_sites, bool chained, cudaStream_t s)
{
    constexpr int block = K * SITE_THREADS, FEW = 2 / K, MANY = 6 / K;   // 256 or 768 sites in registers
    static_assert(MANY * block == SITES_KEPT, "");
    const size_t bytes = (size_t)max_sites * 3 * sizeof(Real);
    if (max_sites <= FEW * block)
        launch(k_sites_pre<Real, K, FEW>, chained, a.n_bodies, block, 0, s, a);
    else if (max_sites <= SITES_KEPT)
        launch(k_sites_pre<Real, K, MANY>, chained, a.n_bodies, block, 0, s, a);
    else if (K == 1 || bytes <= shared_room(k_sites_pre<Real, K, 0>))
        launch(k_sites_pre<Real, K, 0>, chained, a.n_bodies, block, bytes, s, a);
    else   // the running sums of two lanes (3 or 6 KB) do not fit beside the draws
        sites_pre<Real, 1>(a, max_sites, chained, s);
}

cudaError_t configure_body_kernels(int max_sites, int precision)
{
    if (max_sites <= SITES_KEPT) return cudaSuccess;
    const size_t bytes = (size_t)max_sites * 3 * (precision == 1 ? sizeof(float) : sizeof(double));
    const auto configure = [&](auto *one, auto *two) {
        cudaError_t e = allow_shared_memory(one);
        if (e == cudaSuccess) e = allow_shared_memory(two);
        if (e != cudaSuccess) return e;
        return bytes <= shared_room(one) ? cudaSuccess : cudaErrorInvalidValue;
    };
    return precision == 1 ? configure(k_sites_pre<float, 1, 0>, k_sites_pre<float, 2, 0>)
                          : configure(k_sites_pre<double, 1, 0>, k_sites_pre<double, 2, 0>);
}

void launch_sites_pre(const StepArgs &a, int max_sites, int num_sms, bool chained, cudaStream_t s)
{
    if (a.n_bodies == 0) return;
    const bool two = site_lanes(a, num_sms) == 2;
    chained = chained && chain_pays(a);
    if (a.precision == 1) {
        if (two) sites_pre<float, 2>(a, max_sites, chained, s);
        else sites_pre<float, 1>(a, max_sites, chained, s);
    } else {
        if (two) sites_pre<double, 2>(a, max_sites, chained, s);
        else sites_pre<double, 1>(a, max_sites, chained, s);
    }
}

// the sites' draws of the rule are kept, or there are none
static bool draws_kept(const StepArgs &a) { return a.rule == 0 || a.site_xi; }

template <typename Real, bool ANG, bool KEPT>
static void sites_post(const StepArgs &a, bool two, cudaStream_t s)
{
    if (two) k_sites_post<Real, ANG, KEPT, 2><<<a.n_bodies, 2 * SITE_THREADS, 0, s>>>(a);
    else k_sites_post<Real, ANG, KEPT, 1><<<a.n_bodies, SITE_THREADS, 0, s>>>(a);
}

template <typename Real>
static void sites_post(const StepArgs &a, bool two, cudaStream_t s)
{
    const bool ang = a.ang_params != nullptr;
    if (draws_kept(a)) {
        if (ang) sites_post<Real, true, true>(a, two, s);
        else sites_post<Real, false, true>(a, two, s);
    } else {
        if (ang) sites_post<Real, true, false>(a, two, s);
        else sites_post<Real, false, false>(a, two, s);
    }
}

void launch_sites_post(const StepArgs &a, int num_sms, cudaStream_t s)
{
    if (a.n_bodies == 0) return;
    const bool two = site_lanes(a, num_sms) == 2;
    if (a.precision == 1) sites_post<float>(a, two, s);
    else sites_post<double>(a, two, s);
}

// +a variants: the sites' contributions to the angular words of their cells, one
// CTA per body: count, sum Q, sum Q_a Q_b, Q x (P - P*) and P - P* with P from
// the thermalised velocities of Eq. 7 and P* from the rule's (recomputed with
// the same arithmetic as the POST coupling).
__device__ __forceinline__ long long site_mom_term(float m, float v) { return q20(__fmul_rn(m, v)); }
__device__ __forceinline__ double site_mom_term(double m, double v) { return m * v; }

constexpr int ANG_SITE_CTAS = 2;   // CTAs per body (the order of the integer sums is free)

template <typename Real, bool KEPT>
__global__ void __launch_bounds__(SITE_THREADS, SiteMinBlocks<Real>::n) k_ang_sites(StepArgs a)
{
    typedef typename AngWord<Real>::type W;
    __shared__ Real sPose[POSE_W];
    __shared__ int sS[3];
    const DevBody &B = a.bodies[blockIdx.x / ANG_SITE_CTAS];
    const int part = blockIdx.x % ANG_SITE_CTAS;
    const int64_t site_begin = B.site_begin;
    const DevShape &sh = a.shapes[B.shape];
    const DevReplica r = a.reps[B.rep];
    const int64_t step = current_step(a);
    W *words = reinterpret_cast<W *>(a.ang_words);
    if (threadIdx.x < POSE_W) sPose[threadIdx.x] = pose_ptr(a, blockIdx.x / ANG_SITE_CTAS, Real(0))[threadIdx.x];
    if (threadIdx.x == 32) grid_shift(r, step, sS);
    __syncthreads();
    Pose<Real> P;
    for (int k = 0; k < 9; ++k) P.Q[k] = sPose[k];
    for (int k = 0; k < 3; ++k) P.R[k] = sPose[9 + k];
    const Real *SV = reinterpret_cast<const Real *>(a.site_v);
    const int64_t NS = a.n_sites;
    int bad = 0;
    for (int j = part * SITE_THREADS + threadIdx.x; j < sh.n_sites; j += ANG_SITE_CTAS * SITE_THREADS) {
        const int64_t t = sh.site_begin + j, g = site_begin + j;
        const int64_t cell = (int64_t)r.cell_base + a.site_cell[g];
        Real d[3], x[3];
        site_geom(a, t, P, r, d, x, bad);
        const Real v[3] = {SV[g], SV[NS + g], SV[2 * NS + g]};
        const Real m = site_mass<Real>(a, t);
        Real u[3], p[8];
        load_cell<Real>(a, cell, p);
        site_rule<Real, KEPT>(a, r, step, t, g, v, p, u);
        const Real xs[3] = {x[0], x[1], x[2]};
        int Qi[3];
        site_lattice_q(xs, sS, Qi);
        const W q[3] = {(W)Qi[0], (W)Qi[1], (W)Qi[2]};
        W D[3];
        for (int k = 0; k < 3; ++k) D[k] = (W)site_mom_term(m, v[k]) - (W)site_mom_term(m, u[k]);
        W *w = words + AW_SOLVENT * cell, *ws = words + AW_SOLVENT * a.n_cells + AW_SITES * cell;
        ang_red(w + AW_COUNT, (W)AW_SITE);
        ang_red(w + AW_L, q[1] * D[2] - q[2] * D[1]);
        ang_red(w + AW_L + 1, q[2] * D[0] - q[0] * D[2]);
        ang_red(w + AW_L + 2, q[0] * D[1] - q[1] * D[0]);
        for (int k = 0; k < 3; ++k) ang_red(w + AW_P + k, D[k]);
        for (int k = 0; k < 3; ++k) ang_red(ws + AW_SQB + k, q[k]);
        ang_red(ws + AW_QQB + 0, q[0] * q[0]);
        ang_red(ws + AW_QQB + 1, q[1] * q[1]);
        ang_red(ws + AW_QQB + 2, q[2] * q[2]);
        ang_red(ws + AW_QQB + 3, q[0] * q[1]);
        ang_red(ws + AW_QQB + 4, q[0] * q[2]);
        ang_red(ws + AW_QQB + 5, q[1] * q[2]);
    }
    if (bad) atomicOr(a.d_err, ERR_POSITION);
}

void launch_angular_sites(const StepArgs &a, cudaStream_t s)
{
    if (a.n_bodies == 0) return;
    const unsigned grid = (unsigned)a.n_bodies * ANG_SITE_CTAS;
    if (draws_kept(a)) {
        if (a.precision == 1) k_ang_sites<float, true><<<grid, SITE_THREADS, 0, s>>>(a);
        else k_ang_sites<double, true><<<grid, SITE_THREADS, 0, s>>>(a);
    } else {
        if (a.precision == 1) k_ang_sites<float, false><<<grid, SITE_THREADS, 0, s>>>(a);
        else k_ang_sites<double, false><<<grid, SITE_THREADS, 0, s>>>(a);
    }
}

void launch_body_impulse(const StepArgs &a, cudaStream_t s)
{
    if (a.n_bodies == 0) return;
    if (a.precision == 1) k_body_impulse<float><<<(a.n_bodies + 127) / 128, 128, 0, s>>>(a);
    else k_body_impulse<double><<<(a.n_bodies + 127) / 128, 128, 0, s>>>(a);
}

__global__ void k_advance_step(int64_t *step, int64_t n) { *step += n; }

void launch_advance_step(const StepArgs &a, int64_t n, cudaStream_t s)
{
    k_advance_step<<<1, 1, 0, s>>>(const_cast<int64_t *>(a.d_step), n);
}

// FP64 body diagnostics: sum P, sum |P|^2/2M, sum L_b.Ihat^-1.L_b/2 (L_b = Q^T L)
__global__ void k_body_diag(StepArgs a, double *acc)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n_bodies) return;
    const DevBody b = a.bodies[i];
    const DevShape sh = a.shapes[b.shape];
    double Lb[3], Q[9];
    rotmat(b.q, Q);
    mtv(Q, b.Lm, Lb);
    double er = 0.0;
    for (int k = 0; k < 3; ++k) er += sh.Ihat[k] > 0.0 ? 0.5 * Lb[k] * Lb[k] / sh.Ihat[k] : 0.0;
    double et = 0.5 * (b.P[0] * b.P[0] + b.P[1] * b.P[1] + b.P[2] * b.P[2]) / sh.M;
    atomicAdd(acc + 4, b.P[0]);
    atomicAdd(acc + 5, b.P[1]);
    atomicAdd(acc + 6, b.P[2]);
    atomicAdd(acc + 7, et);
    atomicAdd(acc + 8, er);
}

void launch_body_diag(const StepArgs &a, double *acc, cudaStream_t s)
{
    if (a.n_bodies == 0) return;
    k_body_diag<<<(a.n_bodies + 127) / 128, 128, 0, s>>>(a, acc);
}


// ------------------------------------------- velocity autocorrelation
// Sec. III.A: C_T(t) = <V(0).V(t)> and C_R(t) = <omega(0).omega(t)>, every
// sample a time origin.  After every `every`-th completed step each body adds
// V(t).V(t - k) and omega(t).omega(t - k) for the lags k it has samples for;
// the last n_lags samples stay in a per-body ring.  omega is the space-frame
// angular velocity Q Ihat^-1 Q^T L.  FP64, one lag per lane and a warp for 32
// lags of a body: the lags of a body are neighbours in memory, and each lane
// forms V and omega again, which costs a warp no more than one lane (512 bodies,
// 50 lags: 138 us per sample with one thread per body, 13 now).
__global__ void __launch_bounds__(128) k_vacf_sample(StepArgs a, VacfArgs g)
{
    const int64_t done = current_step(a) + 1 - g.start;   // steps completed since the start
    if (done <= 0 || done % g.every != 0) return;
    const int64_t smp = done / g.every - 1;          // this sample's index
    const int nk = (int)(smp + 1 < g.n_lags ? smp + 1 : g.n_lags);
    const int chunks = (g.n_lags + 31) / 32;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t i = w / chunks;
    const int k0 = (int)(w - i * chunks) * 32, k = k0 + (int)(threadIdx.x & 31);
    if (i >= a.n_bodies || k0 >= nk) return;
    if (i == 0 && k < nk) g.count[k] += 1;
    const DevBody &b = a.bodies[i];
    const DevShape &sh = a.shapes[b.shape];
    double Q[9], Lb[3], wb[3], V[3], W[3];
    rotmat(b.q, Q);
    mtv(Q, b.Lm, Lb);
    for (int c = 0; c < 3; ++c) {
        V[c] = div_by(b.P[c], sh.M, sh.rM);
        wb[c] = sh.Ihat[c] > 0.0 ? div_by(Lb[c], sh.Ihat[c], sh.rI[c]) : 0.0;
    }
    mv(Q, wb, W);
    const int64_t base = i * g.n_lags;
    if (k < nk) {
        // lag k: the sample k before this one (lag 0: this one, not in the ring yet)
        const int64_t r = 3 * (base + (smp - k) % g.n_lags);
        double pv[3], pw[3];
        for (int c = 0; c < 3; ++c) {
            pv[c] = k == 0 ? V[c] : g.ring_v[r + c];
            pw[c] = k == 0 ? W[c] : g.ring_w[r + c];
        }
        g.ct[base + k] += V[0] * pv[0] + V[1] * pv[1] + V[2] * pv[2];
        g.cr[base + k] += W[0] * pw[0] + W[1] * pw[1] + W[2] * pw[2];
    }
    if (k == 0) {   // the ring slot of this sample is the one of lag n_lags: nobody reads it
        const int64_t r = 3 * (base + smp % g.n_lags);
        for (int c = 0; c < 3; ++c) {
            g.ring_v[r + c] = V[c];
            g.ring_w[r + c] = W[c];
        }
    }
}

void launch_vacf_sample(const StepArgs &a, const VacfArgs &g, cudaStream_t s)
{
    if (a.n_bodies == 0) return;
    const int64_t warps = (int64_t)a.n_bodies * ((g.n_lags + 31) / 32);
    k_vacf_sample<<<(unsigned)((warps + 3) / 4), 128, 0, s>>>(a, g);
}

}  // namespace mpcd
