// Angular-momentum-conserving variants of the collision rules (SRD+a and
// MPCD-AT+a: the modification of the rules that Sec. II.A of arXiv 2604.14307
// cites from Noguchi and Gompper): the solvent's passes and the per-cell solve;
// the colloid sites' share lives beside the other site kernels.
//
// After the plain rule has produced v*, every cell with two or more members
// gets the rigid rotation v' = v* + w x r_c that gives back its angular
// momentum about its centre of mass:
//     Pi w = sum_i m r_c,i x (v_i - v*_i),
// Pi the inertia tensor of the members about that centre, and w the least-norm
// solution when the members are collinear (two members in particular).  The
// rule conserves the momentum, so the correction keeps it as well.  r_c is
// measured on the 2^-20 lattice of the binning rule: Q = (floor(x 2^20) - S)
// mod 2^20 is the member's offset inside its shifted cell in units of 2^-20,
// an integer, which makes the geometric sums exact.
//
// Passes of a step (all keyed on the same step):
//   k_ang_collide     solvent: the rule, and the cell words: count, sum Q,
//                     sum Q_a Q_b, sum Q x (P - P*), sum (P - P*) (the sites'
//                     words in kernels_bodies.cu, beside it)
//   k_ang_params      per cell: centre of mass, Pi and the angular-momentum
//                     change in FP64, w by the adjugate of Pi (least-norm form
//                     for collinear members); clears the words
//   k_ang_stream      solvent: v = v* + w' x (M Q - sum mu Q), w' = w / (M 2^20),
//                     then streams and bins for the next step (k_ang_apply: the
//                     correction alone); the site POST coupling applies the
//                     same to the sites before it transfers their momentum
//                     change to the body
// so that the particles are read and written twice in a step.  (Binning, sums
// before the rule, rule, sums after it, correction and streaming were six
// passes: 1.08 M particles with 191 bodies 300 us per step.)
// Word layout and record: AW_* and AngParams in mpcd_internal.cuh.  The
// geometric sums are kept per species (solvent, sites) and exact; masses enter
// in the per-cell solve (P32: mu = round(m 2^24), the quantised masses of the
// cell words).  The offset from the centre is formed as the exact integer
// M Q - sum mu Q: for nearly collinear members w is large along their line
// while the offsets across it are small, and an offset rounded in the working
// precision would carry an error of order eps |w| into the velocity.
// P32: every word an int64 sum (exact and independent of the order of the
// atomics; wrap-around of partial sums cancels as long as the final sum lies
// within +-2^63).  P64: the Q sums are exact integers in double, the momentum
// sums FP64 atomics.
#include <algorithm>

#include "solvent_device.cuh"

namespace mpcd {

namespace {

// momentum term P of one particle: the P32 fixed-point value or the FP64 product
__device__ __forceinline__ long long mom_term(float m, float v) { return q20(__fmul_rn(m, v)); }
__device__ __forceinline__ double mom_term(double m, double v) { return m * v; }

__device__ __forceinline__ void ld4v(const float *p, float (&o)[4])
{
    const float4 t = *reinterpret_cast<const float4 *>(p);
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void ld4v(const double *p, double (&o)[4])
{
    const double2 t0 = reinterpret_cast<const double2 *>(p)[0], t1 = reinterpret_cast<const double2 *>(p)[1];
    o[0] = t0.x; o[1] = t0.y; o[2] = t1.x; o[3] = t1.y;
}
__device__ __forceinline__ void st4v(float *p, const float (&o)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ void st4v(double *p, const double (&o)[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(o[0], o[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(o[2], o[3]);
}

// cell and lattice offset Q of each of a thread's 4 particles
template <typename Real>
__device__ __forceinline__ void cells4(const Real (&x)[4], const Real (&y)[4], const Real (&z)[4], int4 S,
                                       const DevReplica &r, int (&c)[4], int (&Q)[4][3])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int X[3] = {lattice_X(x[j]), lattice_X(y[j]), lattice_X(z[j])};
        const int Sk[3] = {S.x, S.y, S.z};
        int cc[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            cc[k] = axis_cell(X[k], Sk[k], r.L[k]);
            Q[j][k] = (X[k] - Sk[k]) & 0xFFFFF;
        }
        c[j] = r.cell_base + cc[0] + r.L[0] * (cc[1] + r.L[1] * cc[2]);   // below 2^31 cells
    }
}

// Work of the solvent passes: a warp takes ANG_UNIT particles of a tile, so that
// a box of few tiles still fills the chip, and ANG_CTAS CTAs of 256 threads share
// an SM (80 registers a thread instead of 104 to 144: both passes wait for gathers
// and reductions, and MPCD-AT+a had one CTA an SM in k_ang_apply).  60^3 cells, 1.08 M
// particles: SRD+a 186 -> 178 us a step (k_ang_collide 58 -> 51), MPCD-AT+a 235
// -> 207; 110^3, 6.7 M: 1098 -> 1033 and 1467 -> 1237 (k_ang_apply 694 -> 458).
// With 64 registers 180 and 208, 1008 and 1222.  The FP64 form is bound by its
// FP64 instructions: 128 registers (40^3 cells: 234 and 319 us; 80: 253 and 353).
constexpr int ANG_UNIT = 256;
template <typename Real> constexpr int ANG_CTAS = sizeof(Real) == 4 ? 3 : 2;

// The rule and the cell words.  Each lane takes 4 consecutive
// particles (128-bit loads; tiles start on multiples of 8 slots, and the slots
// past a replica's last particle are allocated padding) and merges runs of equal
// cells in registers.  The 16 words of a cell are one 128-byte line, and the
// pass is bound by the sectors its L2 reductions touch: the runs that end at a
// slot go through shared memory, and sixteen lanes add the words of one (4 sectors
// a run; word arrays n_cells long touched about 10).
constexpr int ANG_ROW = AW_SOLVENT + 1;   // a lane's row of words, padded against bank conflicts

template <typename Real, int RULE>
__global__ void __launch_bounds__(256, ANG_CTAS<Real>) k_ang_collide(StepArgs a, int subs)
{
    typedef typename AngWord<Real>::type W;
    __shared__ W rows[8][32 * ANG_ROW];
    W *words = reinterpret_cast<W *>(a.ang_words);
    const int64_t step = current_step(a);
    const Real m = Consts<Real>::m(a), ca = Consts<Real>::ca(a), sa = Consts<Real>::sa(a);
    const Real sc = sqrt(Consts<Real>::kT(a) / m);
    const Real *X = reinterpret_cast<const Real *>(a.x), *Y = reinterpret_cast<const Real *>(a.y);
    const Real *Z = reinterpret_cast<const Real *>(a.z);
    Real *VX = reinterpret_cast<Real *>(a.vx), *VY = reinterpret_cast<Real *>(a.vy);
    Real *VZ = reinterpret_cast<Real *>(a.vz);
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    W *row = rows[threadIdx.x >> 5];
    int4 S = make_int4(0, 0, 0, 0);
    int last_rep = -1;
    for (int u = blockIdx.x * warps + (threadIdx.x >> 5); u < a.n_tiles * subs; u += gridDim.x * warps) {
        Tile tl = a.tiles[u / subs];
        tl.begin += (int64_t)(u % subs) * ANG_UNIT;
        tl.end = min(tl.end, tl.begin + ANG_UNIT);
        const DevReplica r = a.reps[tl.rep];
        if (tl.rep != last_rep) {
            int32_t s3[3];
            grid_shift(r, step, s3);
            S = make_int4(s3[0], s3[1], s3[2], 0);
            last_rep = tl.rep;
        }
        for (int64_t i0 = tl.begin; i0 < tl.end; i0 += 128) {   // uniform: the lanes add each other's runs
            const int64_t i = i0 + 4 * lane;
            const int nv = (int)max((int64_t)0, min((int64_t)4, tl.end - i));
            Real x[4] = {}, y[4] = {}, z[4] = {}, vx[4] = {}, vy[4] = {}, vz[4] = {};
            uint32_t tg[4] = {0, 0, 0, 0};
            if (nv > 0) {
                ld4v(X + i, x); ld4v(Y + i, y); ld4v(Z + i, z);
                ld4v(VX + i, vx); ld4v(VY + i, vy); ld4v(VZ + i, vz);
                if (RULE == 1) {
                    const uint4 t4 = *reinterpret_cast<const uint4 *>(a.tag + i);
                    tg[0] = t4.x; tg[1] = t4.y; tg[2] = t4.z; tg[3] = t4.w;
                }
            }
            int c[4];
            int Q[4][3];
            cells4(x, y, z, S, r, c, Q);
            Real nn[4][3];
            if (RULE == 1) at_normals4(a, r, step, tg, nv, i, nn);
            CellParams<Real> p[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) p[j] = get_params<Real>(a.params, j < nv ? c[j] : r.cell_base);
            W D[4][3];   // P - P*
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const W P0 = mom_term(m, vx[j]), P1 = mom_term(m, vy[j]), P2 = mom_term(m, vz[j]);
                const bool on = j < nv && p[j].kappa >= Real(0);
                Real rx = vx[j], ry = vy[j], rz = vz[j];
                if (RULE == 0) {
                    srd_rotate<Real>(p[j], ca, sa, rx, ry, rz);
                } else {
                    rx = p[j].ux + sc * nn[j][0] - p[j].ax;
                    ry = p[j].uy + sc * nn[j][1] - p[j].ay;
                    rz = p[j].uz + sc * nn[j][2] - p[j].az;
                }
                vx[j] = on ? rx : vx[j];
                vy[j] = on ? ry : vy[j];
                vz[j] = on ? rz : vz[j];
                D[j][0] = P0 - mom_term(m, vx[j]);
                D[j][1] = P1 - mom_term(m, vy[j]);
                D[j][2] = P2 - mom_term(m, vz[j]);
            }
            if (nv > 0) { st4v(VX + i, vx); st4v(VY + i, vy); st4v(VZ + i, vz); }
            W acc[AW_SOLVENT];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const W q0 = (W)Q[j][0], q1 = (W)Q[j][1], q2 = (W)Q[j][2];
                const W e[AW_SOLVENT] = {(W)1, q0, q1, q2, q0 * q0, q1 * q1, q2 * q2, q0 * q1, q0 * q2, q1 * q2,
                                         q1 * D[j][2] - q2 * D[j][1], q2 * D[j][0] - q0 * D[j][2],
                                         q0 * D[j][1] - q1 * D[j][0], D[j][0], D[j][1], D[j][2]};
                const bool more = j > 0 && j < nv && c[j] == c[j > 0 ? j - 1 : 0];
#pragma unroll
                for (int k = 0; k < AW_SOLVENT; ++k) acc[k] = more ? acc[k] + e[k] : e[k];
                const bool end = j < nv && (j + 1 >= nv || c[j < 3 ? j + 1 : 3] != c[j]);
                unsigned left = __ballot_sync(0xffffffffu, end);
                if (!left) continue;
                __syncwarp();
                if (end)
#pragma unroll
                    for (int k = 0; k < AW_SOLVENT; ++k) row[lane * ANG_ROW + k] = acc[k];
                __syncwarp();
                while (left) {   // two runs at a time, one per half warp
                    const int r0 = __ffs(left) - 1;
                    left &= left - 1;
                    const int r1 = left ? __ffs(left) - 1 : -1;
                    left &= left - 1;
                    const int src = lane < 16 ? r0 : r1;
                    const int cell = __shfl_sync(0xffffffffu, c[j], max(src, 0));
                    if (src >= 0)
                        ang_red(words + (int64_t)AW_SOLVENT * cell + (lane & 15), row[src * ANG_ROW + (lane & 15)]);
                }
            }
        }
    }
}

__device__ __forceinline__ double word_double(long long v) { return i64_double(v); }
__device__ __forceinline__ double word_double(double v) { return v; }

// record of one cell from its words.  mu_s, mu_b: the solvent and site mass
// in the units of the form (P32: round(m 2^24), P64: m); unit: the P terms' (P32:
// 2^-20, P64: 1) over the mass's (P32: 2^-24, P64: 1).
// FP64 instructions, 64 cycles each, bound the solve: the sites' words enter
// only where a cell has sites, the two forms of the solution share one
// division, and conversions, comparisons and roundings to float go to the
// integer pipe with the same results (216,000 cells: 65.5 -> 57.8 us; with the
// small CTAs below 55).
template <typename Real, typename W, typename MU>
__device__ void cell_record(const W (&wd)[AW_SOLVENT], const W *wb, MU mu_s, MU mu_b, double unit,
                            AngParams<Real> &o)
{
    const long long cnt = (long long)wd[AW_COUNT];
    const int n_s = (int)(cnt & (AW_SITE - 1)), n_b = (int)(cnt / AW_SITE);
    const bool sites = n_b > 0;
    const double ms = word_double(mu_s), mb = sites ? word_double(mu_b) : 0.0;
    o.M = (MU)n_s * mu_s;
    if (sites) o.M += (MU)n_b * mu_b;
    double sw[3];
    for (int k = 0; k < 3; ++k) {
        // P32: exact in int64 (mu Q sums below M 2^20)
        MU v = mu_s * (MU)wd[AW_SQ + k];
        if (sites) v += mu_b * (MU)wb[AW_SQB + k];
        o.sw[k] = v;
        sw[k] = word_double(v);
        o.w[k] = (Real)0;
    }
    const double M = word_double(o.M);
    o.pad = (Real)0;
    if (n_s + n_b < 2) return;
    const double iM = 1.0 / M;
    const double Qc[3] = {sw[0] * iM, sw[1] * iM, sw[2] * iM};
    // mass-weighted lattice covariance about the centre of mass
    double Cm[3][3];
    const int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        double v = ms * word_double(wd[AW_QQ + q]);
        if (sites) v = ms * word_double(wd[AW_QQ + q]) + mb * word_double(wb[AW_QQB + q]);
        v = v - sw[ia[q]] * Qc[ib[q]];
        Cm[ia[q]][ib[q]] = Cm[ib[q]][ia[q]] = v;
    }
    const double tr = Cm[0][0] + Cm[1][1] + Cm[2][2];
    // every member on one lattice point: tr is not above 0
    if ((unsigned long long)__double_as_longlong(tr) - 1 >= 0x7FF0000000000000ull) return;
    // angular-momentum change about the centre (units 2^-20 pscale)
    const double dP[3] = {word_double(wd[AW_P]), word_double(wd[AW_P + 1]), word_double(wd[AW_P + 2])};
    const double dL[3] = {word_double(wd[AW_L]) - (Qc[1] * dP[2] - Qc[2] * dP[1]),
                          word_double(wd[AW_L + 1]) - (Qc[2] * dP[0] - Qc[0] * dP[2]),
                          word_double(wd[AW_L + 2]) - (Qc[0] * dP[1] - Qc[1] * dP[0])};
    // G = tr(C) I - C = Pi / (mscale 2^-40); solve G x = dL by its adjugate
    const double a00 = tr - Cm[0][0], a11 = tr - Cm[1][1], a22 = tr - Cm[2][2];
    const double a01 = -Cm[0][1], a02 = -Cm[0][2], a12 = -Cm[1][2];
    const double c00 = a11 * a22 - a12 * a12, c01 = a02 * a12 - a01 * a22, c02 = a01 * a12 - a02 * a11;
    const double c11 = a00 * a22 - a02 * a02, c12 = a01 * a02 - a00 * a12, c22 = a00 * a11 - a01 * a01;
    const double det = a00 * c00 + a01 * c01 + a02 * c02;
    // collinear members: C = tr(C) d d^T, G = tr(C) (I - d d^T); least-norm x
    // = (dL - d (d.dL)) / tr(C) with d d^T = C / tr(C)
    // (the right side is positive: the bits order as the values do)
    const bool full = __double_as_longlong(det) > __double_as_longlong(1e-12 * tr * tr * tr);
    const double inv = 1.0 / (full ? det : tr);
    double x[3];
    if (full) {
        x[0] = (c00 * dL[0] + c01 * dL[1] + c02 * dL[2]) * inv;
        x[1] = (c01 * dL[0] + c11 * dL[1] + c12 * dL[2]) * inv;
        x[2] = (c02 * dL[0] + c12 * dL[1] + c22 * dL[2]) * inv;
    } else {
        for (int i = 0; i < 3; ++i) {
            const double CdL = Cm[i][0] * dL[0] + Cm[i][1] * dL[1] + Cm[i][2] * dL[2];
            x[i] = (dL[i] - CdL * inv) * inv;
        }
    }
    // Pi w = dL_phys with Pi = mscale 2^-40 G and dL_phys = 2^-20 pscale dL; the
    // record keeps w' = w / (M 2^20); unit = pscale / mscale, a power of two
    const double s = unit * iM;
    for (int k = 0; k < 3; ++k) {
        if constexpr (sizeof(Real) == 4) o.w[k] = double_float(x[k] * s);
        else o.w[k] = x[k] * s;
    }
}

// sixteen bytes of a cell's words at a time: the line of a cell is a thread's own
template <typename W, int N>
__device__ __forceinline__ void take_words(W *p, W (&o)[N])
{
    longlong2 *q = reinterpret_cast<longlong2 *>(p);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
        const longlong2 v = q[k];
        reinterpret_cast<longlong2 *>(o)[k] = v;
        q[k] = make_longlong2(0, 0);   // also 0.0 in the FP64 form
    }
}

// Small CTAs: every SM's FP64 pipe is full, so the cells are spread evenly (64
// threads against 256: 24^3 cells 16.9 -> 12.9 us, 60^3 57.8 -> 55, 110^3 276 -> 262).
constexpr int ANG_CELLS = 64;
template <typename Real>
__global__ void __launch_bounds__(ANG_CELLS) k_ang_params(StepArgs a)
{
    typedef typename AngWord<Real>::type W;
    W *w = reinterpret_cast<W *>(a.ang_words);
    AngParams<Real> *params = reinterpret_cast<AngParams<Real> *>(const_cast<void *>(a.ang_params));
    const int64_t C = a.n_cells;
    W *wsites = w + (int64_t)AW_SOLVENT * C;
    const bool p32 = sizeof(Real) == 4;
    typedef decltype(AngParams<Real>::M) MU;
    const MU mu_s = p32 ? (MU)a.qm_solvent : (MU)a.m_solvent, mu_b = p32 ? (MU)a.qm_site : (MU)a.m_site;
    const double unit = p32 ? 16.0 : 1.0;   // P terms 2^-20 or 1 over mu 2^-24 or 1
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < C; c += (int64_t)gridDim.x * blockDim.x) {
        alignas(16) W wd[AW_SOLVENT];
        W wb[AW_SITES];
        take_words(w + AW_SOLVENT * c, wd);
        if ((long long)wd[AW_COUNT] >= AW_SITE) {   // sites have added their words
#pragma unroll
            for (int k = 0; k < AW_SITES; ++k) {
                wb[k] = wsites[AW_SITES * c + k];
                wsites[AW_SITES * c + k] = (W)0;
            }
        }
        AngParams<Real> o;
        cell_record<Real>(wd, wb, mu_s, mu_b, unit, o);
        params[c] = o;
    }
}

// The correction; STREAM: then the drift and the binning for the next collision
// (the arithmetic of the plain passes, in the layout of k_ang_collide).
template <typename Real, int RULE, bool STREAM>
__global__ void __launch_bounds__(256, ANG_CTAS<Real>) k_ang_apply(StepArgs a, int subs)
{
    const AngParams<Real> *params = reinterpret_cast<const AngParams<Real> *>(a.ang_params);
    typedef typename SumWord<Real>::type SW;
    SW *sums = reinterpret_cast<SW *>(a.sums);
    const int64_t step = current_step(a);
    const Real m = Consts<Real>::m(a), dt = Consts<Real>::dt(a);
    const Real sc = sqrt(Consts<Real>::kT(a) / m);
    Real *X = reinterpret_cast<Real *>(a.x), *Y = reinterpret_cast<Real *>(a.y), *Z = reinterpret_cast<Real *>(a.z);
    Real *VX = reinterpret_cast<Real *>(a.vx), *VY = reinterpret_cast<Real *>(a.vy);
    Real *VZ = reinterpret_cast<Real *>(a.vz);
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    int4 S = make_int4(0, 0, 0, 0);
    typename ShiftT<Real>::type sF[3] = {};
    int last_rep = -1, bad = 0;
    for (int u = blockIdx.x * warps + (threadIdx.x >> 5); u < a.n_tiles * subs; u += gridDim.x * warps) {
        Tile tl = a.tiles[u / subs];
        tl.begin += (int64_t)(u % subs) * ANG_UNIT;
        tl.end = min(tl.end, tl.begin + ANG_UNIT);
        const DevReplica r = a.reps[tl.rep];
        if (tl.rep != last_rep) {
            int32_t s3[3];
            grid_shift(r, step, s3);
            S = make_int4(s3[0], s3[1], s3[2], 0);
            if (STREAM) {
                grid_shift(r, step + 1, s3);
                for (int k = 0; k < 3; ++k) sF[k] = shift_as(s3[k], typename ShiftT<Real>::type());
            }
            last_rep = tl.rep;
        }
        const Real L[3] = {(Real)r.L[0], (Real)r.L[1], (Real)r.L[2]};
        for (int64_t i = tl.begin + 4 * lane; i < tl.end; i += 128) {
            const int nv = (int)min((int64_t)4, tl.end - i);
            Real x[4], y[4], z[4], vx[4], vy[4], vz[4];
            ld4v(X + i, x); ld4v(Y + i, y); ld4v(Z + i, z);
            ld4v(VX + i, vx); ld4v(VY + i, vy); ld4v(VZ + i, vz);
            uint32_t tg[4] = {0, 0, 0, 0};
            if (STREAM && RULE == 1) {
                const uint4 t4 = *reinterpret_cast<const uint4 *>(a.tag + i);
                tg[0] = t4.x; tg[1] = t4.y; tg[2] = t4.z; tg[3] = t4.w;
            }
            int c[4];
            int Q[4][3];
            cells4(x, y, z, S, r, c, Q);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j >= nv) break;
                Real v[3] = {vx[j], vy[j], vz[j]};
                ang_correct(params[c[j]], Q[j], v);
                vx[j] = v[0]; vy[j] = v[1]; vz[j] = v[2];
                if (STREAM) {
                    if (a.accel) {
                        vx[j] = kick(vx[j], Consts<Real>::ah(a, 0));
                        vy[j] = kick(vy[j], Consts<Real>::ah(a, 1));
                        vz[j] = kick(vz[j], Consts<Real>::ah(a, 2));
                    }
                    x[j] = drift(x[j], vx[j], dt, L[0], bad);
                    y[j] = drift(y[j], vy[j], dt, L[1], bad);
                    z[j] = drift(z[j], vz[j], dt, L[2], bad);
                    if (a.accel) {
                        vx[j] = kick(vx[j], Consts<Real>::ah(a, 0));
                        vy[j] = kick(vy[j], Consts<Real>::ah(a, 1));
                        vz[j] = kick(vz[j], Consts<Real>::ah(a, 2));
                    }
                }
            }
            if (STREAM) {
                bin4<Real, RULE, true>(a, x, y, z, vx, vy, vz, tg, nv, sF, r.L[0], r.L[1], r.L[2], r.cell_base, r, step,
                                       m, sc, sums, a.n_cells, i);
                st4v(X + i, x); st4v(Y + i, y); st4v(Z + i, z);
            }
            st4v(VX + i, vx); st4v(VY + i, vy); st4v(VZ + i, vz);
        }
    }
    if (bad) atomicOr(a.d_err, ERR_POSITION);
}

}  // namespace

size_t angular_param_bytes(int precision)
{
    static_assert(sizeof(AngParams<float>) == 48 && sizeof(AngParams<double>) == 64, "record sizes");
    return precision == 1 ? sizeof(AngParams<float>) : sizeof(AngParams<double>);
}

template <typename Real, int RULE>
static void angular_phase(const StepArgs &a, int phase, int tile, int num_sms, cudaStream_t s)
{
    const int grid_p = (int)std::max<int64_t>(1, std::min<int64_t>((a.n_cells + ANG_CELLS - 1) / ANG_CELLS, (int64_t)num_sms * 64));
    const int subs = (tile + ANG_UNIT - 1) / ANG_UNIT;
    const int grid_t = std::max(1, std::min((a.n_tiles * subs + 7) / 8, num_sms * 8));   // 8 warps, one unit each
    if (phase != ANG_PARAMS && a.n_tiles == 0) return;
    switch (phase) {
    case ANG_COLLIDE: k_ang_collide<Real, RULE><<<grid_t, 256, 0, s>>>(a, subs); break;
    case ANG_PARAMS: k_ang_params<Real><<<grid_p, ANG_CELLS, 0, s>>>(a); break;
    case ANG_APPLY: k_ang_apply<Real, 0, false><<<grid_t, 256, 0, s>>>(a, subs); break;
    case ANG_STREAM: k_ang_apply<Real, RULE, true><<<grid_t, 256, 0, s>>>(a, subs); break;
    default: break;
    }
}

void launch_angular(const StepArgs &a, int phase, int tile, int num_sms, cudaStream_t s)
{
    if (a.n_cells == 0) return;
    if (a.precision == 1) {
        if (a.rule == 0) angular_phase<float, 0>(a, phase, tile, num_sms, s);
        else angular_phase<float, 1>(a, phase, tile, num_sms, s);
    } else {
        if (a.rule == 0) angular_phase<double, 0>(a, phase, tile, num_sms, s);
        else angular_phase<double, 1>(a, phase, tile, num_sms, s);
    }
}

}  // namespace mpcd
