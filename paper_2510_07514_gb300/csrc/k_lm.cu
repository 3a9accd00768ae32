// k_lm.cu -- PJ-IK (Sec. V-B, Alg. 4): persistent, warp-cooperative.
//
// Per iteration and candidate: one kinematics pass with frames gives the
// 6 x n geometric Jacobian (Eq. jacobian) and the residual; W normalises the
// Jacobian's rows (orientation rows also scaled by eps_pos / eps_ori).  The
// damped normal equations of Eq. normal-eqs, ((WJ)^T (WJ) + lambda D) d =
// (WJ)^T W r with D = diag((WJ)^T (WJ)), are solved in their 6 x 6
// push-through form
//     d = S Ah^T (Ah Ah^T + lambda I)^-1 W r,   Ah = WJ S,  S = D^(-1/2),
// an exact identity for lambda > 0, so one 6 x 6 Cholesky factorisation runs
// per candidate whatever n is.  The step is clamped to the trust region and
// validated by the backtracking line search of Eq. line-search; failing that,
// the dogleg step (Eq. dogleg), then the single-coordinate step
// (Eq. single-coord) with the same line search, and finally a random
// perturbation.
//
// Mapping.  Each lane of a warp owns one candidate (a slot of per-lane state)
// at a time and takes the next one from a global queue when its candidate
// finishes, so lanes never idle while work remains.  The full-step trial is
// evaluated by each owner.  The failure path is where candidates diverge (a
// third or more of the iterations fail the full step, and such a candidate
// needs up to 2(A+1) more trials), so the warps of a CTA iterate in lock step
// and the failing slots of all of them are compacted into one list that all
// the CTA's threads work through: each failing slot's dogleg and
// single-coordinate steps (whether or not a shorter step will succeed), then
// its remaining line-search trials and the dogleg trial as independent
// kinematics passes, and the trials of its single-coordinate line search, one
// per thread, then per slot the first of them, in the order of Alg. 4, that
// lowered its cost -- the step the sequential method accepts.  The
// single-coordinate trials run in closed form: turning one joint by x about
// its axis z moves the end effector by (1 - cos x) (v x z) + sin x v, with
// v = z x (p_ee - p_j) the joint's Jacobian column, and composes the
// orientation error with the half-angle quaternion [cos x/2, -sin x/2 z], so
// each costs a handful of operations instead of a kinematics pass, and they
// fill the threads the kinematics passes leave idle.  The perturbation's normal pairs of
// the slots that found no step are spread over the CTA as well.
// Per-lane state (joint vector, trial direction, weighted Jacobian, W, W r,
// cost, target row, trial outcomes) lives in shared memory as structure of
// arrays over the lanes, laid out for the largest chain of the launch; joint
// loops are not unrolled, which keeps the kernel small enough for the
// instruction cache at any n.  Each candidate uses its target's robot (the
// launch's robot tables sit in shared memory), also when another lane
// evaluates one of its trials.
#include <algorithm>

#include "hjcd_internal.cuh"

namespace hjcd {

namespace {

constexpr int kLmWarps = 8;  // default warps per CTA; 2 and 4 also built
constexpr int kMaxLsDepth = 31;  // A (validated by the host)

__host__ __device__ constexpr int tri(int r, int c) { return r * (r + 1) / 2 + c; }

// words of per-warp shared state for an n-joint chain and line-search depth A
// W[6], b[6], cost0, t, s, kk, sc_j, sc_step, e[3], q_err[4], sc_z[3], sc_v[3], branch, alpha;
// then one byte per lane and trial: the A + 1 kinematics trials, the A + 1 single-coordinate trials
constexpr int kLmScalars = 33;
__host__ __device__ constexpr int lm_warp_words(int n, int A) { return (8 * n + kLmScalars) * 32 + (A + 1) * 16; }

// trial directions: the LM (or line-search) direction d, the dogleg step d2,
// the single coordinate (joint sc_j by sc_step)
enum TrialKind { kDirLm = 0, kDirDogleg = 1 };

// Per-warp state, field[...][lane] (each lane's own accesses conflict-free);
// n is the layout's chain length (the launch's largest).  A joint's angle and
// trial direction, and rows 2q and 2q + 1 of a Jacobian column, are pairs
// [...][lane][2] that move as one 64-bit access.  The dogleg step d2
// shares its words with row 0 of the weighted Jacobian: it is written column
// by column after that column's last read, and the Jacobian is not read again
// before the next iteration rebuilds it.
struct LmW {
    float* f;
    int n;
    // joint j's angle and LM (or line-search) direction as one pair (one 64-bit access)
    __device__ __forceinline__ float2& thd(int j, int l) const { return reinterpret_cast<float2*>(f)[j * 32 + l]; }
    __device__ __forceinline__ float& th(int j, int l) const { return thd(j, l).x; }
    __device__ __forceinline__ float& d(int j, int l) const { return thd(j, l).y; }
    // rows 2q and 2q + 1 of column i of the weighted Jacobian as one pair (one 64-bit access)
    __device__ __forceinline__ float2& jw2(int q, int i, int l) const {
        return reinterpret_cast<float2*>(f + 2 * n * 32)[(q * n + i) * 32 + l];
    }
    __device__ __forceinline__ float& jw(int r, int i, int l) const {
        return reinterpret_cast<float*>(&jw2(r >> 1, i, l))[r & 1];
    }
    // column i's six rows
    __device__ __forceinline__ void col6(int i, int l, float (&c)[6]) const {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float2 v = jw2(q, i, l);
            c[2 * q] = v.x;
            c[2 * q + 1] = v.y;
        }
    }
    __device__ __forceinline__ void set_col6(int i, int l, const float (&c)[6]) const {
#pragma unroll
        for (int q = 0; q < 3; ++q) jw2(q, i, l) = make_float2(c[2 * q], c[2 * q + 1]);
    }
    __device__ __forceinline__ float& d2(int j, int l) const { return jw(0, j, l); }
    __device__ __forceinline__ float& W(int r, int l) const { return f[(8 * n + r) * 32 + l]; }
    __device__ __forceinline__ float& b(int r, int l) const { return f[(8 * n + 6 + r) * 32 + l]; }
    __device__ __forceinline__ float& cost0(int l) const { return f[(8 * n + 12) * 32 + l]; }
    __device__ __forceinline__ int& t(int l) const { return reinterpret_cast<int*>(f)[(8 * n + 13) * 32 + l]; }
    __device__ __forceinline__ int& s(int l) const { return reinterpret_cast<int*>(f)[(8 * n + 14) * 32 + l]; }
    __device__ __forceinline__ int& kk(int l) const { return reinterpret_cast<int*>(f)[(8 * n + 15) * 32 + l]; }
    __device__ __forceinline__ int& sc_j(int l) const { return reinterpret_cast<int*>(f)[(8 * n + 16) * 32 + l]; }
    __device__ __forceinline__ float& sc_step(int l) const { return f[(8 * n + 17) * 32 + l]; }
    // position error and error quaternion at the iteration's configuration; the single
    // coordinate's axis and position Jacobian column (unweighted)
    __device__ __forceinline__ float& e(int r, int l) const { return f[(8 * n + 18 + r) * 32 + l]; }
    __device__ __forceinline__ float& qe(int r, int l) const { return f[(8 * n + 21 + r) * 32 + l]; }
    __device__ __forceinline__ float& sc_z(int r, int l) const { return f[(8 * n + 25 + r) * 32 + l]; }
    __device__ __forceinline__ float& sc_v(int r, int l) const { return f[(8 * n + 28 + r) * 32 + l]; }
    // the failure path's outcome for the owner: Alg. 4 branch and accepted alpha
    __device__ __forceinline__ int& br(int l) const { return reinterpret_cast<int*>(f)[(8 * n + 31) * 32 + l]; }
    __device__ __forceinline__ float& al(int l) const { return f[(8 * n + 32) * 32 + l]; }
    // trial i lowered the cost (i < A + 1: kinematics trial i; else single-coordinate trial i - A - 1)
    __device__ __forceinline__ uint8_t& ok(int i, int l) const {
        return reinterpret_cast<uint8_t*>(f + (8 * n + kLmScalars) * 32)[i * 32 + l];
    }
};

// In-place Cholesky of a packed 6 x 6 symmetric positive-definite matrix
// (lower triangle, row by row); inv receives the reciprocal pivots.  One
// template instance per column keeps every index a compile-time constant, so
// the matrix stays in registers.
template <int J>
__device__ __forceinline__ void chol_col(float (&a)[21], float (&inv)[6]) {
    float s = a[tri(J, J)];
#pragma unroll
    for (int k = 0; k < J; ++k) s = fmaf(-a[tri(J, k)], a[tri(J, k)], s);
    const float r = rsqrtf(fmaxf(s, 1e-30f));
    a[tri(J, J)] = s * r;
    inv[J] = r;
#pragma unroll
    for (int i = J + 1; i < 6; ++i) {
        float t = a[tri(i, J)];
#pragma unroll
        for (int k = 0; k < J; ++k) t = fmaf(-a[tri(i, k)], a[tri(J, k)], t);
        a[tri(i, J)] = t * r;
    }
}

__device__ __forceinline__ void chol6(float (&a)[21], float (&inv)[6]) {
    chol_col<0>(a, inv);
    chol_col<1>(a, inv);
    chol_col<2>(a, inv);
    chol_col<3>(a, inv);
    chol_col<4>(a, inv);
    chol_col<5>(a, inv);
}

__device__ __forceinline__ void chol6_solve(const float (&L)[21], const float (&inv)[6], const float (&b)[6],
                                            float (&x)[6]) {
    float y[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        float t = b[i];
#pragma unroll
        for (int k = 0; k < i; ++k) t = fmaf(-L[tri(i, k)], y[k], t);
        y[i] = t * inv[i];
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        float t = y[i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) t = fmaf(-L[tri(k, i)], x[k], t);
        x[i] = t * inv[i];
    }
}

struct Y6 {
    float v[6];
};

// Solve M y = b with M the 6 x 6 sum over the joints of col col^T plus reg I,
// for lane l's Jacobian columns, each first weighted by the rows' W (and
// stored back, so the smem Jacobian becomes W J) and then scaled to unit
// length (S = D^-1/2 of the push-through LM step).
__device__ __noinline__ Y6 normal_solve(const LmW S, int l, int n, float reg, Y6 w, Y6 b) {
    float M[21], inv[6];
#pragma unroll
    for (int q = 0; q < 21; ++q) M[q] = 0.0f;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        float col[6], dd = 1e-9f;
        S.col6(i, l, col);
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            col[r] *= w.v[r];
            dd = fmaf(col[r], col[r], dd);
        }
        S.set_col6(i, l, col);
        const float rs = rsqrtf(dd);
#pragma unroll
        for (int r = 0; r < 6; ++r) col[r] *= rs;
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int q = 0; q <= r; ++q) M[tri(r, q)] = fmaf(col[r], col[q], M[tri(r, q)]);
    }
#pragma unroll
    for (int r = 0; r < 6; ++r) M[tri(r, r)] += reg;
    chol6(M, inv);
    Y6 y;
    chol6_solve(M, inv, b.v, y.v);
    return y;
}

// alpha_i = 1 / beta^i by repeated division, i = 0 .. A, into a table of the CTA (one set of bits
// for every thread)
__device__ __forceinline__ void ls_alphas(float* tab, int A, float beta) {
    float a = 1.0f;
    for (int i = 0; i <= A; ++i) {
        tab[i] = a;
        a = a / beta;
    }
}

// CTA-wide lists of the failure path (after the warps' state): per warp its mask of failing
// lanes, the failing slots compacted, the slots left to the perturbation and their count.
template <int WARPS>
struct LmCta {
    unsigned* wm;
    int* fl;
    int* pl;
    int* np;
    int* hand;  // the CTA leaves its candidates to the next launch
};
template <int WARPS>
__host__ __device__ constexpr int lm_cta_words() { return WARPS + 2 * WARPS * 32 + 2; }
template <int WARPS>
__device__ __forceinline__ LmCta<WARPS> lm_cta(float* f) {
    int* b = reinterpret_cast<int*>(f);
    return LmCta<WARPS>{reinterpret_cast<unsigned*>(b), b + WARPS, b + WARPS + WARPS * 32, b + WARPS + 2 * WARPS * 32,
                        b + WARPS + 2 * WARPS * 32 + 1};
}

// 1/2 |W r|^2 of a residual r = (e, om)
__device__ __forceinline__ float weighted_cost(const float (&w)[6], const V3 e, const V3 om) {
    const float e0 = w[0] * e.x, e1 = w[1] * e.y, e2 = w[2] * e.z;
    const float e3 = w[3] * om.x, e4 = w[4] * om.y, e5 = w[5] * om.z;
    return 0.5f * fmaf(e0, e0, fmaf(e1, e1, fmaf(e2, e2, fmaf(e3, e3, fmaf(e4, e4, e5 * e5)))));
}

// weighted cost 1/2 |W r|^2 at the trial point clamp(theta + alpha dir) of lane s
// (the kinematics passes, the 6 x 6 solve and the trial spreading each exist
// once in the kernel, called from every branch that needs them, which keeps
// the per-iteration body inside the instruction cache)
template <bool RED>
__device__ __noinline__ float trial_cost(const RobotParams* rob, const TargetDesc* tg, int row, const LmW S, int s,
                                        float alpha, int kind) {
    const TargetDesc T = tg[row];
    const RobotParams& R = rob[T.robot];
    Frame F = frame_identity();
#pragma unroll 1
    for (int j = 0; j < R.n; ++j) {
        const float2 td = S.thd(j, s);
        const float dir = kind == kDirDogleg ? S.d2(j, s) : td.y;
        fk_step<RED>(R, j, clampf(fmaf(alpha, dir, td.x), R.lim[j].x, R.lim[j].y), F);
    }
    const Frame E = fk_flange(R, F);
    const V3 w = quat_log(quat_error(T, quat_from_frame(E)));
    const float w6[6] = {S.W(0, s), S.W(1, s), S.W(2, s), S.W(3, s), S.W(4, s), S.W(5, s)};
    return weighted_cost(w6, v3(T.p[0] - E.p.x, T.p[1] - E.p.y, T.p[2] - E.p.z), w);
}

// theta <- clamp(theta + alpha dir) for lane s (the trial point the cost was taken at)
__device__ __noinline__ void take_step(const RobotParams& R, const LmW S, int s, float alpha, int kind) {
#pragma unroll 1
    for (int j = 0; j < R.n; ++j) {
        const float2 td = S.thd(j, s);
        const float dir = kind == kDirDogleg ? S.d2(j, s) : td.y;
        S.th(j, s) = clampf(fmaf(alpha, dir, td.x), R.lim[j].x, R.lim[j].y);
    }
}

// The kinematics-pass trials that follow a failed full step, in the order Alg. 4
// takes them: item i < A is the line-search trial alpha = 1/beta^(i+1) along d,
// item A the dogleg step.
__device__ __forceinline__ void trial_item(int i, int A, const float* alphas, int* kind, float* alpha) {
    *kind = i < A ? kDirLm : kDirDogleg;
    *alpha = i < A ? alphas[i + 1] : 1.0f;
}

// Weighted cost of a configuration (position error e0, error quaternion q) with its single
// coordinate (axis z, position Jacobian column v) turned by x: the end effector rotated by x about
// the joint's axis (see the mapping notes above).
__device__ __forceinline__ float coord_cost_at(const float (&w6)[6], const V3 z, const V3 v, const V3 e0, const Q4 q,
                                               float x) {
    float sh, ch;
    sincos_red(0.5f * x, &sh, &ch);
    const V3 up = cross(v, z);  // component of p_ee - p_j normal to the axis
    const float a = 2.0f * sh * sh, b = 2.0f * sh * ch;  // 1 - cos x, sin x
    const V3 e = fma3(a, up, fma3(-b, v, e0));
    Q4 q2{fmaf(q.w, ch, sh * dot(q.v, z)), fma3(ch, q.v, (-sh) * fma3(q.w, z, cross(q.v, z)))};
    if (q2.w < 0.0f) {
        q2.w = -q2.w;
        q2.v = (-1.0f) * q2.v;
    }
    return weighted_cost(w6, e, quat_log(q2));
}
__device__ __noinline__ float coord_cost(const LmW S, int l, float x) {
    const float w6[6] = {S.W(0, l), S.W(1, l), S.W(2, l), S.W(3, l), S.W(4, l), S.W(5, l)};
    return coord_cost_at(w6, v3(S.sc_z(0, l), S.sc_z(1, l), S.sc_z(2, l)), v3(S.sc_v(0, l), S.sc_v(1, l), S.sc_v(2, l)),
                         v3(S.e(0, l), S.e(1, l), S.e(2, l)), Q4{S.qe(0, l), v3(S.qe(1, l), S.qe(2, l), S.qe(3, l))}, x);
}

// One joint's terms of |d_gn|^2 and, for the segment from d_gn to the Cauchy point ac g, of
// |d_cp - d_gn|^2 and 2 d_gn.(d_cp - d_gn)
__device__ __forceinline__ void dogleg_terms(float dgn, float g, float ac, float& ngn2, float& qa, float& qb) {
    const float di = fmaf(ac, g, -dgn);
    ngn2 = fmaf(dgn, dgn, ngn2);
    qa = fmaf(di, di, qa);
    qb = fmaf(2.0f * dgn, di, qb);
}

// The dogleg step wgn d_gn + wgd g inside the radius Rt (ngd2 = |d_cp|^2)
__device__ __forceinline__ void dogleg_weights(float ngn2, float ngd2, float qa, float qb, float ac, float Rt, float& wgn,
                                               float& wgd) {
    const float R2 = Rt * Rt;
    wgn = 1.0f;
    wgd = 0.0f;
    if (ngn2 <= R2) {
        wgn = 1.0f;
        wgd = 0.0f;
    } else if (ngd2 >= R2) {
        wgn = 0.0f;
        wgd = ngd2 > 0.0f ? Rt * rsqrtf(ngd2) * ac : 0.0f;
    } else {
        // the point of the segment from the Gauss-Newton step to the Cauchy point on the boundary
        const float qc = ngn2 - R2;
        const float disc = fmaxf(fmaf(qb, qb, -4.0f * qa * qc), 0.0f);
        const float tau = (2.0f * qc) / (sqrtf(disc) - qb);  // smaller root, stable form (qb < 0 here)
        wgn = 1.0f - tau;
        wgd = tau * ac;
    }
}

// The dogleg step of Eq. dogleg and the single-coordinate step of Eq. single-coord for lane l,
// from its weighted Jacobian W J (columns in shared memory) and W r: into S.d2, S.sc_j,
// S.sc_step.  With M0 = (WJ)(WJ)^T the Gauss-Newton step is (WJ)^T y2, y2 = (M0 + reg I)^-1 W r,
// and the Cauchy point's quantities reduce to 6 x 6 forms: J g = M0 W r, |g|^2 = (W r).M0 W r.
// |d_gn|^2 is summed over the step's components instead of as y2.M0 y2: when M0 is nearly
// singular y2 is large and that form cancels catastrophically (its binary32 value could fall
// inside the trust region while the step is far outside).  The first pass over the columns
// gives |d_gn|^2 and the coefficients of the segment's crossing of the boundary, the second
// forms the step.
__device__ __noinline__ void dogleg_prepare(const LmW S, int l, int n, float Rt, float gn_reg) {
    float M0[21], M[21], inv[6], b[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) b[r] = S.b(r, l);
#pragma unroll
    for (int q = 0; q < 21; ++q) M0[q] = 0.0f;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        float col[6];
        S.col6(i, l, col);
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int q = 0; q <= r; ++q) M0[tri(r, q)] = fmaf(col[r], col[q], M0[tri(r, q)]);
    }
#pragma unroll
    for (int q = 0; q < 21; ++q) M[q] = M0[q];
#pragma unroll
    for (int r = 0; r < 6; ++r) M[tri(r, r)] += gn_reg;
    chol6(M, inv);
    float y2[6];
    chol6_solve(M, inv, b, y2);
    // J g = M0 W r
    float Jg[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        float a = 0.0f;
#pragma unroll
        for (int q = 0; q < 6; ++q) a = fmaf(r >= q ? M0[tri(r, q)] : M0[tri(q, r)], b[q], a);
        Jg[r] = a;
    }
    float gg = 0.0f, jgjg = 0.0f;
#pragma unroll
    for (int r = 0; r < 6; ++r) {
        gg = fmaf(b[r], Jg[r], gg);
        jgjg = fmaf(Jg[r], Jg[r], jgjg);
    }
    const float ac = jgjg > 0.0f ? __fdividef(gg, jgjg) : 0.0f;
    const float ngd2 = ac * ac * gg;
    // |d_gn|^2 and, for the segment from d_gn to the Cauchy point, |d_cp - d_gn|^2 and 2 d_gn.(d_cp - d_gn)
    float ngn2 = 0.0f, qa = 0.0f, qb = 0.0f;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        float dgn = 0.0f, g = 0.0f, col[6];
        S.col6(i, l, col);
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            dgn = fmaf(col[r], y2[r], dgn);
            g = fmaf(col[r], b[r], g);
        }
        dogleg_terms(dgn, g, ac, ngn2, qa, qb);
    }
    float wgn, wgd;
    dogleg_weights(ngn2, ngd2, qa, qb, ac, Rt, wgn, wgd);
    // the step, and the single coordinate: the joint with the largest |g_i| (the first of
    // equals), a 1-D Gauss-Newton step on it clamped to R
    int is = 0;
    float gbest = -1.0f, cn = 0.0f, gsel = 0.0f, csel[6];
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        float dgn = 0.0f, g = 0.0f, q2 = 0.0f, col[6];
        S.col6(i, l, col);
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            dgn = fmaf(col[r], y2[r], dgn);
            g = fmaf(col[r], b[r], g);
            q2 = fmaf(col[r], col[r], q2);
        }
        S.d2(i, l) = fmaf(wgn, dgn, wgd * g);
        if (fabsf(g) > gbest) {
            gbest = fabsf(g);
            is = i;
            gsel = g;
            cn = q2;
#pragma unroll
            for (int r = 0; r < 6; ++r) csel[r] = col[r];
        }
    }
    S.sc_j(l) = is;
    S.sc_step(l) = cn > 0.0f ? clampf(__fdividef(gsel, cn), -Rt, Rt) : 0.0f;
    // the chosen joint's position column and axis without the row weights
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        S.sc_v(r, l) = __fdividef(csel[r], S.W(r, l));
        S.sc_z(r, l) = __fdividef(csel[3 + r], S.W(3 + r, l));
    }
}

// RED = false: the launch's joint vectors lie within the limits of plain robots (no offsets and
// no range reduction in the kinematics steps; the same bits)
// HAND: the launch leaves its last candidates to the next one: each CTA, from its hand_at-th iteration
// on, once the queue is empty and hand_lim candidates of the launch or fewer are unfinished
template <bool TRACE, int WARPS, bool RED, bool HAND>
__global__ void __launch_bounds__(WARPS * 32, 16 / WARPS) k_lm(const LmArgs A) {
    extern __shared__ __align__(16) float smem_f[];
    __shared__ float alphas[kMaxLsDepth + 1];
    if (threadIdx.x == 0) ls_alphas(alphas, A.P.lm_A, A.P.lm_beta);  // visible after the staging barrier
    const RobotParams* rob = stage_robots(smem_f, A.rs);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* const warps_f = smem_f + robots_smem_bytes(A.rs.n) / sizeof(float);
    const int words = lm_warp_words(A.rs.n_max, A.P.lm_A);
    const LmW S{warps_f + warp * words, A.rs.n_max};
    // the state of slot sl = warp * 32 + lane, whichever thread works on it
    auto slot_state = [&](int sl) { return LmW{warps_f + (sl >> 5) * words, A.rs.n_max}; };
    const LmCta<WARPS> CL = lm_cta<WARPS>(warps_f + WARPS * words);
    if (HAND) {
        if (threadIdx.x == 0) CL.hand[0] = 0;
        __syncthreads();
    }

    const hjcd_params& P = A.P;
    const float Rt = P.lm_trust_R;
    unsigned long long n_it = 0, n_fk = 0, n_sc = 0;

    bool has = false;
    int rounds = 0;
    int64_t c = 0;
    int32_t t = 0, s = 0, kk = 0, cap = 0;
    TargetDesc T{};

    for (;;) {
        // refill idle lanes from the global queue (one atomic per warp)
        const unsigned need = __ballot_sync(0xffffffffu, !has);
        if (HAND) {  // those whose candidate is finished
            const unsigned fin = __ballot_sync(0xffffffffu, !has && rounds > 0 && c < A.C);
            if (fin && lane == 0) atomicAdd(A.n_done, __popc(fin));
        }
        if (need) {
            const int leader = __ffs(need) - 1;
            long long base = 0;
            if (lane == leader) base = (long long)atomicAdd(A.queue, (unsigned long long)__popc(need));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (!has) {
                c = base + __popc(need & ((1u << lane) - 1u));
                if (c < A.C && A.map.lookup(c, t, s)) {
                    T = A.tg[t];
                    kk = 0;
                    cap = A.n_iters >= 0 ? A.n_iters : T.lm_iters;
                    if (T.eps_pos > 0.0f) {
                        has = true;
                        load_joints<8>(A.th, A.ld, c, rob[T.robot].n, [&](int j, float v) { S.th(j, lane) = v; });
                    } else {  // invalid target: no iterations, infinite score
                        if (A.score) A.score[c] = __int_as_float(0x7f800000);
                        if (A.perr) A.perr[c] = 0.0f;
                        if (A.oerr) A.oerr[c] = 0.0f;
                        if (A.iters) A.iters[c] = cap;
                    }
                }
            }
        }
        // ---- phase A: kinematics with frames, residual, LM step (owner) ----
        const RobotParams& R = rob[T.robot];
        const int n = R.n;
        bool act = false;
        if (has) {
            // joint origins and axes are parked in the lane's J slots
            Frame F = frame_identity();
#pragma unroll 1
            for (int j = 0; j < n; ++j) {
                fk_step<RED>(R, j, S.th(j, lane), F);
                S.jw2(0, j, lane) = make_float2(F.p.x, F.p.y);
                S.jw2(1, j, lane) = make_float2(F.p.z, F.c2.x);
                S.jw2(2, j, lane) = make_float2(F.c2.y, F.c2.z);
            }
            const Frame E = fk_flange(R, F);
            ++n_fk;
            const V3 pt = v3(T.p[0], T.p[1], T.p[2]);
            const Q4 qerr = quat_error(T, quat_from_frame(E));
            const V3 om = quat_log(qerr);
            const V3 epv = pt - E.p;
            const float ep = sqrt_approx(dot(epv, epv)), eo = sqrt_approx(dot(om, om));
            if ((kk > 0 && ep < T.eps_pos && eo < T.eps_ori) || kk == cap) {
                // Alg. 4 break (checked after each update) or the iteration cap
#pragma unroll 1
                for (int j = 0; j < n; ++j) A.th[j * A.ld + c] = S.th(j, lane);
                if (A.score) {
                    const float a = ep / T.eps_pos, bb = eo / T.eps_ori;
                    A.score[c] = fmaf(a, a, bb * bb);
                }
                if (A.perr) A.perr[c] = ep;
                if (A.oerr) A.oerr[c] = eo;
                if (A.iters) A.iters[c] = kk;
                has = false;
            } else {
                act = true;
                // Jacobian columns z_i x (P_ee - P_i), z_i (in place), and the row norms
                float rn[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                for (int i = 0; i < n; ++i) {
                    float fr[6];
                    S.col6(i, lane, fr);
                    const V3 Pi = v3(fr[0], fr[1], fr[2]);
                    const V3 Zi = v3(fr[3], fr[4], fr[5]);
                    const V3 jp = cross(Zi, E.p - Pi);
                    S.jw2(0, i, lane) = make_float2(jp.x, jp.y);
                    S.jw2(1, i, lane) = make_float2(jp.z, Zi.x);
                    const float col[6] = {jp.x, jp.y, jp.z, Zi.x, Zi.y, Zi.z};
#pragma unroll
                    for (int r = 0; r < 6; ++r) {
                        rn[r] = fmaf(col[r], col[r], rn[r]);
                        if (TRACE && kk == 0 && A.tr.J) A.tr.J[(r * n + i) * A.ld + c] = col[r];
                    }
                }
                const float e[6] = {epv.x, epv.y, epv.z, om.x, om.y, om.z};
                const float wo = __fdividef(T.eps_pos, T.eps_ori);
                float W[6], b[6], cost0 = 0.0f;
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    W[r] = (r < 3 ? 1.0f : wo) * rsqrtf(fmaxf(rn[r], 1e-12f));  // c / max(|row|, 1e-6)
                    b[r] = W[r] * e[r];
                    cost0 = fmaf(b[r], b[r], cost0);
                    S.W(r, lane) = W[r];
                    S.b(r, lane) = b[r];
                    if (TRACE && kk == 0 && A.tr.W) A.tr.W[r * A.ld + c] = W[r];
                }
                S.cost0(lane) = 0.5f * cost0;
                S.t(lane) = t;
                S.e(0, lane) = epv.x;
                S.e(1, lane) = epv.y;
                S.e(2, lane) = epv.z;
                S.qe(0, lane) = qerr.w;
                S.qe(1, lane) = qerr.v.x;
                S.qe(2, lane) = qerr.v.y;
                S.qe(3, lane) = qerr.v.z;
                // the push-through LM step on the weighted Jacobian
                Y6 wv, bv;
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    wv.v[r] = W[r];
                    bv.v[r] = b[r];
                }
                const Y6 yy = normal_solve(S, lane, n, P.lm_lambda, wv, bv);
                float y[6];
#pragma unroll
                for (int r = 0; r < 6; ++r) y[r] = yy.v[r];
#pragma unroll 1
                for (int i = 0; i < n; ++i) {
                    float a = 0.0f, dd = 1e-9f, cl[6];
                    S.col6(i, lane, cl);
#pragma unroll
                    for (int r = 0; r < 6; ++r) {
                        a = fmaf(cl[r], y[r], a);
                        dd = fmaf(cl[r], cl[r], dd);
                    }
                    const float st = clampf(__fdividef(a, dd), -Rt, Rt);  // trust region
                    S.d(i, lane) = st;
                    if (TRACE && kk == 0 && A.tr.d_lm) A.tr.d_lm[i * A.ld + c] = st;
                }
            }
        }

        // ---- the full step by its owner ----
        int branch = 3;
        float alpha_acc = 0.0f;
        if (act) {
            ++n_fk;
            if (trial_cost<RED>(rob, A.tg, t, S, lane, 1.0f, kDirLm) < S.cost0(lane)) {
                take_step(R, S, lane, 1.0f, kDirLm);
                branch = 0;
                alpha_acc = 1.0f;
            }
        }
        const bool failed = act && branch != 0;
        if (failed) {
            S.s(lane) = s;
            S.kk(lane) = kk;
        }

        // ---- the failure path over the CTA: the failing slots of all warps, compacted ----
        // (the same barrier ends the loop once no lane holds a candidate and the queue is drained)
        const unsigned fail = __ballot_sync(0xffffffffu, failed);
        if (lane == 0) CL.wm[warp] = fail;
        // (a lane whose candidate just finished still holds an index below C and asks again)
        if (HAND && threadIdx.x == 0 && rounds + 1 >= A.hand_at)
            CL.hand[0] = *(volatile const unsigned long long*)A.queue >= (unsigned long long)A.C &&
                         A.C - *(volatile const int32_t*)A.n_done <= A.hand_lim;
        if (!__syncthreads_or(has || c < A.C)) break;
        const bool hand = HAND && CL.hand[0] != 0;
        int nf = 0, before = 0;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            const int k = __popc(CL.wm[w]);
            before += w < warp ? k : 0;
            nf += k;
        }
        if (failed) CL.fl[before + __popc(fail & ((1u << lane) - 1u))] = threadIdx.x;
        if (threadIdx.x == 0) CL.np[0] = 0;
        __syncthreads();
        if (nf > 0) {
            // dogleg and single-coordinate steps of each failing slot
            for (int i = threadIdx.x; i < nf; i += blockDim.x) {
                const int sl = CL.fl[i], l = sl & 31;
                const LmW Sx = slot_state(sl);
                dogleg_prepare(Sx, l, rob[A.tg[Sx.t(l)].robot].n, Rt, P.lm_gn_reg);
            }
            __syncthreads();
            // the remaining line-search trials and the dogleg trial, one kinematics pass each, then
            // the single-coordinate line search's trials in closed form (each slot's A + 1 of
            // them, whether or not the sequential method gets that far: they take the threads the
            // kinematics passes leave idle)
            const int per = P.lm_A + 1;
            const int nk = nf * per;
            for (int w = threadIdx.x; w < 2 * nk; w += blockDim.x) {
                const int wi = w < nk ? w : w - nk;
                const int sl = CL.fl[wi / per], l = sl & 31, i = wi % per;
                const LmW Sx = slot_state(sl);
                if (w < nk) {
                    int kind;
                    float alpha;
                    trial_item(i, P.lm_A, alphas, &kind, &alpha);
                    Sx.ok(i, l) = trial_cost<RED>(rob, A.tg, Sx.t(l), Sx, l, alpha, kind) < Sx.cost0(l) ? 1 : 0;
                } else {
                    const RobotParams& Rx = rob[A.tg[Sx.t(l)].robot];
                    const int j = Sx.sc_j(l);
                    const float th0 = Sx.th(j, l);
                    const float thj = clampf(fmaf(alphas[i], Sx.sc_step(l), th0), Rx.lim[j].x, Rx.lim[j].y);
                    Sx.ok(per + i, l) = coord_cost(Sx, l, thj - th0) < Sx.cost0(l) ? 1 : 0;
                }
            }
            __syncthreads();
            // each slot's first successful trial in the order of Alg. 4, else the first successful
            // trial of its single-coordinate line search, else the perturbation
            for (int i = threadIdx.x; i < nf; i += blockDim.x) {
                const int sl = CL.fl[i], l = sl & 31;
                const LmW Sx = slot_state(sl);
                const RobotParams& Rx = rob[A.tg[Sx.t(l)].robot];
                int pick = per;
                for (int q = 0; q < per; ++q)
                    if (Sx.ok(q, l)) {
                        pick = q;
                        break;
                    }
                n_fk += pick < per ? pick + 1 : per;  // the passes the sequential method evaluates
                int br = 3;
                float al = 0.0f;
                if (pick < per) {
                    int kind;
                    trial_item(pick, P.lm_A, alphas, &kind, &al);
                    take_step(Rx, Sx, l, al, kind);
                    br = kind == kDirLm ? 0 : 1;
                    if (kind == kDirDogleg) al = 0.0f;  // no line-search alpha (as traced)
                } else {
                    int qc = per;
                    for (int q = 0; q < per; ++q)
                        if (Sx.ok(per + q, l)) {
                            qc = q;
                            break;
                        }
                    n_sc += qc < per ? qc + 1 : per;  // the trials the sequential method evaluates
                    if (qc < per) {
                        const int j = Sx.sc_j(l);
                        const float th0 = Sx.th(j, l);
                        Sx.th(j, l) = clampf(fmaf(alphas[qc], Sx.sc_step(l), th0), Rx.lim[j].x, Rx.lim[j].y);
                        br = 2;
                        al = alphas[qc];
                    } else {
                        CL.pl[atomicAdd(CL.np, 1)] = sl;
                    }
                }
                Sx.br(l) = br;
                Sx.al(l) = al;
            }
            __syncthreads();
            // the perturbation of Alg. 4: normal pairs of every slot that found no step
            const int np = CL.np[0];
            if (np > 0) {
                const int pp = (A.rs.n_max + 1) / 2;
                for (int w = threadIdx.x; w < np * pp; w += blockDim.x) {
                    const int sl = CL.pl[w / pp], l = sl & 31, q = w % pp;
                    const LmW Sx = slot_state(sl);
                    const TargetDesc& Tx = A.tg[Sx.t(l)];
                    const RobotParams& Rx = rob[Tx.robot];
                    const int j0 = 2 * q, j1 = 2 * q + 1;
                    if (j0 >= Rx.n) continue;
                    const float2 z = normal_pair(Tx, (uint32_t)Sx.s(l), kPhaseLm, (uint32_t)A.k0 + (uint32_t)Sx.kk(l), q);
                    Sx.th(j0, l) = clampf(fmaf(P.lm_sigma, z.x, Sx.th(j0, l)), Rx.lim[j0].x, Rx.lim[j0].y);
                    if (j1 < Rx.n) Sx.th(j1, l) = clampf(fmaf(P.lm_sigma, z.y, Sx.th(j1, l)), Rx.lim[j1].x, Rx.lim[j1].y);
                }
                __syncthreads();
            }
            if (failed) {
                branch = S.br(lane);
                alpha_acc = S.al(lane);
            }
        }
        if (act) {
            if (TRACE && kk == 0) {
                if (A.tr.branch) A.tr.branch[c] = branch;
                if (A.tr.alpha) A.tr.alpha[c] = alpha_acc;
                if (failed) {  // the fallback steps exist for the slots whose full step failed
                    if (A.tr.d_dog)
#pragma unroll 1
                        for (int j = 0; j < n; ++j) A.tr.d_dog[j * A.ld + c] = S.d2(j, lane);
                    if (A.tr.sc_joint) A.tr.sc_joint[c] = S.sc_j(lane);
                    if (A.tr.sc_step) A.tr.sc_step[c] = S.sc_step(lane);
                }
            }
            ++kk;
            ++n_it;
        }
        __syncwarp();
        if (HAND) ++rounds;
        if (hand) {
            // the candidates that are left, packed afresh, take less time in the kernel that spreads a
            // candidate over a CTA
            const unsigned m = __ballot_sync(0xffffffffu, has);
            int at = 0;
            if (lane == 0 && m) at = atomicAdd(A.n_list, __popc(m));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
            if (has) {
                A.list[at] = (int32_t)c;
                A.list_k[at] = kk;
#pragma unroll 1
                for (int j = 0; j < n; ++j) A.th[j * A.ld + c] = S.th(j, lane);
            }
            break;
        }
    }
    if (A.cnt) {
        n_it = warp_sum(n_it);
        n_fk = warp_sum(n_fk);
        n_sc = warp_sum(n_sc);
        if (lane == 0) {
            atomicAdd(&A.cnt->v[1], n_it);
            atomicAdd(&A.cnt->v[2], n_fk);
            atomicAdd(&A.cnt->v[7], n_sc);
        }
    }
}

// ----------------------------------------------------------------------------
// PJ-IK with a candidate's work spread over a CTA, for batches too small to fill the GPU with one
// lane per candidate: there the time is the latency of one candidate's chain of iterations.  A CTA
// takes 16 candidates; a half warp (a unit) works on one part of all of them at a time -- a row of a
// kinematics chain, a joint's column, an entry of a normal matrix, a trial -- and the units exchange
// through shared memory.  Every trial of Alg. 4 is taken at once (the line search, the dogleg step,
// the single coordinate), and so is the set-up of the dogleg step beside that of the LM step: with
// 16 candidates some full step nearly always fails, and the units would idle otherwise.  The
// perturbation's draws are made beside the factorisations.  Each quantity is formed by k_lm's
// operations in their order (the sums over the joints and over the rows as well), so the results
// are its bits.  Bound by latency: thirteen exchanges per iteration, the residuals (a lone warp's
// chain of about 150 dependent instructions) and the 6 x 6 solve the longest stages; about an eighth of
// the warps' time outside barriers is instruction fetch (a stage's code runs once per iteration and all of
// it does not stay in the first cache), so work moved beside other work pays only where it adds little
// code.  Loads stand ahead of stores, which the compiler does not move them across.  One Panda target of
// 1000 seeds: 70 us for at most 20 iterations, where k_lm takes 172 us (74 before the loads were moved
// ahead in the kinematics rows, columns and matrix entries).
constexpr int kCoopCands = 16;    // candidates per CTA
constexpr int kCoopLmWarps = 16;  // most warps per CTA
constexpr int kCoopMaxA = 6;      // deepest line search taken here

// Shared state [field][candidate], pointers at this thread's candidate; nl joints in the layout.
struct LmC {
    int nl;
    float4* e4;  // [set][row]: that row of the last frame (its axes c0, c1, c2 and origin); set 0 the
                 // configuration, 1 + i trial i
    float2* c2;  // [set][joint]: cosine and sine of the joint's angle
    float* f;
    __device__ __forceinline__ float4& e(int set, int row) const { return e4[(set * 3 + row) * kCoopCands]; }
    __device__ __forceinline__ float2& cs(int set, int j) const { return c2[(set * nl + j) * kCoopCands]; }
    __device__ __forceinline__ float& at(int i) const { return f[i * kCoopCands]; }
    __device__ __forceinline__ float& th(int j) const { return at(j); }
    __device__ __forceinline__ float& st(int j) const { return at(nl + j); }       // LM step
    __device__ __forceinline__ float& dgn(int j) const { return at(2 * nl + j); }  // Gauss-Newton step
    __device__ __forceinline__ float& g(int j) const { return at(3 * nl + j); }    // gradient
    __device__ __forceinline__ float& dd(int j) const { return at(4 * nl + j); }   // squared column norm
    __device__ __forceinline__ float& jc(int r, int j) const { return at((5 + r) * nl + j); }   // J, then W J
    __device__ __forceinline__ float& sc(int r, int j) const { return at((11 + r) * nl + j); }  // W J S
    __device__ __forceinline__ float& fr(int r, int j) const { return at((17 + r) * nl + j); }  // joint origin, axis
    __device__ __forceinline__ float& nz(int j) const { return at(23 * nl + j); }  // normal draws, nl + 1 rows
    __device__ __forceinline__ float& s(int i) const { return at(24 * nl + 1 + i); }
    __device__ __forceinline__ int& si(int i) const { return reinterpret_cast<int&>(s(i)); }
};
// scalars of LmC::s: M of the LM step and of the Gauss-Newton step, their solutions, W, W r, the
// error, the error quaternion, the single coordinate's axis, column, joint and step, ...
enum { kM = 0, kM0 = 21, kY = 42, kY2 = 48, kW = 54, kB = 60, kE = 66, kQ = 72, kSz = 76, kSv = 79, kSj = 82, kSstep = 83,
       kCost = 84, kAc = 85, kNgd2 = 86, kWgn = 87, kWgd = 88, kStat = 89, kMask = 90, kLmCScalars = 91 };
__host__ __device__ constexpr size_t coop_lm_bytes(int n, int A) {
    return sizeof(float) * kCoopCands * ((size_t)12 * (A + 3) + (size_t)2 * (A + 3) * n + 24 * n + 1 + kLmCScalars);
}

// One row of a kinematics chain (fk_step's operations on that row) from the sines and cosines of
// `set`; with FRAMES every joint's origin and axis go to C.fr
template <int N, bool FRAMES>
__device__ __forceinline__ void lmc_fk_row(const LmC& C, const RobotParams& R, int n_, int set, int row) {
    const int n = N ? N : n_;
    float c0 = row == 0 ? 1.0f : 0.0f, c1 = row == 1 ? 1.0f : 0.0f, c2 = row == 2 ? 1.0f : 0.0f, p = 0.0f;
    auto step = [&](int j, const float4 g, const float2 cs) {
        const float b1 = fmaf(g.x, c1, g.y * c2);
        const float b2 = fmaf(g.x, c2, (-g.y) * c1);
        p = fmaf(g.w, b2, fmaf(g.z, c0, p));
        const float n0 = fmaf(cs.x, c0, cs.y * b1);
        c1 = fmaf(cs.x, b1, (-cs.y) * c0);
        c0 = n0;
        c2 = b2;
        if (FRAMES) {
            C.fr(row, j) = p;
            C.fr(3 + row, j) = c2;
        }
    };
    if (N) {  // all loads come before the stores, which the compiler may not move them across
        float4 g[N ? N : 1];
        float2 cs[N ? N : 1];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            g[j] = R.dh[j];
            cs[j] = C.cs(set, j);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) step(j, g[j], cs[j]);
    } else {
#pragma unroll 4
        for (int j = 0; j < n; ++j) step(j, R.dh[j], C.cs(set, j));
    }
    C.e(set, row) = make_float4(c0, c1, c2, p);
}
// flange frame of a set
__device__ __forceinline__ Frame lmc_flange(const LmC& C, const RobotParams& R, int set) {
    const float4 a = C.e(set, 0), b = C.e(set, 1), c = C.e(set, 2);
    return fk_flange(R, Frame{v3(a.x, b.x, c.x), v3(a.y, b.y, c.y), v3(a.z, b.z, c.z), v3(a.w, b.w, c.w)});
}

// row and column of entry q of a packed lower triangle
__device__ __constant__ int8_t kTriRow[21] = {0, 1, 1, 2, 2, 2, 3, 3, 3, 3, 4, 4, 4, 4, 4, 5, 5, 5, 5, 5, 5};
__device__ __constant__ int8_t kTriCol[21] = {0, 0, 1, 0, 1, 2, 0, 1, 2, 3, 0, 1, 2, 3, 4, 0, 1, 2, 3, 4, 5};

// RED as for k_lm; N > 0: the launch's one robot has N joints (unrolled loops); N = 0: any robots;
// LIST: the candidates that a k_lm launch handed over, from the iterations they had reached
template <bool RED, int N, bool LIST>
__global__ void __launch_bounds__(kCoopLmWarps * 32, 1) k_lm_coop(const LmArgs A) {
    extern __shared__ __align__(16) float smem_f[];
    grid_follow();
    __shared__ float alphas[kCoopMaxA + 1];
    if (threadIdx.x == 0) ls_alphas(alphas, A.P.lm_A, A.P.lm_beta);  // visible after the staging barrier
    const RobotParams* rob = stage_robots(smem_f, A.rs);
    const hjcd_params& P = A.P;
    const float Rt = P.lm_trust_R;
    const int lsA = P.lm_A, nt = lsA + 2;  // kinematics trials: the full step, the line search, the dogleg
    const int nl = N ? N : A.rs.n_max;
    const int W = (int)blockDim.x >> 5, U = 2 * W;
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const int l = lane & (kCoopCands - 1), half = lane >> 4, u = 2 * warp + half;
    LmC C;
    C.nl = nl;
    C.e4 = reinterpret_cast<float4*>(reinterpret_cast<char*>(smem_f) + robots_smem_bytes(A.rs.n)) + l;
    C.c2 = reinterpret_cast<float2*>(C.e4 - l + 3 * (nt + 1) * kCoopCands) + l;
    C.f = reinterpret_cast<float*>(C.c2 - l + (nt + 1) * nl * kCoopCands) + l;
    unsigned long long n_it = 0, n_fk = 0, n_sc = 0;
    auto sincos_of = [&](const RobotParams& R, int j, float th) {
        float sn, cn;
        if (RED) sincos_red(th + R.off[j], &sn, &cn);
        else __sincosf(th, &sn, &cn);
        return make_float2(cn, sn);
    };

    // the normal matrices' entries of this unit: q and q + U of 42, their operands found once
    auto entry = [&](int q, const float*& a, const float*& b) {
        const int k = q < 21 ? q : q - 21;
        a = q < 21 ? &C.sc(kTriRow[k], 0) : &C.jc(kTriRow[k], 0);
        b = q < 21 ? &C.sc(kTriCol[k], 0) : &C.jc(kTriCol[k], 0);
    };
    const float *a0, *b0, *a1, *b1;
    entry(u, a0, b0);  // (u < 32)
    entry(min(u + U, 41), a1, b1);
    const int64_t items = LIST ? (int64_t)*A.n_list : A.C;
    for (int64_t base = kCoopCands * (int64_t)blockIdx.x; base < items; base += kCoopCands * (int64_t)gridDim.x) {
        __syncthreads();  // the last group's state is no longer read
        int32_t t = 0, s = 0;
        bool have = base + l < items;
        const int64_t c = LIST && have ? (int64_t)A.list[base + l] : base + l;
        const int kbase = LIST && have ? A.list_k[base + l] : 0;  // iterations taken before the hand-over
        if (have) have = A.map.lookup(c, t, s);
        const TargetDesc T = A.tg[have ? t : 0];
        const RobotParams& R = N ? rob[0] : rob[have ? T.robot : 0];
        const int n = N ? N : R.n;  // (a lane without a candidate runs along on a robot's joints, unread)
        const int cap = A.n_iters >= 0 ? A.n_iters : T.lm_iters;
        bool alive = have && T.eps_pos > 0.0f;
        if (have && !alive && u == 0) {  // invalid target: no iterations, infinite score
            if (A.score) A.score[c] = __int_as_float(0x7f800000);
            if (A.perr) A.perr[c] = 0.0f;
            if (A.oerr) A.oerr[c] = 0.0f;
            if (A.iters) A.iters[c] = cap;
        }
        const bool mine = alive;
        for (int j = u; j < n; j += U) {
            const float th = mine ? A.th[j * A.ld + c] : 0.0f;
            C.th(j) = th;
            C.cs(0, j) = sincos_of(R, j, th);
        }
        if (u == 0) C.si(kStat) = 0;
        __syncthreads();

        auto trial_sincos = [&](int i, int j) {  // of trial i's angle of joint j
            const float dir = i <= lsA ? C.st(j) : fmaf(C.s(kWgn), C.dgn(j), C.s(kWgd) * C.g(j));
            const float al = i <= lsA ? alphas[i] : 1.0f;
            C.cs(1 + i, j) = sincos_of(R, j, clampf(fmaf(al, dir, C.th(j)), R.lim[j].x, R.lim[j].y));
        };
        for (int kk = kbase;; ++kk) {
            // kinematics with frames
            if (u < 3) lmc_fk_row<N, true>(C, R, n, 0, u);
            __syncthreads();

            // the last warp: residual and break; the others: Jacobian columns z_i x (P_ee - P_i), z_i
            {
                const Frame E = lmc_flange(C, R, 0);
                if (warp == W - 1) {
                    const Q4 qerr = quat_error(T, quat_from_frame(E));
                    const V3 om = quat_log(qerr);
                    const V3 epv = v3(T.p[0], T.p[1], T.p[2]) - E.p;
                    const float ep = sqrt_approx(dot(epv, epv)), eo = sqrt_approx(dot(om, om));
                    if (alive && half == 0) {
                        ++n_fk;
                        if ((kk > 0 && ep < T.eps_pos && eo < T.eps_ori) || kk == cap) {
                            if (A.score) {
                                const float a = ep / T.eps_pos, bb = eo / T.eps_ori;
                                A.score[c] = fmaf(a, a, bb * bb);
                            }
                            if (A.perr) A.perr[c] = ep;
                            if (A.oerr) A.oerr[c] = eo;
                            if (A.iters) A.iters[c] = kk;
                            C.si(kStat) = 1;
                        }
                        C.s(kE) = epv.x;
                        C.s(kE + 1) = epv.y;
                        C.s(kE + 2) = epv.z;
                        C.s(kE + 3) = om.x;
                        C.s(kE + 4) = om.y;
                        C.s(kE + 5) = om.z;
                        C.s(kQ) = qerr.w;
                        C.s(kQ + 1) = qerr.v.x;
                        C.s(kQ + 2) = qerr.v.y;
                        C.s(kQ + 3) = qerr.v.z;
                    }
                } else {
                    for (int j = u; j < n; j += U - 2) {
                        const V3 Zi = v3(C.fr(3, j), C.fr(4, j), C.fr(5, j));
                        const V3 jp = cross(Zi, E.p - v3(C.fr(0, j), C.fr(1, j), C.fr(2, j)));
                        C.jc(0, j) = jp.x;
                        C.jc(1, j) = jp.y;
                        C.jc(2, j) = jp.z;
                        C.jc(3, j) = Zi.x;
                        C.jc(4, j) = Zi.y;
                        C.jc(5, j) = Zi.z;
                    }
                }
            }
            __syncthreads();
            alive = alive && C.si(kStat) == 0;

            // row norms, W and W r
            if (u < 6) {
                float rn = 0.0f;
#pragma unroll 4
                for (int j = 0; j < n; ++j) {
                    const float v = C.jc(u, j);
                    rn = fmaf(v, v, rn);
                }
                const float wo = __fdividef(T.eps_pos, T.eps_ori);
                const float w = (u < 3 ? 1.0f : wo) * rsqrtf(fmaxf(rn, 1e-12f));  // c / max(|row|, 1e-6)
                C.s(kW + u) = w;
                C.s(kB + u) = w * C.s(kE + u);
            }
            if (!__syncthreads_or(alive)) break;

            // weighted columns and those scaled to unit length; the last warp: the cost
            if (warp == W - 1) {
                float cost0 = 0.0f;
#pragma unroll
                for (int r = 0; r < 6; ++r) cost0 = fmaf(C.s(kB + r), C.s(kB + r), cost0);
                if (half == 0) {
                    C.s(kCost) = 0.5f * cost0;
                    C.si(kMask) = 0;
                }
            } else {
                for (int j = u; j < n; j += U - 2) {
                    float col[6], w[6], dd = 1e-9f;
#pragma unroll
                    for (int r = 0; r < 6; ++r) {
                        col[r] = C.jc(r, j);
                        w[r] = C.s(kW + r);
                    }
#pragma unroll
                    for (int r = 0; r < 6; ++r) {
                        col[r] *= w[r];
                        dd = fmaf(col[r], col[r], dd);
                    }
#pragma unroll
                    for (int r = 0; r < 6; ++r) C.jc(r, j) = col[r];
                    const float rs = rsqrtf(dd);
                    C.dd(j) = dd;
#pragma unroll
                    for (int r = 0; r < 6; ++r) C.sc(r, j) = col[r] * rs;
                }
            }
            __syncthreads();

            // the normal matrices: entry q of the scaled columns' (LM), of the columns' (Gauss-Newton)
            {
                float m0 = 0.0f, m1 = 0.0f;
#pragma unroll(N ? N : 4)
                for (int j = 0; j < n; ++j) {
                    m0 = fmaf(a0[j * kCoopCands], b0[j * kCoopCands], m0);
                    m1 = fmaf(a1[j * kCoopCands], b1[j * kCoopCands], m1);
                }
                C.s(kM + u) = m0;
                if (u + U < 42) C.s(kM + u + U) = m1;
                for (int q = u + 2 * U; q < 42; q += U) {
                    const float *a, *b;
                    entry(q, a, b);
                    float m = 0.0f;
#pragma unroll 4
                    for (int j = 0; j < n; ++j) m = fmaf(a[j * kCoopCands], b[j * kCoopCands], m);
                    C.s(kM + q) = m;
                }
            }
            __syncthreads();

            // factorisations and solutions, the LM system in the lower half of warp 0 and the
            // Gauss-Newton system in the upper one; the other warps draw the perturbation
            if (warp == 0) {
                const int m0 = half ? kM0 : kM;
                const float reg = half ? P.lm_gn_reg : P.lm_lambda;
                float M[21], inv[6], b[6], y[6];
#pragma unroll
                for (int q = 0; q < 21; ++q) M[q] = C.s(m0 + q);
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    b[r] = C.s(kB + r);
                    M[tri(r, r)] += reg;
                }
                chol6(M, inv);
                chol6_solve(M, inv, b, y);
#pragma unroll
                for (int r = 0; r < 6; ++r) C.s((half ? kY2 : kY) + r) = y[r];
            } else if (warp == 1) {
                // J g = M0 W r, the Cauchy point
                float Jg[6], gg = 0.0f, jgjg = 0.0f;
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    float a = 0.0f;
#pragma unroll
                    for (int q = 0; q < 6; ++q) a = fmaf(C.s(kM0 + (r >= q ? tri(r, q) : tri(q, r))), C.s(kB + q), a);
                    Jg[r] = a;
                }
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    gg = fmaf(C.s(kB + r), Jg[r], gg);
                    jgjg = fmaf(Jg[r], Jg[r], jgjg);
                }
                const float ac = jgjg > 0.0f ? __fdividef(gg, jgjg) : 0.0f;
                C.s(kAc) = ac;
                C.s(kNgd2) = ac * ac * gg;
            } else if (alive) {
                for (int q = u - 4; 2 * q < n; q += U - 4) {
                    const float2 z = normal_pair(T, (uint32_t)s, kPhaseLm, (uint32_t)A.k0 + (uint32_t)kk, q);
                    C.nz(2 * q) = z.x;
                    C.nz(2 * q + 1) = z.y;
                }
            }
            __syncthreads();

            // each joint's LM step, Gauss-Newton step and gradient
            for (int j = u; j < n; j += U) {
                float a = 0.0f, dgn = 0.0f, g = 0.0f;
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    const float v = C.jc(r, j);
                    a = fmaf(v, C.s(kY + r), a);
                    dgn = fmaf(v, C.s(kY2 + r), dgn);
                    g = fmaf(v, C.s(kB + r), g);
                }
                C.st(j) = clampf(__fdividef(a, C.dd(j)), -Rt, Rt);  // trust region
                C.dgn(j) = dgn;
                C.g(j) = g;
            }
            __syncthreads();

            // the dogleg's weights; the single coordinate; of long chains, the sines and cosines of the line
            // search beside them (24 joints: 133 -> 129 us; of short ones all trials' take two passes of the next stage)
            if (warp == 0) {
                const float ac = C.s(kAc);
                float ngn2 = 0.0f, qa = 0.0f, qb = 0.0f;
#pragma unroll 4
                for (int j = 0; j < n; ++j) dogleg_terms(C.dgn(j), C.g(j), ac, ngn2, qa, qb);
                float wgn, wgd;
                dogleg_weights(ngn2, C.s(kNgd2), qa, qb, ac, Rt, wgn, wgd);
                C.s(kWgn) = wgn;
                C.s(kWgd) = wgd;
            } else if (warp == 1) {
                int is = 0;
                float gbest = -1.0f;
#pragma unroll 4
                for (int j = 0; j < n; ++j) {
                    const float g = fabsf(C.g(j));
                    if (g > gbest) {
                        gbest = g;
                        is = j;
                    }
                }
                float cn = 0.0f, col[6];
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    col[r] = C.jc(r, is);
                    cn = fmaf(col[r], col[r], cn);
                }
                C.si(kSj) = is;
                C.s(kSstep) = cn > 0.0f ? clampf(__fdividef(C.g(is), cn), -Rt, Rt) : 0.0f;
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    C.s(kSv + r) = __fdividef(col[r], C.s(kW + r));
                    C.s(kSz + r) = __fdividef(col[3 + r], C.s(kW + 3 + r));
                }
            } else if (!N) {
                for (int w = u - 4; w < (nt - 1) * n; w += U - 4) trial_sincos(w / n, w % n);
            }
            __syncthreads();

            // sines and cosines of the trials' angles
            for (int w = (N ? 0 : (nt - 1) * n) + u; w < nt * n; w += U) trial_sincos(w / n, w % n);
            __syncthreads();

            // the trials' kinematics rows
            for (int w = u; w < 3 * nt; w += U) lmc_fk_row<N, false>(C, R, n, 1 + w / 3, w % 3);
            __syncthreads();

            // the trials' costs (first the warps with kinematics trials, then those with the single
            // coordinate's); bit i of the mask: trial i lowered the cost, in the order of Alg. 4
            {
                const int kw = (nt + 1) / 2, items = kw + (lsA + 2) / 2;  // warps' worth of either
                for (int w = warp; w < items; w += W) {
                    const bool kin = w < kw;
                    const int i = 2 * (kin ? w : w - kw) + half;
                    if (i >= (kin ? nt : lsA + 1)) continue;
                    const float w6[6] = {C.s(kW), C.s(kW + 1), C.s(kW + 2), C.s(kW + 3), C.s(kW + 4), C.s(kW + 5)};
                    float cost;
                    if (kin) {
                        const Frame E = lmc_flange(C, R, 1 + i);
                        const V3 om = quat_log(quat_error(T, quat_from_frame(E)));
                        cost = weighted_cost(w6, v3(T.p[0], T.p[1], T.p[2]) - E.p, om);
                    } else {
                        const int j = C.si(kSj);
                        const float th0 = C.th(j);
                        const float thj = clampf(fmaf(alphas[i], C.s(kSstep), th0), R.lim[j].x, R.lim[j].y);
                        cost = coord_cost_at(w6, v3(C.s(kSz), C.s(kSz + 1), C.s(kSz + 2)),
                                             v3(C.s(kSv), C.s(kSv + 1), C.s(kSv + 2)), v3(C.s(kE), C.s(kE + 1), C.s(kE + 2)),
                                             Q4{C.s(kQ), v3(C.s(kQ + 1), C.s(kQ + 2), C.s(kQ + 3))}, thj - th0);
                    }
                    if (cost < C.s(kCost)) atomicOr(&C.si(kMask), 1 << (kin ? i : nt + i));
                }
            }
            __syncthreads();

            // the first success in the order of Alg. 4, else the perturbation
            if (alive) {
                const int pick = __ffs(C.si(kMask)) - 1;
                for (int j = u; j < n; j += U) {
                    const float lo = R.lim[j].x, hi = R.lim[j].y;
                    float th = C.th(j);
                    if (pick < 0) {
                        th = clampf(fmaf(P.lm_sigma, C.nz(j), th), lo, hi);
                    } else if (pick < nt) {
                        const float dir = pick <= lsA ? C.st(j) : fmaf(C.s(kWgn), C.dgn(j), C.s(kWgd) * C.g(j));
                        th = clampf(fmaf(pick <= lsA ? alphas[pick] : 1.0f, dir, th), lo, hi);
                    } else if (j == C.si(kSj)) {
                        th = clampf(fmaf(alphas[pick - nt], C.s(kSstep), th), lo, hi);
                    }
                    C.th(j) = th;
                    C.cs(0, j) = sincos_of(R, j, th);
                }
                if (u == U - 2) {  // the passes and trials the sequential method evaluates
                    ++n_it;
                    n_fk += pick >= 0 && pick < nt ? pick + 1 : nt;
                    if (pick < 0 || pick >= nt) n_sc += pick < 0 ? lsA + 1 : pick - nt + 1;
                }
            }
            __syncthreads();
            if (!LIST && kk + 1 == A.hand_at) {  // the candidates that are left are packed afresh by the next launch
                if (u == 0 && alive) {
                    const int at = atomicAdd(A.n_list, 1);
                    A.list[at] = (int32_t)c;
                    A.list_k[at] = kk + 1;
                }
                break;
            }
        }
        if (mine)
            for (int j = u; j < n; j += U) A.th[j * A.ld + c] = C.th(j);
    }
    if (A.cnt) {
        n_it = warp_sum(n_it);
        n_fk = warp_sum(n_fk);
        n_sc = warp_sum(n_sc);
        if (lane == 0 && (warp == 0 || warp == W - 1)) {
            atomicAdd(&A.cnt->v[1], n_it);
            atomicAdd(&A.cnt->v[2], n_fk);
            atomicAdd(&A.cnt->v[7], n_sc);
        }
    }
}

template <bool RED, int N, bool LIST>
void launch_lm_coop_n(const LmArgs& A, int warps, cudaStream_t st) {
    const size_t smem = robots_smem_bytes(A.rs.n) + coop_lm_bytes(A.rs.n_max, A.P.lm_A);
    static SmemLimit lim;
    allow_dyn_smem(k_lm_coop<RED, N, LIST>, lim,
                   robots_smem_bytes(kMaxLaunchRobots) + coop_lm_bytes(N ? N : kMaxDof, kCoopMaxA));
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lm_coop<RED, N, LIST>, 32 * warps, smem);
    const int g = (int)std::min<int64_t>((A.C + kCoopCands - 1) / kCoopCands, (int64_t)sm_count() * std::max(per_sm, 1));
    // Set up while the kernel before still runs -- but where CTAs outnumber the SMs, they are then placed
    // among that kernel's, unevenly, which the long iterations of long chains show: 24 joints, 5000 / 8000 /
    // 10000 candidates, a solve 453 / 494 / 586 us so, 428 / 469 / 549 launched after it; 18 joints 387 / 419 / 484
    // and 369 / 402 / 479; 12 joints 297 / 318 / 358 and 285 / 320 / 361; 7 joints 223 and 225 us at 7000.
    if (g > sm_count() && A.rs.n_max > 8) k_lm_coop<RED, N, LIST><<<g, 32 * warps, smem, st>>>(A);
    else launch_next<LmArgs>(k_lm_coop<RED, N, LIST>, g, 32 * warps, smem, st, A);
}

template <bool RED, bool LIST>
void launch_lm_coop(const LmArgs& A, int warps, cudaStream_t st) {
    const int n = A.rs.n == 1 ? A.rs.n_max : 0;
    if (n == 6) launch_lm_coop_n<RED, 6, LIST>(A, warps, st);
    else if (n == 7) launch_lm_coop_n<RED, 7, LIST>(A, warps, st);
    else launch_lm_coop_n<RED, 0, LIST>(A, warps, st);
}

template <bool TRACE, int WARPS, bool RED, bool HAND>
void launch_lm_t(const LmArgs& A, cudaStream_t st) {
    const size_t smem = robots_smem_bytes(A.rs.n) +
                        sizeof(float) * ((size_t)lm_warp_words(A.rs.n_max, A.P.lm_A) * WARPS + lm_cta_words<WARPS>());
    static SmemLimit lim;
    allow_dyn_smem(k_lm<TRACE, WARPS, RED, HAND>, lim,
                   robots_smem_bytes(kMaxLaunchRobots) +
                       sizeof(float) * ((size_t)lm_warp_words(kMaxDof, kMaxLsDepth) * WARPS + lm_cta_words<WARPS>()));
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lm<TRACE, WARPS, RED, HAND>, WARPS * 32, smem);
    if (per_sm < 1) per_sm = 1;
    const int64_t want = (A.C + 32 * WARPS - 1) / (32 * WARPS);
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sm_count() * per_sm));
    k_lm<TRACE, WARPS, RED, HAND><<<g, WARPS * 32, smem, st>>>(A);
}

// Warps per CTA of a launch of one lane per candidate for which `asked` are set
int lm_warps_for(const LmArgs& A, int asked) {
    // fewer warps per CTA when the requested count's state does not fit in shared memory
    int optin = 0;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, current_device());
    const size_t per_warp = sizeof(float) * (size_t)lm_warp_words(A.rs.n_max, A.P.lm_A);
    int warps = asked == 2 || asked == 4 || asked == 8 ? asked : kLmWarps;
    // a batch too small to give every SM a CTA of two warps (a single target, say): two-warp CTAs,
    // spread over more SMs with shorter lock-step stages (latency, not throughput, is at stake)
    if (A.C <= (int64_t)sm_count() * 64) warps = 2;
    // (the CTA lists: 65 words per warp and two; 256 bytes kept for the kernel's static arrays)
    auto bytes = [&](int w) { return robots_smem_bytes(A.rs.n) + (per_warp + sizeof(float) * 65) * w + 8 + 256; };
    while (warps > 2 && bytes(warps) > (size_t)optin) warps /= 2;
    // or where that lets a fifth more warps reside, or as many of no more than eight (which then wait at
    // barriers of their own).  us with eight warps -> so, 250 targets x 1000 seeds: 12 joints (one CTA of 8
    // warps, three of 4) 864 -> 707, 16 joints (8, 5 of 2) 853 -> 787, 18 joints (8, 4 of 2) 836 -> 774, 24
    // joints (4, 3 of 2) 1202 -> 905; 7 and 9 joints keep two CTAs of 8 (512 against 565 with 2).
    int sm_bytes = 0;
    cudaDeviceGetAttribute(&sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, current_device());
    auto resident = [&](int w) { return std::min(16, (int)((size_t)sm_bytes / (bytes(w) + 1024)) * w); };
    for (int w = warps / 2; w >= 2; w /= 2) {
        const int r = resident(w), r0 = resident(warps);
        if (5 * r >= 6 * r0 || (r >= r0 && r0 <= 8)) warps = w;
    }
    return warps;
}

template <bool TRACE, bool RED, bool HAND>
void launch_lm_w(const LmArgs& A, cudaStream_t st) {
    const int warps = lm_warps_for(A, A.warps);
    if (warps == 2) launch_lm_t<TRACE, 2, RED, HAND>(A, st);
    else if (warps == 4) launch_lm_t<TRACE, 4, RED, HAND>(A, st);
    else launch_lm_t<TRACE, 8, RED, HAND>(A, st);
}

constexpr int kCoopShort = 3;  // joints of a chain that one lane polishes quickly
// Whether a launch goes, in whole or in its first iterations, to the spread kernel, and whether it leaves
// candidates to a second launch (both explained in launch_lm)
struct LmRoute {
    bool spread, hand;
};
LmRoute lm_route(const LmArgs& A, bool trace) {
    const int64_t sms = sm_count();
    const int64_t most = sms * (A.list ? 216 : (A.rs.n_max == 1 ? 2 : 4) * kCoopCands);
    if (trace || A.P.lm_A > kCoopMaxA || A.C > most) return {false, false};
    const bool hand = A.list && A.C > sms * 2 * kCoopCands;
    return {!hand || (A.C <= sms * 80 && A.rs.n_max > kCoopShort), hand};
}

}  // namespace

int lm_warps_used(const LmArgs& A, int asked) {
    if (A.C <= 0 || lm_route(A, false).spread) return 0;
    return lm_warps_for(A, asked);
}

int launch_lm(const LmArgs& B, bool trace, cudaStream_t st) {
    if (B.C <= 0) return 0;
    LmArgs A = B;
    A.hand_at = A.hand_lim = 0;
    const bool plain = A.in_limits && A.rs.plain;
    const int64_t sms = sm_count();
    auto lanes = [&]() {
        const bool hand = A.hand_at > 0;
        if (trace) launch_lm_w<true, true, false>(A, st);
        else if (hand && plain) launch_lm_w<false, false, true>(A, st);
        else if (hand) launch_lm_w<false, true, true>(A, st);
        else if (plain) launch_lm_w<false, false, false>(A, st);
        else launch_lm_w<false, true, false>(A, st);
    };
    // Up to 64 candidates per SM (two resident CTAs of 16 on every SM, twice) the spread kernel's
    // shorter iterations win; past that its extra work does.  Phase time of the polish, spread /
    // one lane per candidate, us (7, 20, 24 joints): 1000 candidates 70 / 172, 115 / 328, 129 / 360;
    // 4000: 84 / 200, 164 / 346, 178 / 356; 8000: 166 / 221, 322 / 346, 338 / 356; 16000: 311 / 240,
    // 594 / 395, 616 / 363 (the last two with loads not yet ahead of the stores, 3 to 6% of its time).  A
    // single joint leaves nothing to spread: up to 32 per SM (9000 candidates 151 / 95, 4800: 84 / 97; two
    // joints 161 / 176).  Twelve warps while a CTA has its SM to itself (8: 76, 139, 150), eight (two CTAs
    // per SM) beyond.
    //
    // Where the caller gives a list, batches of up to 216 candidates per SM leave the candidates that
    // need more than a few iterations to a second launch of the spread kernel, packed afresh: most candidates
    // converge in those, and the rest (a fifth of Panda's run to the cap of 20) fit it.  Up to 80 per SM four
    // iterations of the spread kernel; beyond, and for a chain of up to three joints, six of one lane per
    // candidate, and on until no more than 64 per SM are unfinished: a chain that rarely reaches its targets
    // may never get there, and then one launch does it all.  One launch / two, us, the quarter of the seeds
    // duplicated: 7 joints 8000: 252 / 106, 16000: 250 / 141, 32000: 248 / 207; 12 joints 285 / 149, 291 / 180,
    // 293 / 252; 20 joints 381 / 203, 389 / 235, 406 / 373; 6 joints of which a third run to the cap 270 / 156,
    // 293 / 266, 283 / 283.  Every seed polished (a ratio of 1): 7 joints 305 / 160, 324 / 270, 338 / 336; 6 joints
    // 289 / 158, 328 / 338, 330 / 340.  (Handing over at six iterations whatever was left, and only in CTAs
    // with a lane that had asked the queue in vain, the last two took 534 and 503.)  48000 no gain.
    const auto [spread, hand] = lm_route(A, trace);
    if (!spread && !hand) {
        lanes();
        return 1;
    }
    if (hand) {
        A.hand_at = spread ? 4 : 6;
        A.hand_lim = (int32_t)(sms * 4 * kCoopCands);
    }
    if (spread) {
        const int warps = A.C <= sms * kCoopCands ? 12 : 8;
        if (plain) launch_lm_coop<false, false>(A, warps, st);
        else launch_lm_coop<true, false>(A, warps, st);
    } else {
        lanes();
    }
    if (!hand) return 1;
    A.hand_at = 0;
    if (plain) launch_lm_coop<false, true>(A, 8, st);
    else launch_lm_coop<true, true>(A, 8, st);
    return 2;
}

}  // namespace hjcd
