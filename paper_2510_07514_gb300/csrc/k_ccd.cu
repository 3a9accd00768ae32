// k_ccd.cu -- seed sampling (Alg. 3) and PO-CCD iterations (Sec. IV,
// Alg. 3), one candidate per thread.
//
// Per iteration one forward-kinematics pass gives every joint's origin and
// axis.  The 2n trial updates are evaluated in O(1) each: rotating joint j by
// d moves the end effector about the axis (Rodrigues) and composes the error
// quaternion with the joint rotation, so both parts of each trial's task
// residual follow from the projected vectors of Eq. vec_proj and one half-angle
// sine/cosine.  The proposed theta_hat changes at most two joints; its
// residual is the composition of the two joint rotations applied to the
// current end-effector pose (the more distal joint first), so acceptance
// needs no second kinematics pass.
//
// Each thread keeps its joint vector and the joint origins/axes of the last
// kinematics pass in a column of shared memory ([quantity][thread], so the
// accesses of a warp hit 32 different banks); joint loops are not unrolled,
// which keeps the kernel small enough for the instruction cache at any n.
// The robot tables of the launch sit in shared memory in front of the
// columns; each candidate uses its target's robot.
#include <algorithm>

#include "hjcd_internal.cuh"

namespace hjcd {

namespace {

// CTA size of the seed-sampling kernel, and of the PO-CCD kernel when the launch names none of
// 64, 128, 256 (a context starts at 64 candidates per CTA: hjcd_set_launch_config)
constexpr int kCcdThreads = 128;

// shared-memory column of a thread in a CTA of TH threads, laid out [quantity][thread] (a warp's
// accesses hit 32 different banks): per joint j the pairs (px, py), (pz, theta_j), (zx, zy),
// (zz, -) of joint j's frame after its kinematics step, 8 n words in all; each pair moves as one
// 64-bit access
template <int TH, bool PACK = false>
struct ColT {
    static constexpr int kWords = 8;  // per joint
    float2* base;  // this thread's first pair
    __device__ __forceinline__ ColT(float2* b, int) : base(b) {}
    __device__ __forceinline__ ColT lane(int d) const { return ColT(base + d, 0); }  // the column d threads on
    __device__ __forceinline__ float& zz(int j) const { return base[(4 * j + 3) * TH].x; }
    __device__ __forceinline__ float2& a(int j) const { return base[4 * j * TH]; }
    __device__ __forceinline__ float2& b(int j) const { return base[(4 * j + 1) * TH]; }
    __device__ __forceinline__ float2& c(int j) const { return base[(4 * j + 2) * TH]; }
    __device__ __forceinline__ float& th(int j) const { return b(j).y; }
    // joint j's origin and axis
    __device__ __forceinline__ void frame(int j, V3& p, V3& z) const {
        const float2 pa = a(j), pb = b(j), za = c(j);
        p = v3(pa.x, pa.y, pb.x);
        z = v3(za.x, za.y, zz(j));
    }
    __device__ __forceinline__ void set_frame(int j, const Frame& F, float theta) const {
        a(j) = make_float2(F.p.x, F.p.y);
        b(j) = make_float2(F.p.z, theta);
        c(j) = make_float2(F.c2.x, F.c2.y);
        zz(j) = F.c2.z;
    }
};
// The same with zz in words of its own after all the pairs, 7 n words in all: one address more to
// keep (2.5% of a Panda launch), but room for more resident CTAs of long chains.
template <int TH>
struct ColT<TH, true> {
    static constexpr int kWords = 7;
    float2* base;  // this thread's first pair
    float* zb;     // this thread's first zz
    __device__ __forceinline__ ColT(float2* b, float* z) : base(b), zb(z) {}
    // the column of a CTA whose thread 0 has its first pair at b - threadIdx.x, for chains of n joints
    __device__ __forceinline__ ColT(float2* b, int n)
        : base(b), zb(reinterpret_cast<float*>(b - threadIdx.x + 3 * n * TH) + threadIdx.x) {}
    __device__ __forceinline__ ColT lane(int d) const { return ColT(base + d, zb + d); }
    __device__ __forceinline__ float2& a(int j) const { return base[3 * j * TH]; }
    __device__ __forceinline__ float2& b(int j) const { return base[(3 * j + 1) * TH]; }
    __device__ __forceinline__ float2& c(int j) const { return base[(3 * j + 2) * TH]; }
    __device__ __forceinline__ float& zz(int j) const { return zb[j * TH]; }
    __device__ __forceinline__ float& th(int j) const { return b(j).y; }
    __device__ __forceinline__ void frame(int j, V3& p, V3& z) const {
        const float2 pa = a(j), pb = b(j), za = c(j);
        p = v3(pa.x, pa.y, pb.x);
        z = v3(za.x, za.y, zz(j));
    }
    __device__ __forceinline__ void set_frame(int j, const Frame& F, float theta) const {
        a(j) = make_float2(F.p.x, F.p.y);
        b(j) = make_float2(F.p.z, theta);
        c(j) = make_float2(F.c2.x, F.c2.y);
        zz(j) = F.c2.z;
    }
};

// the joint vector alone, theta[n] (the seed-sampling kernel)
template <int TH>
struct ThetaCol {
    float* base;
    __device__ __forceinline__ float& th(int j) const { return base[j * TH]; }
};

template <class Col>
__device__ __forceinline__ void sample_seed(const RobotParams& R, const TargetDesc& T, uint32_t s, const Col& col) {
#pragma unroll 1
    for (int b = 0; 4 * b < R.n; ++b) {
        const uint4 w = rnd_block(T, s, kPhaseSeed, 0, (uint32_t)b);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int j = 4 * b + q;
            if (j < R.n) col.th(j) = fmaf(u01(word(w, q)), R.lim[j].y - R.lim[j].x, R.lim[j].x);
        }
    }
}

// Both trials of joint j (origin pj, unit axis z, angle thj in [lo, hi]) against the end
// effector at Ep and the error quaternion qerr (angle phi): the position step d of Eq.
// theta_proj and the orientation step dq of Eq. ori_update, each clamped to the limits, with the
// task residual each leaves (position error squared, orientation angle) and its score.  Rotating
// joint j by x moves the end effector to pj + uz z + cos x up + sin x (z x up) and turns the error
// quaternion into qerr [cos(x/2), -sin(x/2) z].
struct CcdTrials {
    float d, rp2, op, sp;   // position trial
    float dq, pq2, rq, so;  // orientation trial
};

// The two trials of a joint share their arithmetic once the steps are known, so from there on
// they run as pairs (.x the position trial, .y the orientation trial) on the packed FP32
// instructions of sm_100+ (two IEEE operations per instruction, each half rounded on its own), in
// the order of the scalar helpers (dot, fma3, quat_angle); where the compiler contracts the scalar
// helpers differently the results differ by an ulp.

// p(t^2) of atan01 for both halves (atan t = t p(t^2), t in [0, 1])
__device__ __forceinline__ float2 atan_poly2(float2 t) {
    const float2 s = mul2(t, t);
    float2 p = fma2(bc2(-4.166443301e-03f), s, bc2(2.232482877e-02f));
    p = fma2(p, s, bc2(-5.666722692e-02f));
    p = fma2(p, s, bc2(9.704074739e-02f));
    p = fma2(p, s, bc2(-1.393516270e-01f));
    p = fma2(p, s, bc2(1.995220255e-01f));
    p = fma2(p, s, bc2(-3.333036250e-01f));
    return fma2(p, s, bc2(9.999994549e-01f));
}

// quat_angle of both halves: 2 atan2(sqrt(vv), |w|); the reflection about pi/4 takes the last
// product into one rounding, 2 (pi/2 - t p) = pi - 2 t p
__device__ __forceinline__ float2 quat_angle2(float2 w, float2 vv) {
    const float yx = sqrt_approx(vv.x), yy = sqrt_approx(vv.y);
    const float xx = fabsf(w.x), xy = fabsf(w.y);
    const float mxx = fmaxf(fmaxf(xx, yx), 1e-30f), mnx = fminf(xx, yx);
    const float mxy = fmaxf(fmaxf(xy, yy), 1e-30f), mny = fminf(xy, yy);
    const float2 t = make_float2(__fdividef(mnx, mxx), __fdividef(mny, mxy));
    const float2 p = atan_poly2(t);
    const float2 a = mul2(mul2(bc2(2.0f), t), p);                                      // 2 t p
    const float2 r = fma2(mul2(bc2(-2.0f), t), p, bc2(2.0f * 1.57079632679489662f));  // pi - 2 t p
    return make_float2(yx > xx ? r.x : a.x, yy > xy ? r.y : a.y);
}

// Both residual parts of a trial in closed form.  With r = p_t - p_ee, split along z and the
// plane normal to it, the rotated end effector leaves the axial part r.z and, in the plane,
// v_p - cos x u_p - sin x (z x u_p); u_p and z x u_p are orthogonal with equal norms, so the
// in-plane part squared is ((u_p.v_p - cos x |u_p|^2)^2 + ((z x u_p).v_p - sin x |u_p|^2)^2) / |u_p|^2.
// The error quaternion's vector part, split the same way into a_z z + q_perp, becomes
// (cos a_z - sin w) z + cos q_perp - sin (q_perp x z), of squared norm (cos a_z - sin w)^2 + |q_perp|^2
// (cos, sin of x/2).  The only differences are those that form the residual's own components, as
// in the direct evaluation, and the squares are summed, so the closed form is as accurate (a float32
// emulation against the float64 method agrees to 2e-7 on Panda).
__device__ __forceinline__ CcdTrials ccd_joint_trials(const V3 pj, const V3 z, float thj, float lo, float hi,
                                                      const V3 Ep, const V3 pt, const Q4 qerr, float nqw,
                                                      float dphi, float pe2, float inv_p2, float inv_o2) {
    CcdTrials o;
    const V3 u = Ep - pj;
    const V3 v = pt - pj;
    const float uz = dot(u, z), vz = dot(v, z);
    const V3 up = fma3(-uz, z, u);
    const V3 vp = fma3(-vz, z, v);
    const float nup2 = dot(up, up), nvp2 = dot(vp, vp);
    const float nu2 = fmaf(uz, uz, nup2), nv2 = fmaf(vz, vz, nvp2);
    const V3 zxu = cross(z, up);
    const float ez = vz - uz;
    const float az = dot(qerr.v, z);
    const V3 qp = fma3(-az, z, qerr.v);
    const float qp2 = dot(qp, qp);

    // Eq. theta_proj, signed about the axis: atan2(z.(up x vp), up.vp) = atan2(zxu.vp, up.vp)
    const float cs = dot(up, vp), sn = dot(zxu, vp);
    const bool deg = nu2 < 1e-24f || nv2 < 1e-24f || nup2 <= pe2 * nu2 || nvp2 <= pe2 * nv2;
    const float d = deg ? 0.0f : atan2_all(sn, cs);
    // Eq. ori_update: delta(k) sgn(a.z) phi
    const float dq = (az > 0.0f) ? dphi : ((az < 0.0f) ? -dphi : 0.0f);

    // both steps clamped to the limits
    float2 st = add2(bc2(thj), make_float2(d, dq));
    st = make_float2(clampf(st.x, lo, hi), clampf(st.y, lo, hi));
    st = add2(st, bc2(-thj));
    o.d = st.x;
    o.dq = st.y;
    const float2 hs = mul2(bc2(0.5f), st);
    float2 sh, ch;
    __sincosf(hs.x, &sh.x, &ch.x);
    __sincosf(hs.y, &sh.y, &ch.y);
    const float2 m2sh = mul2(bc2(-2.0f), sh);
    const float2 msn = mul2(m2sh, ch);             // -sin(step)
    const float2 cst = fma2(m2sh, sh, bc2(1.0f));  // cos(step)
    // position residual of each trial.  Where u_p is at the rounding level of u (the end effector
    // on the axis, as the flange on a last joint's axis) its direction is noise that leaves the
    // plane, and the quotient would drop part of v_p; there the expanded form
    // |v_p|^2 + |u_p|^2 - 2 (cos u_p.v_p + sin (z x u_p).v_p), which cannot cancel while
    // |u_p| << |u|, is taken instead.
    float2 r2;
    if (nup2 <= 1e-6f * nu2) {
        r2 = fma2(bc2(2.0f), fma2(msn, bc2(sn), mul2(cst, bc2(-cs))), bc2(fmaf(ez, ez, nvp2 + nup2)));
    } else {
        const float2 ex = fma2(cst, bc2(-nup2), bc2(cs));
        const float2 ey = fma2(msn, bc2(nup2), bc2(sn));
        r2 = fma2(fma2(ex, ex, mul2(ey, ey)), bc2(__fdividef(1.0f, nup2)), bc2(ez * ez));
    }
    // error quaternion of each trial: qerr [cos, -sin z]
    const float2 w2 = fma2(bc2(qerr.w), ch, mul2(sh, bc2(az)));
    const float2 tz = fma2(ch, bc2(az), mul2(sh, bc2(nqw)));
    const float2 vv = fma2(tz, tz, bc2(qp2));
    const float2 ang = quat_angle2(w2, vv);
    const float2 sc = fma2(r2, bc2(inv_p2), mul2(mul2(ang, ang), bc2(inv_o2)));
    o.rp2 = r2.x;
    o.op = ang.x;
    o.sp = sc.x;
    o.pq2 = r2.y;
    o.rq = ang.y;
    o.so = sc.y;
    return o;
}

// One iteration of a candidate: kinematics with frames into the column, the
// residual (ep2 = |e_p|^2, eo = |omega|), the break test (kk > 0) and the cap,
// then the update of Alg. 3 (or Alg. 1 with cd_variant = 1) of the joint
// vector in the column.  Returns 1 when the candidate has converged, 2 at the
// cap (no update in either case), 0 after an update.
constexpr int kSlotWords = 8;  // per-thread shared-memory slot of the cooperative perturbation

// w / nb = (w * kDivMagic[nb]) >> 16 exactly for 1 <= nb <= 12 and 0 <= w < 32 nb (the normal
// pairs of a joint vector, at most 12, times the lanes of a warp); kDivMagic[nb] = ceil(2^16 / nb)
__constant__ uint32_t kDivMagic[13] = {0, 65536, 32768, 21846, 16384, 13108, 10923, 9363, 8192, 7282, 6554, 5958, 5462};
static_assert((kMaxDof + 1) / 2 <= 12, "the normal pairs of a joint vector index kDivMagic");

template <bool TRACE, int TH, bool RED = true, bool PACK = false>
__device__ __forceinline__ int ccd_step(const RobotParams* rob, const RobotParams& R, const TargetDesc& T,
                                        const hjcd_params& P, const ColT<TH, PACK>& col, uint32_t* slots, const CcdArgs& A,
                                        int64_t c, uint32_t s, int kk, int cap, float delta_k, const V3 pt, float pe2,
                                        float one_m_tie, float inv_p2, float inv_o2, float& ep2, float& eo) {
    const int n = R.n;
    // kinematics with frames
    Frame F = frame_identity();
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        const float thj = col.th(j);
        fk_step<RED>(R, j, thj, F);
        col.set_frame(j, F, thj);
    }
    const Frame E = fk_flange(R, F);
    const Q4 qerr = quat_error(T, quat_from_frame(E));
    const V3 e = pt - E.p;
    ep2 = dot(e, e);
    eo = quat_angle(qerr.w, dot(qerr.v, qerr.v));
    // Alg. 3 coarse break, checked after each update (Alg. 1: the position part only)
    if (kk > 0 && ep2 < P.cd_eps_pos2 && (P.cd_variant == 1 || eo * eo < P.cd_eps_ori2)) return 1;
    if (kk == cap) return 2;
    const int k = A.k0 + kk;
    const float ep0 = sqrt_approx(ep2);

    if (P.cd_variant == 1) {
        // Alg. 1: joints from the last to the first, each rotated at once by its Eq. theta_proj
        // step; rotating joint j leaves the frames of joints <= j in place and moves the end
        // effector about joint j's axis
        V3 x = E.p;
#pragma unroll 1
        for (int j = n - 1; j >= 0; --j) {
            V3 pj, z;
            col.frame(j, pj, z);
            const float thj = col.th(j);
            const V3 u = x - pj, v = pt - pj;
            const float uz = dot(u, z), vz = dot(v, z);
            const V3 up = fma3(-uz, z, u), vp = fma3(-vz, z, v);
            const float nu2 = dot(u, u), nv2 = dot(v, v), nup2 = dot(up, up), nvp2 = dot(vp, vp);
            const V3 zxu = cross(z, up);
            const bool deg = nu2 < 1e-24f || nv2 < 1e-24f || nup2 <= pe2 * nu2 || nvp2 <= pe2 * nv2;
            float d = deg ? 0.0f : atan2_all(dot(zxu, vp), dot(up, vp));
            d = clampf(thj + d, R.lim[j].x, R.lim[j].y) - thj;
            float sd, cd;
            sincos_red(d, &sd, &cd);  // |d| may exceed pi
            x = pj + fma3(uz, z, fma3(cd, up, sd * zxu));
            col.th(j) = thj + d;
            if (TRACE && kk == 0 && A.tr.dp) A.tr.dp[j * A.ld + c] = d;
        }
        return 0;
    }

    // one position and one orientation proposal per joint, the
    // task residual each leaves, and the greedy choice by its score
    // (|e_p|/eps_pos)^2 + (|omega|/eps_ori)^2; a later joint replaces the
    // choice only when its score is lower by more than the fraction cd_tie
    float best_p = __int_as_float(0x7f800000), dP = 0.0f, best_o = __int_as_float(0x7f800000), dO = 0.0f;
    int jp = 0, jo = 0;
    const float dphi = delta_k * eo, nqw = -qerr.w;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        const float2 pa = col.a(j), pb = col.b(j), za = col.c(j);
        const V3 pj = v3(pa.x, pa.y, pb.x);
        const V3 z = v3(za.x, za.y, col.zz(j));
        const CcdTrials tr =
            ccd_joint_trials(pj, z, pb.y, R.lim[j].x, R.lim[j].y, E.p, pt, qerr, nqw, dphi, pe2, inv_p2, inv_o2);
        if (tr.sp < best_p * one_m_tie) {  // joint 0 against +inf
            best_p = tr.sp;
            jp = j;
            dP = tr.d;
        }
        if (tr.so < best_o * one_m_tie) {
            best_o = tr.so;
            jo = j;
            dO = tr.dq;
        }
        if (TRACE && kk == 0) {
            if (A.tr.dp) A.tr.dp[j * A.ld + c] = tr.d;
            if (A.tr.rp) A.tr.rp[j * A.ld + c] = sqrtf(tr.rp2);
            if (A.tr.op) A.tr.op[j * A.ld + c] = tr.op;
            if (A.tr.dq) A.tr.dq[j * A.ld + c] = tr.dq;
            if (A.tr.pq) A.tr.pq[j * A.ld + c] = sqrtf(tr.pq2);
            if (A.tr.rq) A.tr.rq[j * A.ld + c] = tr.rq;
        }
    }

    // apply both; on the same joint the larger step
    float aP = dP, aO = dO;
    if (jp == jo) {
        if (fabsf(dP) >= fabsf(dO)) aO = 0.0f;
        else aP = 0.0f;
    }
    // residual at theta_hat: the distal joint's rotation first, then the proximal one
    // (the chosen joints' origins and axes are still in the shared-memory column)
    const bool p_hi = jp > jo;
    V3 Pa, Za, Pb, Zb;
    col.frame(p_hi ? jp : jo, Pa, Za);  // the distal joint
    col.frame(p_hi ? jo : jp, Pb, Zb);
    const float da = p_hi ? aP : aO, db = p_hi ? aO : aP;
    float sa_, ca_, sb_, cb_;
    __sincosf(0.5f * da, &sa_, &ca_);
    __sincosf(0.5f * db, &sb_, &cb_);
    V3 x = Pa + rotate_half(Za, sa_, ca_, E.p - Pa);
    x = Pb + rotate_half(Zb, sb_, cb_, x - Pb);
    Q4 q1 = qmul(qerr, Q4{ca_, (-sa_) * Za});
    q1 = qmul(q1, Q4{cb_, (-sb_) * Zb});
    const V3 e1 = pt - x;
    const float ep1 = sqrt_approx(dot(e1, e1));
    const float eo1 = quat_angle(q1.w, dot(q1.v, q1.v));
    // acceptance (reading: an improvement above gamma in position or in orientation)
    const bool acc = (ep0 - ep1 > P.cd_gamma_pos) || (eo - eo1 > P.cd_gamma_ori);

    if (TRACE && kk == 0) {
        if (A.tr.jp) A.tr.jp[c] = jp;
        if (A.tr.jo) A.tr.jo[c] = jo;
        if (A.tr.accepted) A.tr.accepted[c] = acc ? 1 : 0;
        if (A.tr.th_hat) {
#pragma unroll 1
            for (int j = 0; j < n; ++j)
                A.tr.th_hat[j * A.ld + c] = col.th(j) + (j == jp ? aP : 0.0f) + (j == jo ? aO : 0.0f);
        }
    }
    if (acc) {  // clamped again: theta + (clamp(theta + d) - theta) can round an ulp past a limit
        col.th(jp) = clampf(col.th(jp) + aP, R.lim[jp].x, R.lim[jp].y);
        col.th(jo) = clampf(col.th(jo) + aO, R.lim[jo].x, R.lim[jo].y);
    }
    // rejection: theta + N(0, sigma^2 I), kept inside the limits.  Few lanes reject at a time,
    // so the lanes executing here together share the work: each rejected lane publishes its
    // stream (key, target index, candidate, iteration) and robot, and the (lane, normal pair)
    // items are spread over all of them; every joint column lives in shared memory.
    const unsigned am = __activemask();
    const unsigned rej = __ballot_sync(am, !acc);
    if (rej) {
        const int lane = threadIdx.x & 31;
        uint32_t* const slot = slots + (threadIdx.x & ~31u) * kSlotWords;  // this warp's slots
        if (!acc) {
            uint32_t* me = slot + lane * kSlotWords;
            me[0] = T.key[0];
            me[1] = T.key[1];
            me[2] = (uint32_t)T.t_local;
            me[3] = s;
            me[4] = (uint32_t)k;
            me[5] = (uint32_t)T.robot;
        }
        const int NB = (int)__reduce_max_sync(am, acc ? 0u : (uint32_t)((n + 1) / 2));
        __syncwarp(am);
        const int items = __popc(rej) * NB, step = __popc(am);
        const uint32_t magic = kDivMagic[NB];
        for (int w = __popc(am & ((1u << lane) - 1u)); w < items; w += step) {
            const int r = (int)(((uint32_t)w * magic) >> 16), b = w - r * NB;
            const int sl = __fns(rej, 0, r + 1);
            const uint32_t* q = slot + sl * kSlotWords;
            const RobotParams& Rs = rob[q[5]];
            if (2 * b >= Rs.n) continue;
            TargetDesc Tq;
            Tq.key[0] = q[0];
            Tq.key[1] = q[1];
            Tq.t_local = (int32_t)q[2];
            const float2 z = normal_pair(Tq, q[3], kPhaseCd, q[4], b);
            const ColT<TH, PACK> cs = col.lane(sl - lane);
            const int j0 = 2 * b, j1 = 2 * b + 1;
            cs.th(j0) = clampf(fmaf(P.cd_sigma, z.x, cs.th(j0)), Rs.lim[j0].x, Rs.lim[j0].y);
            if (j1 < Rs.n) cs.th(j1) = clampf(fmaf(P.cd_sigma, z.y, cs.th(j1)), Rs.lim[j1].x, Rs.lim[j1].y);
        }
        __syncwarp(am);
    }
    return 0;
}

// resident threads per SM the register allocation aims at: 768 gives 80 registers, the budget
// that leaves no spill, for 24 resident warps
#ifndef HJCD_CCD_THREADS_PER_SM
#define HJCD_CCD_THREADS_PER_SM 768
#endif
// RED = false: the launch's joint vectors lie within the limits of plain robots (no offsets and
// no range reduction in the kinematics steps; the same bits)
template <bool TRACE, int TH, bool RED, bool PACK>
__global__ void __launch_bounds__(TH, HJCD_CCD_THREADS_PER_SM / TH) k_ccd(const CcdArgs A) {
    using Col = ColT<TH, PACK>;
    extern __shared__ __align__(16) float sm[];
    const RobotParams* rob = stage_robots(sm, A.rs);
    uint32_t* const slots = reinterpret_cast<uint32_t*>(sm + robots_smem_bytes(A.rs.n) / sizeof(float));
    float2* const colbase =
        reinterpret_cast<float2*>(sm + robots_smem_bytes(A.rs.n) / sizeof(float) + TH * kSlotWords) + threadIdx.x;
    const hjcd_params& P = A.P;
    const float pe2 = P.proj_eps * P.proj_eps;
    const float one_m_tie = 1.0f - P.cd_tie;
    unsigned long long n_it = 0, n_cand = 0;

    // a segment of the iterations (seg_end > 0): candidates still iterating at seg_end are handed
    // to the next launch through list_out, which runs them from there (list_in)
    const int64_t items = A.list_in ? (int64_t)*A.n_in : A.C;
    const int k_end = A.seg_end > 0 ? A.seg_end : 0x7fffffff;
    // the order of the items: a grid stride, or (A.queue set, a grid of resident CTAs) 32
    // consecutive items per warp from the queue at a time, so that every SM keeps working until
    // the queue is drained whatever the number of waves the items would fill
    const bool dyn = A.queue != nullptr;
    const int wl = threadIdx.x & 31;
    int64_t wbase = 0;
    if (dyn) {
        unsigned long long b0 = 0;
        if (wl == 0) b0 = atomicAdd(A.queue, 32ull);
        wbase = (int64_t)__shfl_sync(0xffffffffu, b0, 0);
    }
    for (int64_t it = dyn ? wbase + wl : blockIdx.x * (int64_t)blockDim.x + threadIdx.x; dyn ? wbase < items : it < items;) {
      do {  // one item (break: done with it)
        if (it >= items) break;  // past the end in the queue's last batch
        const int64_t c = A.list_in ? (int64_t)A.list_in[it] : it;
        int32_t t, s;
        if (!A.map.lookup_search(c, t, s)) break;
        s += A.seed_base;
        const TargetDesc T = A.tg[t];
        const RobotParams& R = rob[T.robot];
        const int n = R.n;
        const Col col(colbase, A.rs.n_max);
        const V3 pt = v3(T.p[0], T.p[1], T.p[2]);
        if (!A.list_in) ++n_cand;

        if (A.list_in) {  // the state the previous segment left
#pragma unroll 1
            for (int j = 0; j < n; ++j) col.th(j) = A.th_out[j * A.ld + c];
        } else if (A.th_in) {
#pragma unroll 1
            for (int j = 0; j < n; ++j) col.th(j) = A.th_in[j * A.ld + c];
        } else {
            sample_seed(R, T, (uint32_t)s, col);
        }

        const int cap = A.n_iters >= 0 ? A.n_iters : T.cd_iters;
        float delta_k = P.cd_delta0 * powf(P.cd_rho, (float)A.k0);
#pragma unroll 1
        for (int q = 0; q < A.seg_begin; ++q) delta_k *= P.cd_rho;  // the bits of one run from k0
        const float inv_p2 = 1.0f / (T.eps_pos * T.eps_pos), inv_o2 = 1.0f / (T.eps_ori * T.eps_ori);
        int iters = cap;
        float ep2 = 0.0f, eo = 0.0f;
        const bool valid = T.eps_pos > 0.0f;
        bool handed = false;

        for (int kk = A.seg_begin; valid; ++kk) {
            if (kk == k_end && kk < cap) {
                // still iterating at the segment's end: keep the state, list the candidate
                const unsigned m = __activemask();
                const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
                int base = 0;
                if (lane == leader) base = atomicAdd(A.n_out, __popc(m));
                base = __shfl_sync(m, base, leader);
                A.list_out[base + __popc(m & ((1u << lane) - 1u))] = (int32_t)c;
                handed = true;
                break;
            }
            const int r = ccd_step<TRACE, TH, RED, PACK>(rob, R, T, P, col, slots, A, c, (uint32_t)s, kk, cap, delta_k, pt, pe2,
                                              one_m_tie, inv_p2, inv_o2, ep2, eo);
            if (r == 1) iters = kk;
            if (r) break;
            delta_k *= P.cd_rho;
            ++n_it;
        }

        if (handed) {
#pragma unroll 1
            for (int j = 0; j < n; ++j) A.th_out[j * A.ld + c] = col.th(j);
            break;
        }
        if (A.th_out) {
#pragma unroll 1
            for (int j = 0; j < n; ++j) A.th_out[j * A.ld + c] = col.th(j);
        }
        const float ep = sqrtf(ep2);
        if (A.score) {
            const float a = ep / T.eps_pos, b = eo / T.eps_ori;
            A.score[c] = valid ? fmaf(a, a, b * b) : __int_as_float(0x7f800000);
        }
        if (A.perr) A.perr[c] = ep;
        if (A.oerr) A.oerr[c] = eo;
        if (A.iters) A.iters[c] = iters;
      } while (0);
        if (dyn) {
            __syncwarp();
            unsigned long long b0 = 0;
            if (wl == 0) b0 = atomicAdd(A.queue, 32ull);
            wbase = (int64_t)__shfl_sync(0xffffffffu, b0, 0);
            it = wbase + wl;
        } else {
            it += (int64_t)gridDim.x * blockDim.x;
        }
    }
    if (A.cnt) {
        n_it = warp_sum(n_it);
        n_cand = warp_sum(n_cand);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&A.cnt->v[0], n_it);
            atomicAdd(&A.cnt->v[5], n_cand);
        }
    }
}

// ----------------------------------------------------------------------------
// PO-CCD with a candidate's work spread over a CTA, for batches too small to fill the GPU with one
// thread per candidate: there the time is the latency of one candidate's chain of iterations, and a
// thread that walks all of its joints one after another makes that chain long (a lone warp issues
// an instruction every four cycles or so, whatever the instruction).  A CTA takes 16 candidates;
// lanes l and l + 16 of every warp belong to candidate l, and the warps share its joints,
// exchanging through shared memory with five barriers per iteration:
//   1. warps 0 and 1, one half warp per row: the x, y and z rows of the kinematics chain, which never
//      meet (a frame's row is updated from the same row only), from the joints' sines and cosines
//   2. the last warp: flange pose, error quaternion, break test; beside it the other warps: their
//      joints' geometry and position step, which need the end effector only
//   3. those warps: the trials of their joints, the position trial in the lower half warp and the
//      orientation trial in the upper one
//   4. warps 0 and 1: greedy choice, acceptance by the position and by the orientation; beside them
//      the others draw the perturbation that the lanes about to reject will need
//   5. every half warp: the accepted update or the perturbation of its joints, their sines and cosines
// The arithmetic is ccd_step's, operation by operation, so the results are its bits.  Bound by
// latency: about 2800 cycles per iteration on Panda (kinematics rows 370, residual 760, trials 475,
// choice and acceptance 525, update 345, the barriers the rest).  One target of 1000 seeds: 45 us for
// at most 32 iterations, where k_ccd takes 119 us (kernel times).
constexpr int kCoopCands = 16;     // candidates per CTA
constexpr int kCoopMaxWarps = 16;  // joint warps and the residual's

struct CoopCol {  // [joint][candidate] fields, nl joints in the layout
    int nl;
    float4* q;     // [candidate]: error quaternion
    float4* pick;  // [candidate]: chosen joints (jp | jo << 8), their steps, accepted by the position
    float2* tr;    // [joint][lane]: score and step of the position (lower half) and orientation trials
    float2* fr;    // [row][joint][candidate]: component `row` of the joint's origin and of its axis
    float2* e;     // [row][candidate]: that component of the last frame's first two axes
    float2* er;    // [candidate]: angle of the error quaternion, position error (0, -1: done)
    float2* cs;    // cosine and sine of the joint angle
    float *th, *nz;  // joint angle, normal draw
    int* acc_o;      // [candidate]: accepted by the orientation
    __device__ __forceinline__ void frame(int j, int l, V3& p, V3& z) const {
        const float2 a = fr[j * kCoopCands + l], b = fr[(nl + j) * kCoopCands + l], c = fr[(2 * nl + j) * kCoopCands + l];
        p = v3(a.x, b.x, c.x);
        z = v3(a.y, b.y, c.y);
    }
};
__host__ __device__ constexpr size_t coop_ccd_bytes(int n) {
    return (size_t)kCoopCands * (sizeof(float4) * 2 + sizeof(float2) * (2 * n + 3 * n + 3 + 1 + n) + sizeof(float) * (2 * n + 1) +
                                 sizeof(int));
}
__device__ __forceinline__ CoopCol coop_col(void* base, int nl) {
    CoopCol C;
    C.nl = nl;
    C.q = reinterpret_cast<float4*>(base);
    C.pick = C.q + kCoopCands;
    C.tr = reinterpret_cast<float2*>(C.pick + kCoopCands);
    C.fr = C.tr + 2 * kCoopCands * nl;
    C.e = C.fr + kCoopCands * 3 * nl;
    C.er = C.e + kCoopCands * 3;
    C.cs = C.er + kCoopCands;
    C.th = reinterpret_cast<float*>(C.cs + kCoopCands * nl);
    C.nz = C.th + kCoopCands * nl;
    C.acc_o = reinterpret_cast<int*>(C.nz + kCoopCands * (nl + 1));  // nz: one row more, an odd chain's last pair
    return C;
}

// One row of the kinematics chain (fk_step's operations on that row): component `row` of every
// joint's origin and axis, and of the last frame's other axes
template <int N>
__device__ __forceinline__ void coop_fk_row(const CoopCol& C, const RobotParams& R, int n, int row, int l) {
    float c0 = row == 0 ? 1.0f : 0.0f, c1 = row == 1 ? 1.0f : 0.0f, c2 = row == 2 ? 1.0f : 0.0f, p = 0.0f;
    float2* const fr = C.fr + row * C.nl * kCoopCands + l;
    const float2* const csl = C.cs + l;
    auto step = [&](int j, const float4 g, const float2 cs) {
        const float b1 = fmaf(g.x, c1, g.y * c2);
        const float b2 = fmaf(g.x, c2, (-g.y) * c1);
        p = fmaf(g.w, b2, fmaf(g.z, c0, p));
        const float n0 = fmaf(cs.x, c0, cs.y * b1);
        c1 = fmaf(cs.x, b1, (-cs.y) * c0);
        c0 = n0;
        c2 = b2;
        fr[j * kCoopCands] = make_float2(p, c2);
    };
    if (N) {  // all loads come before the stores, which the compiler may not move them across
        float4 g[N ? N : 1];
        float2 cs[N ? N : 1];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            g[j] = R.dh[j];
            cs[j] = csl[j * kCoopCands];
        }
#pragma unroll
        for (int j = 0; j < N; ++j) step(j, g[j], cs[j]);
    } else {
#pragma unroll 4
        for (int j = 0; j < n; ++j) step(j, R.dh[j], csl[j * kCoopCands]);
    }
    C.e[row * kCoopCands + l] = make_float2(c0, c1);
}

// The part of ccd_joint_trials that needs the end effector only: a joint's geometry and its position
// step, which here come before the error quaternion is known
struct CcdGeom {
    float nup2, nvp2, nu2, ez, cs, sn, d;
};
__device__ __forceinline__ CcdGeom ccd_joint_geom(const V3 pj, const V3 z, const V3 Ep, const V3 pt, float pe2) {
    CcdGeom g;
    const V3 u = Ep - pj;
    const V3 v = pt - pj;
    const float uz = dot(u, z), vz = dot(v, z);
    const V3 up = fma3(-uz, z, u);
    const V3 vp = fma3(-vz, z, v);
    g.nup2 = dot(up, up);
    g.nvp2 = dot(vp, vp);
    g.nu2 = fmaf(uz, uz, g.nup2);
    const float nv2 = fmaf(vz, vz, g.nvp2);
    const V3 zxu = cross(z, up);
    g.ez = vz - uz;
    g.cs = dot(up, vp);
    g.sn = dot(zxu, vp);
    const bool deg = g.nu2 < 1e-24f || nv2 < 1e-24f || g.nup2 <= pe2 * g.nu2 || g.nvp2 <= pe2 * nv2;
    g.d = deg ? 0.0f : atan2_all(g.sn, g.cs);
    return g;
}

// One trial of a joint: ccd_joint_trials' operations on one half of its pairs, for the step x
__device__ __forceinline__ float2 ccd_joint_trial(const CcdGeom& g, float az, float qp2, float x, float thj, float lo,
                                                  float hi, float qw, float inv_p2, float inv_o2) {
    const float st = __fadd_rn(clampf(__fadd_rn(thj, x), lo, hi), -thj);
    float sh, ch;
    __sincosf(__fmul_rn(0.5f, st), &sh, &ch);
    const float m2sh = __fmul_rn(-2.0f, sh);
    const float msn = __fmul_rn(m2sh, ch);
    const float cst = fmaf(m2sh, sh, 1.0f);
    // both forms of the position residual (ccd_joint_trials says when the first is taken)
    const float ra = fmaf(2.0f, fmaf(msn, g.sn, __fmul_rn(cst, -g.cs)), fmaf(g.ez, g.ez, g.nvp2 + g.nup2));
    const float ex = fmaf(cst, -g.nup2, g.cs), ey = fmaf(msn, g.nup2, g.sn);
    const float rb = fmaf(fmaf(ex, ex, __fmul_rn(ey, ey)), __fdividef(1.0f, g.nup2), __fmul_rn(g.ez, g.ez));
    const float r2 = g.nup2 <= 1e-6f * g.nu2 ? ra : rb;
    const float w = fmaf(qw, ch, __fmul_rn(sh, az));
    const float tz = fmaf(ch, az, __fmul_rn(sh, -qw));
    const float vv = fmaf(tz, tz, qp2);
    // quat_angle2
    const float ay = sqrt_approx(vv), ax = fabsf(w);
    const float t = __fdividef(fminf(ax, ay), fmaxf(fmaxf(ax, ay), 1e-30f));
    const float s = __fmul_rn(t, t);
    float p = fmaf(-4.166443301e-03f, s, 2.232482877e-02f);
    p = fmaf(p, s, -5.666722692e-02f);
    p = fmaf(p, s, 9.704074739e-02f);
    p = fmaf(p, s, -1.393516270e-01f);
    p = fmaf(p, s, 1.995220255e-01f);
    p = fmaf(p, s, -3.333036250e-01f);
    p = fmaf(p, s, 9.999994549e-01f);
    const float ang = ay > ax ? fmaf(__fmul_rn(-2.0f, t), p, 2.0f * 1.57079632679489662f) : __fmul_rn(__fmul_rn(2.0f, t), p);
    return make_float2(fmaf(r2, inv_p2, __fmul_rn(__fmul_rn(ang, ang), inv_o2)), st);
}

// ccd_step's acceptance of theta_hat by the position and by the orientation:
// its residual is the end effector at Ep and the error quaternion turned by da about the distal
// chosen joint (origin Pa, axis Za) first, then by db about the proximal one; ep0 and eo are the
// current errors.
__device__ __forceinline__ bool ccd_accept_pos(float gamma, const V3 Ep, const V3 pt, float ep0, const V3 Pa, const V3 Za,
                                               float da, const V3 Pb, const V3 Zb, float db) {
    float sa_, ca_, sb_, cb_;
    __sincosf(0.5f * da, &sa_, &ca_);
    __sincosf(0.5f * db, &sb_, &cb_);
    V3 x = Pa + rotate_half(Za, sa_, ca_, Ep - Pa);
    x = Pb + rotate_half(Zb, sb_, cb_, x - Pb);
    const V3 e1 = pt - x;
    const float ep1 = sqrt_approx(dot(e1, e1));
    return ep0 - ep1 > gamma;
}
__device__ __forceinline__ bool ccd_accept_ori(float gamma, const Q4 qerr, float eo, const V3 Za, float da, const V3 Zb,
                                               float db) {
    float sa_, ca_, sb_, cb_;
    __sincosf(0.5f * da, &sa_, &ca_);
    __sincosf(0.5f * db, &sb_, &cb_);
    Q4 q1 = qmul(qerr, Q4{ca_, (-sa_) * Za});
    q1 = qmul(q1, Q4{cb_, (-sb_) * Zb});
    const float eo1 = quat_angle(q1.w, dot(q1.v, q1.v));
    return eo - eo1 > gamma;
}

// RED as for k_ccd; N > 0: the launch's one robot has N joints (unrolled loops); N = 0: any robots
template <bool RED, int N>
__global__ void __launch_bounds__(kCoopMaxWarps * 32, 1) k_ccd_coop(const CcdArgs A) {
    extern __shared__ __align__(16) float sm[];
    grid_follow();
    __shared__ long long s_base;
    const RobotParams* rob = stage_robots(sm, A.rs);
    const int WJ = ((int)blockDim.x >> 5) - 1;  // the warps that share the joints
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const int l = lane & (kCoopCands - 1), half = lane >> 4;
    const CoopCol C = coop_col(reinterpret_cast<char*>(sm) + robots_smem_bytes(A.rs.n), N ? N : A.rs.n_max);
    const hjcd_params& P = A.P;
    const float pe2 = P.proj_eps * P.proj_eps;
    const float one_m_tie = 1.0f - P.cd_tie;
    unsigned long long n_it = 0, n_cand = 0;
    auto sincos_of = [&](const RobotParams& R, int j, float th) {
        float s, c;
        if (RED) sincos_red(th + R.off[j], &s, &c);
        else __sincosf(th, &s, &c);
        return make_float2(c, s);
    };

    for (int64_t g = blockIdx.x;; g += gridDim.x) {
        __syncthreads();  // the last group's state is no longer read
        int64_t base = kCoopCands * g;
        if (A.queue) {
            if (threadIdx.x == 0) s_base = (long long)atomicAdd(A.queue, (unsigned long long)kCoopCands);
            __syncthreads();
            base = s_base;
        }
        if (base >= A.C) break;
        const int64_t c = base + l;
        int32_t t = 0, s = 0;
        bool have = c < A.C;
        if (have) have = A.map.lookup_search(c, t, s);
        s += A.seed_base;
        const TargetDesc T = A.tg[have ? t : 0];
        const RobotParams& R = N ? rob[0] : rob[have ? T.robot : 0];
        const int n = N ? N : R.n;  // (a lane without a candidate runs along on a robot's joints, unread)
        const V3 pt = v3(T.p[0], T.p[1], T.p[2]);
        const int cap = A.n_iters >= 0 ? A.n_iters : T.cd_iters;
        const float inv_p2 = 1.0f / (T.eps_pos * T.eps_pos), inv_o2 = 1.0f / (T.eps_ori * T.eps_ori);
        const bool valid = have && T.eps_pos > 0.0f;
        bool alive = valid;
        int iters = cap;              // the residual warp's
        float ep2 = 0.0f, eo = 0.0f;  // the residual warp's
        float delta_k = P.cd_delta0 * powf(P.cd_rho, (float)A.k0);

        // seeds (or the caller's joint vectors), their sines and cosines
        for (int j = 2 * warp + half; j < n; j += 2 * (WJ + 1)) {
            float th = 0.0f;
            if (have && A.th_in) {
                th = A.th_in[j * A.ld + c];
            } else if (have) {
                const uint4 w = rnd_block(T, (uint32_t)s, kPhaseSeed, 0, (uint32_t)(j >> 2));
                th = fmaf(u01(word(w, j & 3)), R.lim[j].y - R.lim[j].x, R.lim[j].x);
            }
            C.th[j * kCoopCands + l] = th;
            C.cs[j * kCoopCands + l] = sincos_of(R, j, th);
        }
        __syncthreads();

        for (int kk = 0;; ++kk) {
            // 1. kinematics rows
            if (2 * warp + half < 3) coop_fk_row<N>(C, R, n, 2 * warp + half, l);
            __syncthreads();

            // 2. residual and break test; beside it the joints' geometry.  (A candidate that is done
            // keeps its errors and runs along: its trials are not read.)
            Frame F;
            {
                const float2 r0 = C.e[l], r1 = C.e[kCoopCands + l], r2 = C.e[2 * kCoopCands + l];
                F.c0 = v3(r0.x, r1.x, r2.x);
                F.c1 = v3(r0.y, r1.y, r2.y);
                C.frame(n - 1, l, F.p, F.c2);
            }
            const Frame E = fk_flange(R, F);
            int j = min(warp, n - 1);
            V3 pj{}, z{};
            CcdGeom g0{};
            if (warp == WJ) {
                const Q4 qe = quat_error(T, quat_from_frame(E));
                const V3 e = pt - E.p;
                if (alive) {
                    ep2 = dot(e, e);
                    eo = quat_angle(qe.w, dot(qe.v, qe.v));
                    if (kk > 0 && ep2 < P.cd_eps_pos2 && eo * eo < P.cd_eps_ori2) {
                        iters = kk;
                        alive = false;
                    } else if (kk == cap) {
                        alive = false;
                    }
                    if (half == 0) {
                        C.q[l] = make_float4(qe.w, qe.v.x, qe.v.y, qe.v.z);
                        C.er[l] = make_float2(eo, alive ? sqrt_approx(ep2) : -1.0f);
                        if (alive) ++n_it;
                    }
                }
            } else {
                C.frame(j, l, pj, z);
                g0 = ccd_joint_geom(pj, z, E.p, pt, pe2);
            }
            if (!__syncthreads_or(warp == WJ && alive)) break;

            // 3. trials
            const float4 q4 = C.q[l];
            const Q4 qerr{q4.x, v3(q4.y, q4.z, q4.w)};
            const float2 er = C.er[l];  // eo, ep
            if (warp != WJ) {
                alive = alive && er.y >= 0.0f;
                const float dphi = delta_k * er.x;
                for (;;) {
                    const float az = dot(qerr.v, z);
                    const V3 qp = fma3(-az, z, qerr.v);
                    // Eq. theta_proj; Eq. ori_update
                    const float x = half == 0 ? g0.d : ((az > 0.0f) ? dphi : ((az < 0.0f) ? -dphi : 0.0f));
                    const float2 tr = ccd_joint_trial(g0, az, dot(qp, qp), x, C.th[j * kCoopCands + l], R.lim[j].x,
                                                      R.lim[j].y, qerr.w, inv_p2, inv_o2);
                    if (warp < n) C.tr[j * 32 + lane] = tr;
                    j += WJ;
                    if (j >= n) break;
                    C.frame(j, l, pj, z);
                    g0 = ccd_joint_geom(pj, z, E.p, pt, pe2);
                }
            }
            __syncthreads();

            // 4. greedy choice and acceptance; the perturbation's draws
            if (warp < 2) {
                float best = __int_as_float(0x7f800000), d = 0.0f;  // of this half's kind of trial
                int jb = 0;
                auto scan = [&](int j) {
                    const float2 v = C.tr[j * 32 + lane];
                    const bool w = v.x < best * one_m_tie;
                    best = w ? v.x : best;
                    jb = w ? j : jb;
                    d = w ? v.y : d;
                };
                if (N) {
#pragma unroll
                    for (int j = 0; j < N; ++j) scan(j);
                } else {
#pragma unroll 4
                    for (int j = 0; j < n; ++j) scan(j);
                }
                const int j2 = __shfl_xor_sync(0xffffffffu, jb, 16);
                const float d2 = __shfl_xor_sync(0xffffffffu, d, 16);
                const int jp = half ? j2 : jb, jo = half ? jb : j2;
                float aP = half ? d2 : d, aO = half ? d : d2;
                if (jp == jo) {  // the larger step
                    if (fabsf(aP) >= fabsf(aO)) aO = 0.0f;
                    else aP = 0.0f;
                }
                const bool p_hi = jp > jo;
                V3 Pa, Za, Pb, Zb;
                C.frame(p_hi ? jp : jo, l, Pa, Za);
                C.frame(p_hi ? jo : jp, l, Pb, Zb);
                const float da = p_hi ? aP : aO, db = p_hi ? aO : aP;
                if (warp == 0) {
                    const bool acc = ccd_accept_pos(P.cd_gamma_pos, E.p, pt, er.y, Pa, Za, da, Pb, Zb, db);
                    C.pick[l] = make_float4(__int_as_float(jp | jo << 8), aP, aO, acc ? 1.0f : 0.0f);
                } else {
                    C.acc_o[l] = ccd_accept_ori(P.cd_gamma_ori, qerr, er.x, Za, da, Zb, db);
                }
            } else if (alive) {
                for (int q = 2 * (warp - 2) + half; 2 * q < n; q += 2 * (WJ - 1)) {
                    const float2 zz = normal_pair(T, (uint32_t)s, kPhaseCd, (uint32_t)(A.k0 + kk), q);
                    C.nz[2 * q * kCoopCands + l] = zz.x;
                    C.nz[(2 * q + 1) * kCoopCands + l] = zz.y;
                }
            }
            __syncthreads();

            // 5. the accepted steps, or theta + N(0, sigma^2 I) (clamped as in ccd_step); the sines and
            // cosines of the next pass
            {
                const float4 pk = C.pick[l];
                const bool acc = pk.w != 0.0f || C.acc_o[l] != 0;
                const int jp = __float_as_int(pk.x) & 255, jo = __float_as_int(pk.x) >> 8;
                for (int i = 2 * warp + half; i < n; i += 2 * (WJ + 1)) {
                    const float th = C.th[i * kCoopCands + l], nz = C.nz[i * kCoopCands + l];
                    const float lo = R.lim[i].x, hi = R.lim[i].y;
                    const float t1 = i == jp ? clampf(th + pk.y, lo, hi) : th;
                    const float t2 = i == jo ? clampf(t1 + pk.z, lo, hi) : t1;
                    const float tn = acc ? t2 : clampf(fmaf(P.cd_sigma, nz, th), lo, hi);
                    if (alive) {
                        C.th[i * kCoopCands + l] = tn;
                        C.cs[i * kCoopCands + l] = sincos_of(R, i, tn);
                    }
                }
            }
            delta_k *= P.cd_rho;
            __syncthreads();
        }

        if (have && A.th_out)
            for (int i = 2 * warp + half; i < n; i += 2 * (WJ + 1)) A.th_out[i * A.ld + c] = C.th[i * kCoopCands + l];
        if (warp == WJ && have && half == 0) {
            ++n_cand;
            const float ep = sqrtf(ep2);
            if (A.score) {
                const float a = ep / T.eps_pos, b = eo / T.eps_ori;
                A.score[c] = valid ? fmaf(a, a, b * b) : __int_as_float(0x7f800000);
            }
            if (A.perr) A.perr[c] = ep;
            if (A.oerr) A.oerr[c] = eo;
            if (A.iters) A.iters[c] = iters;
        }
    }
    if (A.cnt && warp == WJ) {
        n_it = warp_sum(n_it);
        n_cand = warp_sum(n_cand);
        if (lane == 0) {
            atomicAdd(&A.cnt->v[0], n_it);
            atomicAdd(&A.cnt->v[5], n_cand);
        }
    }
}

// cd_variant = 2, the target-wide break: one CTA per target runs all of its
// seeds in lock-step, iteration by iteration, and stops every seed once any
// seed passes the coarse test.  Pass kk tests each seed's state after kk
// updates and writes its update to the other buffer; when some seed passed,
// the updates of that pass are dropped and every seed keeps its state after
// kk updates.
template <int TH>
__global__ void __launch_bounds__(TH, 4) k_ccd_lock(const CcdArgs A) {
    extern __shared__ __align__(16) float sm[];
    __shared__ int any;
    const RobotParams* rob = stage_robots(sm, A.rs);
    uint32_t* const slots = reinterpret_cast<uint32_t*>(sm + robots_smem_bytes(A.rs.n) / sizeof(float));
    float2* const colbase =
        reinterpret_cast<float2*>(sm + robots_smem_bytes(A.rs.n) / sizeof(float) + TH * kSlotWords) + threadIdx.x;
    const int t = blockIdx.x;
    const hjcd_params& P = A.P;
    const TargetDesc T = A.tg[t];
    const RobotParams& R = rob[T.robot];
    const int n = R.n;
    const ColT<TH> col(colbase, A.rs.n_max);
    const int64_t m0 = A.map.off[t];
    const int M = (int)(A.map.off[t + 1] - m0);
    const bool valid = T.eps_pos > 0.0f;
    const int cap = A.n_iters >= 0 ? A.n_iters : T.cd_iters;
    const V3 pt = v3(T.p[0], T.p[1], T.p[2]);
    const float pe2 = P.proj_eps * P.proj_eps, one_m_tie = 1.0f - P.cd_tie;
    const float inv_p2 = 1.0f / (T.eps_pos * T.eps_pos), inv_o2 = 1.0f / (T.eps_ori * T.eps_ori);
    float* cur = A.th_out;
    float* nxt = A.th_tmp;
    for (int s = threadIdx.x; s < M; s += TH) {
        const int64_t c = m0 + s;
        if (A.th_in) {
            for (int j = 0; j < n; ++j) cur[j * A.ld + c] = A.th_in[j * A.ld + c];
        } else {
            sample_seed(R, T, (uint32_t)s, col);
            for (int j = 0; j < n; ++j) cur[j * A.ld + c] = col.th(j);
        }
    }
    unsigned long long n_it = 0;
    float delta_k = P.cd_delta0 * powf(P.cd_rho, (float)A.k0);
    int kk = 0;
    for (; valid; ++kk) {
        if (threadIdx.x == 0) any = 0;
        __syncthreads();
        for (int s = threadIdx.x; s < M; s += TH) {
            const int64_t c = m0 + s;
#pragma unroll 1
            for (int j = 0; j < n; ++j) col.th(j) = cur[j * A.ld + c];
            float ep2 = 0.0f, eo = 0.0f;
            const int r = ccd_step<false, TH>(rob, R, T, P, col, slots, A, c, (uint32_t)s, kk, cap, delta_k, pt, pe2,
                                              one_m_tie, inv_p2, inv_o2, ep2, eo);
            const float ep = sqrtf(ep2), a = ep / T.eps_pos, b = eo / T.eps_ori;
            if (A.score) A.score[c] = fmaf(a, a, b * b);
            if (A.perr) A.perr[c] = ep;
            if (A.oerr) A.oerr[c] = eo;
            if (r == 1) any = 1;
            if (r == 0) {
                ++n_it;
#pragma unroll 1
                for (int j = 0; j < n; ++j) nxt[j * A.ld + c] = col.th(j);
            }
        }
        __syncthreads();
        if (any || kk == cap) break;
        float* sw = cur;
        cur = nxt;
        nxt = sw;
        delta_k *= P.cd_rho;
    }
    for (int s = threadIdx.x; s < M; s += TH) {
        const int64_t c = m0 + s;
        if (cur != A.th_out)
            for (int j = 0; j < n; ++j) A.th_out[j * A.ld + c] = cur[j * A.ld + c];
        if (!valid && A.score) A.score[c] = __int_as_float(0x7f800000);
        if (A.iters) A.iters[c] = valid ? kk : cap;
    }
    if (A.cnt) {
        n_it = warp_sum(n_it);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&A.cnt->v[0], n_it);
            if (threadIdx.x == 0) atomicAdd(&A.cnt->v[5], (unsigned long long)M);
        }
    }
}

__global__ void __launch_bounds__(kCcdThreads) k_sample(const RobotParams R, uint32_t k0, uint32_t k1, CandMap map,
                                                        int64_t C, float* th_out, int64_t ld) {
    extern __shared__ float sm[];
    const ThetaCol<kCcdThreads> col{sm + threadIdx.x};
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < C; c += (int64_t)gridDim.x * blockDim.x) {
        int32_t t, s;
        map.lookup(c, t, s);  // only the row index keys the stream
        TargetDesc T{};
        T.key[0] = k0;
        T.key[1] = k1;
        T.t_local = t;
        sample_seed(R, T, (uint32_t)s, col);
#pragma unroll 1
        for (int j = 0; j < R.n; ++j) th_out[j * ld + c] = col.th(j);
    }
}


template <bool PACK>
size_t ccd_smem(int robots, int n, int th) {
    return robots_smem_bytes(robots) + sizeof(float) * (ColT<64, PACK>::kWords * n + kSlotWords) * th;
}

template <bool TRACE, int TH, bool RED, bool PACK>
int prepare_ccd(const CcdArgs& A) {  // resident CTAs per SM
    static SmemLimit lim;
    allow_dyn_smem(k_ccd<TRACE, TH, RED, PACK>, lim, ccd_smem<PACK>(kMaxLaunchRobots, kMaxDof, TH));
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ccd<TRACE, TH, RED, PACK>, TH,
                                                  ccd_smem<PACK>(A.rs.n, A.rs.n_max, TH));
    return std::max(per_sm, 1);
}

template <bool TRACE, int TH, bool RED, bool PACK>
void launch_ccd_p(const CcdArgs& A, int per_sm, cudaStream_t st) {
    int g = grid_for(A.C, TH, 16 * 128 / TH);
    if (A.queue) g = std::min(g, sm_count() * per_sm);  // the resident CTAs only: the queue spreads the items
    k_ccd<TRACE, TH, RED, PACK><<<g, TH, ccd_smem<PACK>(A.rs.n, A.rs.n_max, TH), st>>>(A);
}

template <bool TRACE, int TH, bool RED>
void launch_ccd_t(const CcdArgs& A, cudaStream_t st) {
    const int per_sm = prepare_ccd<TRACE, TH, RED, false>(A);
    if (!TRACE) {
        // the packed column where it lets a fifth more CTAs reside (8 robots of up to 20 joints: 4 -> 5,
        // 1.42 -> 1.27 ms; at 12 joints, 7 -> 8, it costs 1%)
        const int packed = prepare_ccd<TRACE, TH, RED, !TRACE>(A);
        if (5 * packed >= 6 * per_sm) return launch_ccd_p<TRACE, TH, RED, !TRACE>(A, packed, st);
    }
    launch_ccd_p<TRACE, TH, RED, false>(A, per_sm, st);
}

template <bool RED, int N>
void launch_ccd_coop_n(const CcdArgs& A, int warps, cudaStream_t st) {
    const size_t smem = robots_smem_bytes(A.rs.n) + coop_ccd_bytes(A.rs.n_max);
    static SmemLimit lim;
    allow_dyn_smem(k_ccd_coop<RED, N>, lim, robots_smem_bytes(kMaxLaunchRobots) + coop_ccd_bytes(kMaxDof));
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ccd_coop<RED, N>, 32 * warps, smem);
    const int g = (int)std::min<int64_t>((A.C + kCoopCands - 1) / kCoopCands, (int64_t)sm_count() * std::max(per_sm, 1));
    launch_next<CcdArgs>(k_ccd_coop<RED, N>, g, 32 * warps, smem, st, A);
}

template <bool RED>
void launch_ccd_coop(const CcdArgs& A, int warps, cudaStream_t st) {
    const int n = A.rs.n == 1 ? A.rs.n_max : 0;
    if (n == 6) launch_ccd_coop_n<RED, 6>(A, warps, st);
    else if (n == 7) launch_ccd_coop_n<RED, 7>(A, warps, st);
    else launch_ccd_coop_n<RED, 0>(A, warps, st);
}

template <bool TRACE, bool RED>
void launch_ccd_b(const CcdArgs& A, cudaStream_t st) {
    if (A.block == 64) launch_ccd_t<TRACE, 64, RED>(A, st);
    else if (A.block == 256) launch_ccd_t<TRACE, 256, RED>(A, st);
    else launch_ccd_t<TRACE, 128, RED>(A, st);
}

}  // namespace

constexpr int kCoopShort = 4;  // joints up to which the spread kernel gains little
// Whether a launch goes to the spread kernel (explained in launch_ccd)
static bool ccd_spread(const CcdArgs& A, bool trace) {
    const bool whole = !trace && A.P.cd_variant == 0 && !A.list_in && A.seg_begin == 0 && A.seg_end == 0;
    return whole && A.C <= (int64_t)sm_count() * (A.rs.n_max <= kCoopShort ? 2 : 4) * kCoopCands;
}

int ccd_block_used(const CcdArgs& A, int asked) {
    return A.C <= 0 || A.P.cd_variant == 2 || ccd_spread(A, false) ? 0 : asked;
}

void launch_ccd(const CcdArgs& A, bool trace, cudaStream_t st) {
    if (A.C <= 0) return;
    if (A.P.cd_variant == 2) {  // one CTA per target (offset maps only)
        const size_t smem =
            ccd_smem<false>(A.rs.n, A.rs.n_max, 128);
        static SmemLimit lim;
        allow_dyn_smem(k_ccd_lock<128>, lim, ccd_smem<false>(kMaxLaunchRobots, kMaxDof, 128));
        k_ccd_lock<128><<<A.map.T, 128, smem, st>>>(A);
        return;
    }
    // Up to 64 candidates per SM (two resident CTAs of 16 on every SM, twice) the spread kernel's
    // shorter iterations win; past that its extra work does, and for a chain of up to four joints, which
    // leaves little to spread, past 32 (one to four joints, 9000 candidates: 101 / 61, 104 / 72, 107 / 85,
    // 109 / 96 us; 4800: 55 / 61 to 57 / 96; five joints 112 / 110).  Phase time, spread / one thread per
    // candidate, us (7, 20, 24 joints): 1000 candidates 55 / 125, 91 / 267, 106 / 311; 4000: 59 / 125, 118 / 269, 135 / 313;
    // 8000: 109 / 126, 224 / 269, 258 / 313; 16000: 198 / 126, 400 / 272, 464 / 314.  Eight warps (the
    // residual's and seven joint warps), twelve for a long chain while a CTA has its SM to itself
    // (20 joints, 1000 candidates: 99 with eight).
    if (ccd_spread(A, trace)) {
        const int warps = A.rs.n_max > 8 && A.C <= (int64_t)sm_count() * kCoopCands ? 12 : 8;
        if (A.in_limits && A.rs.plain) launch_ccd_coop<false>(A, warps, st);
        else launch_ccd_coop<true>(A, warps, st);
        return;
    }
    if (trace) launch_ccd_b<true, true>(A, st);
    else if (A.in_limits && A.rs.plain) launch_ccd_b<false, false>(A, st);
    else launch_ccd_b<false, true>(A, st);
}

void launch_sample(const RobotParams& R, uint64_t seed, CandMap map, int64_t C, float* th, int64_t ld,
                   cudaStream_t st) {
    if (C <= 0) return;
    const uint32_t k0 = (uint32_t)(seed & 0xffffffffu), k1 = (uint32_t)(seed >> 32);
    k_sample<<<grid_for(C, kCcdThreads), kCcdThreads, sizeof(float) * R.n * kCcdThreads, st>>>(R, k0, k1, map, C,
                                                                                               th, ld);
}

}  // namespace hjcd
