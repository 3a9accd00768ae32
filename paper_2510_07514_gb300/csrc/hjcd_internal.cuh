// hjcd_internal.cuh -- types and device math shared by the HJCD-IK kernels.
//
// All arithmetic is binary32.  Joint vectors are structure-of-arrays
// (theta[j * ld + c]).  One launch may mix robots and scenes: every target
// row names its robot and scene in the launch's tables, and the kernels copy
// the (small) kinematic tables of the launch's robots into shared memory.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "hjcd.h"

namespace hjcd {

constexpr int kMaxDof = HJCD_MAX_DOF;
constexpr int kMaxBodies = HJCD_MAX_DOF + 2;
constexpr int kMaxLaunchRobots = HJCD_MAX_BATCH_ROBOTS;  // robots one launch can mix

// Philox stream phases (third counter word, high byte).
enum : uint32_t { kPhaseSeed = 1, kPhaseCd = 2, kPhaseDup = 3, kPhaseLm = 4 };

// Robot as seen by the kernels: modified-DH table, limits, flange transform
// (736 bytes).  A joint's cos alpha, sin alpha, a and d sit together, so one
// 16-byte load per kinematics step fetches them.
struct __align__(16) RobotParams {
    int32_t n;
    int32_t n_sph;
    int32_t plain;  // 1: every joint offset is 0 and every theta within the limits lies inside (-pi, pi)
    int32_t fl_eye; // 1: the flange rotation is the identity (the flange frame's axes are the last joint's)
    float4 dh[kMaxDof];  // cos alpha, sin alpha, a, d
    float off[kMaxDof];
    float2 lim[kMaxDof];  // joint limits lo, hi
    float fl_r[9];  // flange rotation, row-major
    float fl_p[3];  // flange translation
};
static_assert(sizeof(RobotParams) % 16 == 0, "RobotParams tables are 16-byte aligned in shared memory");

// Collision tables of a robot in device memory: spheres grouped by body
// (float4 x y z r in the body frame) with their bodies, per-body
// [first, count) ranges and bounding spheres, the body pairs checked for
// self-collision.
struct RobotDev {
    const float4* sph;    // [n_sph], grouped by body
    const int32_t* body;  // [n_sph]
    const int2* range;    // [n + 2]: first sphere, count
    const float4* coarse; // [n + 2]: bounding sphere in the body frame (r = 0: no spheres)
    const int2* pairs;    // [n_pairs]
    int32_t n_pairs;
    int32_t n_sph;
};

// Obstacles of a scene in device memory: spheres (float4) followed by boxes
// (two float4: lo.xyz, hi.xyz); 16-byte aligned.  A large scene also carries
// a uniform grid over its sphere centres: the spheres are sorted by cell and
// cell[k] .. cell[k+1] are the spheres whose centre lies in cell k (cells
// numbered x fastest); a query for a ball of radius R searches the cells
// within R + reach of its centre.
struct SceneDev {
    const float4* obj;
    int32_t n_sph, n_box;
    const int32_t* cell;  // [dim.x * dim.y * dim.z + 1], or null: no grid
    float lo[3];          // grid origin
    float inv_h;          // 1 / cell edge
    int32_t dim[3];       // cells per axis
    float reach;          // largest obstacle radius, plus a margin beyond binary32 rounding
};

// The robots of one launch and the maxima the kernels size shared memory by.
struct RobotSet {
    const RobotParams* rp;  // [n] (device)
    const RobotDev* rd;     // [n] (device; read by the collision kernel only)
    int32_t n;
    int32_t n_max;          // largest DoF
    int32_t ns_max;         // most link spheres
    int32_t pairs_max;      // most self-collision body pairs
    int32_t plain = 0;      // 1: every robot of the set is plain (see RobotParams)
};

// One target pose with its request's tolerances, random-stream key, robot,
// scene and iteration caps (64 bytes).
struct __align__(16) TargetDesc {
    float p[3];
    float eps_pos;
    float q[4];  // w x y z, unit
    uint32_t key[2];
    int32_t t_local;  // target index inside its request (keys the streams)
    float eps_ori;
    int32_t robot;     // row of the launch's RobotSet
    int32_t scene;     // row of the launch's scene table, -1: no obstacles
    int16_t cd_iters;  // PO-CCD iteration cap
    int16_t lm_iters;  // PJ-IK iteration cap
    int32_t top_k;     // solutions returned; kNearestFlag set: ranked nearest-first (RankArgs::q_ref)
};
constexpr int32_t kNearestFlag = 1 << 30;
static_assert(sizeof(TargetDesc) == 64, "TargetDesc layout");

// Copy the launch's robot tables into shared memory (all threads of the CTA
// take part; ends with a barrier).
__device__ __forceinline__ const RobotParams* stage_robots(void* smem, const RobotSet& rs) {
    const uint4* src = reinterpret_cast<const uint4*>(rs.rp);
    uint4* dst = reinterpret_cast<uint4*>(smem);
    const int words = rs.n * (int)(sizeof(RobotParams) / 16);
    for (int i = threadIdx.x; i < words; i += blockDim.x) dst[i] = __ldg(src + i);
    __syncthreads();
    return reinterpret_cast<const RobotParams*>(smem);
}

__host__ __device__ constexpr size_t robots_smem_bytes(int n) { return (sizeof(RobotParams) * (size_t)n + 15) / 16 * 16; }

// Candidate -> (target row, candidate index inside the target).
struct CandMap {
    const int32_t* tgt;   // explicit [C], or null
    const int32_t* cand;  // explicit [C]
    const int64_t* off;   // [T+1] prefix offsets, used when tgt is null
    int32_t T;
    int32_t stride;       // > 0: every target has this many candidates (off[t] = t * stride)

    // false when an explicit target row is outside [0, T): the candidate is skipped
    __device__ __forceinline__ bool lookup(int64_t c, int32_t& t, int32_t& s) const {
        if (!tgt && stride > 0) {  // no search: a division
            if (c < 0x7fffffff) {
                const uint32_t q = (uint32_t)c / (uint32_t)stride;
                t = (int32_t)q;
                s = (int32_t)((uint32_t)c - q * (uint32_t)stride);
            } else {
                t = (int32_t)(c / stride);
                s = (int32_t)(c - (int64_t)t * stride);
            }
            return true;
        }
        return lookup_search(c, t, s);
    }

    // the same without the stride (kernels that look a candidate up once)
    __device__ __forceinline__ bool lookup_search(int64_t c, int32_t& t, int32_t& s) const {
        if (tgt) {
            t = tgt[c];
            s = cand[c];
            return (uint32_t)t < (uint32_t)T;
        }
        int lo = 0, hi = T - 1;  // largest t with off[t] <= c
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (__ldg(off + mid) <= c) lo = mid;
            else hi = mid - 1;
        }
        t = lo;
        s = (int32_t)(c - __ldg(off + lo));
        return true;
    }
};

// Copy joint vector c (structure of arrays, src[j * ld + c], j < n) into dst(j), K loads in
// flight at a time: a rolled loop would wait out one global-memory latency per joint.
template <int K, class Dst>
__device__ __forceinline__ void load_joints(const float* src, int64_t ld, int64_t c, int n, Dst dst) {
#pragma unroll 1
    for (int j0 = 0; j0 < n; j0 += K) {
        float v[K];
#pragma unroll
        for (int q = 0; q < K; ++q) v[q] = j0 + q < n ? src[(int64_t)(j0 + q) * ld + c] : 0.0f;
#pragma unroll
        for (int q = 0; q < K; ++q)
            if (j0 + q < n) dst(j0 + q, v[q]);
    }
}

// Device work counters (see hjcd_counters).
struct Counters {
    unsigned long long v[8];
};

// ----------------------------------------------------------------------------
// small vector algebra

struct V3 {
    float x, y, z;
};

__device__ __forceinline__ V3 v3(float x, float y, float z) { return V3{x, y, z}; }
__device__ __forceinline__ V3 operator+(V3 a, V3 b) { return V3{a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ V3 operator-(V3 a, V3 b) { return V3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ V3 operator*(float s, V3 a) { return V3{s * a.x, s * a.y, s * a.z}; }
// s * a + b with fused multiply-adds
__device__ __forceinline__ V3 fma3(float s, V3 a, V3 b) {
    return V3{fmaf(s, a.x, b.x), fmaf(s, a.y, b.y), fmaf(s, a.z, b.z)};
}
__device__ __forceinline__ float dot(V3 a, V3 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ V3 cross(V3 a, V3 b) {
    return V3{fmaf(a.y, b.z, -a.z * b.y), fmaf(a.z, b.x, -a.x * b.z), fmaf(a.x, b.y, -a.y * b.x)};
}

__device__ __forceinline__ float clampf(float x, float lo, float hi) { return fminf(fmaxf(x, lo), hi); }

// sin and cos after reducing x to [-pi, pi] (Cody-Waite, 2*pi split into a
// binary32 head and its residual), where the hardware approximation is
// accurate to ~4e-7 absolute.
__device__ __forceinline__ void sincos_red(float x, float* s, float* c) {
    const float k = rintf(x * 0.159154943091895336f);
    float r = fmaf(-k, 6.28318548202514648f, x);
    r = fmaf(-k, -1.74845553e-07f, r);
    __sincosf(r, s, c);
}

// ----------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11) and the maps to (0,1) and N(0,1)

__device__ __forceinline__ uint4 philox(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

__device__ __forceinline__ uint4 rnd_block(const TargetDesc& T, uint32_t cand, uint32_t phase, uint32_t iter,
                                           uint32_t block) {
    return philox(make_uint4(cand, (uint32_t)T.t_local, (phase << 24) | (iter & 0xFFFFFFu), block), T.key[0],
                  T.key[1]);
}

// ((x >> 9) + 1/2) * 2^-23: exact in binary32, inside (0, 1)
__device__ __forceinline__ float u01(uint32_t x) { return ((float)(x >> 9) + 0.5f) * 1.1920928955078125e-07f; }

// Square root by the hardware approximation (PTX sqrt.approx.f32, a few ulp):
// for the angles and norms that rank trials and test tolerances, where the
// IEEE-rounded sqrtf's correction steps cost issue slots of issue-bound
// kernels and buy no decision the binary32 kinematics can resolve.
__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// ln u of u = u01(x) in (0, 1).  The hardware logarithm's absolute error (at most 2^-21.4) would
// dominate ln u near 1, so below v = 1 - u = 2^-8 (v exact for u >= 1/2) three terms of
// -ln(1 - v) = v + v^2/2 + v^3/3 + ... take over (truncation below 2e-8 of ln u).
__device__ __forceinline__ float ln_u01(uint32_t x) {
    const float u = u01(x);
    const float v = 1.0f - u;
    return v < 0.00390625f ? -v * fmaf(v, fmaf(v, 0.333333343f, 0.5f), 1.0f) : __logf(u);
}

// N(0, 1) by Box-Muller, cosine branch: sqrt(-2 ln u0) cos(2 pi u1), with the hardware
// approximations (the angle taken as 2 pi (u1 - 1/2) in [-pi, pi), whose cosine is the negated
// one); the absolute error stays below 5e-6 against the exact mapping.
__device__ __forceinline__ float normal01(uint32_t a, uint32_t b) {
    return sqrt_approx(-2.0f * ln_u01(a)) * -__cosf(6.28318530718f * (u01(b) - 0.5f));
}

__device__ __forceinline__ uint32_t word(uint4 w, int i) { return i == 0 ? w.x : (i == 1 ? w.y : (i == 2 ? w.z : w.w)); }

// the pair of normals of block b of a stream: normal 2b from words (x, y),
// normal 2b+1 from words (z, w)
__device__ __forceinline__ float2 normal_pair(const TargetDesc& T, uint32_t cand, uint32_t phase, uint32_t iter,
                                              int b) {
    const uint4 w = rnd_block(T, cand, phase, iter, (uint32_t)b);
    return make_float2(normal01(w.x, w.y), normal01(w.z, w.w));
}

// ----------------------------------------------------------------------------
// forward kinematics (Eq. fk), modified DH in column form
//
// With C0 C1 C2 the columns of R_{0,i-1}: R_{0,i-1} Rx(alpha) has columns
// C0, B1 = ca C1 + sa C2, B2 = ca C2 - sa C1; the origin moves by a C0 + d B2;
// Rz(theta) then gives C0' = c C0 + s B1, C1' = c B1 - s C0, C2' = B2.  The
// joint axis is B2 and the new origin lies on it.

struct Frame {
    V3 c0, c1, c2, p;
};

__device__ __forceinline__ Frame frame_identity() {
    return Frame{v3(1.f, 0.f, 0.f), v3(0.f, 1.f, 0.f), v3(0.f, 0.f, 1.f), v3(0.f, 0.f, 0.f)};
}

__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 xy(V3 a) { return make_float2(a.x, a.y); }

// The x and y components run as packed FP32 pairs, the operations of the scalar form in its order.
// RED = false leaves out the offset and the range reduction of theta + offset: the caller
// guarantees theta within the limits of a plain robot, whose offsets are 0 and where the
// reduction's multiple of 2 pi is 0, so both return their argument unchanged (the same bits either
// way, up to the sign of an exact zero).
template <bool RED = true>
__device__ __forceinline__ void fk_step(const RobotParams& R, int j, float theta, Frame& F) {
    const float4 g = R.dh[j];
    const float ca = g.x, sa = g.y;
    const float2 b1 = fma2(bc2(ca), xy(F.c1), mul2(bc2(sa), xy(F.c2)));
    const float b1z = fmaf(ca, F.c1.z, sa * F.c2.z);
    const float2 b2 = fma2(bc2(ca), xy(F.c2), mul2(bc2(-sa), xy(F.c1)));
    const float b2z = fmaf(ca, F.c2.z, (-sa) * F.c1.z);
    const float2 p = fma2(bc2(g.w), b2, fma2(bc2(g.z), xy(F.c0), xy(F.p)));
    F.p = v3(p.x, p.y, fmaf(g.w, b2z, fmaf(g.z, F.c0.z, F.p.z)));
    float s, c;
    if (RED) sincos_red(theta + R.off[j], &s, &c);
    else __sincosf(theta, &s, &c);
    const float2 n0 = fma2(bc2(c), xy(F.c0), mul2(bc2(s), b1));
    const float2 n1 = fma2(bc2(c), b1, mul2(bc2(-s), xy(F.c0)));
    const float n0z = fmaf(c, F.c0.z, s * b1z), n1z = fmaf(c, b1z, (-s) * F.c0.z);
    F.c0 = v3(n0.x, n0.y, n0z);
    F.c1 = v3(n1.x, n1.y, n1z);
    F.c2 = v3(b2.x, b2.y, b2z);
}

// fk_step's operations with the cosine c and sine s of the joint's angle given
__device__ __forceinline__ void fk_step_cs(const RobotParams& R, int j, float c, float s, Frame& F) {
    const float4 g = R.dh[j];
    const float ca = g.x, sa = g.y;
    const float2 b1 = fma2(bc2(ca), xy(F.c1), mul2(bc2(sa), xy(F.c2)));
    const float b1z = fmaf(ca, F.c1.z, sa * F.c2.z);
    const float2 b2 = fma2(bc2(ca), xy(F.c2), mul2(bc2(-sa), xy(F.c1)));
    const float b2z = fmaf(ca, F.c2.z, (-sa) * F.c1.z);
    const float2 p = fma2(bc2(g.w), b2, fma2(bc2(g.z), xy(F.c0), xy(F.p)));
    F.p = v3(p.x, p.y, fmaf(g.w, b2z, fmaf(g.z, F.c0.z, F.p.z)));
    const float2 n0 = fma2(bc2(c), xy(F.c0), mul2(bc2(s), b1));
    const float2 n1 = fma2(bc2(c), b1, mul2(bc2(-s), xy(F.c0)));
    const float n0z = fmaf(c, F.c0.z, s * b1z), n1z = fmaf(c, b1z, (-s) * F.c0.z);
    F.c0 = v3(n0.x, n0.y, n0z);
    F.c1 = v3(n1.x, n1.y, n1z);
    F.c2 = v3(b2.x, b2.y, b2z);
}

// flange frame from the last joint frame
__device__ __forceinline__ Frame fk_flange(const RobotParams& R, const Frame& F) {
    Frame E;
    if (R.fl_eye) {  // the general form's products with 1 and 0 (up to the sign of an exact zero)
        E.c0 = F.c0;
        E.c1 = F.c1;
        E.c2 = F.c2;
        E.p = fma3(R.fl_p[2], F.c2, fma3(R.fl_p[1], F.c1, fma3(R.fl_p[0], F.c0, F.p)));
        return E;
    }
    E.c0 = fma3(R.fl_r[6], F.c2, fma3(R.fl_r[3], F.c1, R.fl_r[0] * F.c0));
    E.c1 = fma3(R.fl_r[7], F.c2, fma3(R.fl_r[4], F.c1, R.fl_r[1] * F.c0));
    E.c2 = fma3(R.fl_r[8], F.c2, fma3(R.fl_r[5], F.c1, R.fl_r[2] * F.c0));
    E.p = fma3(R.fl_p[2], F.c2, fma3(R.fl_p[1], F.c1, fma3(R.fl_p[0], F.c0, F.p)));
    return E;
}

// Flange frame of the joint vector theta[j * stride] (joint loop not
// unrolled: the kernels keep their code small enough for the instruction
// cache, with per-joint state in shared memory).
__device__ __forceinline__ Frame fk_ee_col(const RobotParams& R, const float* th, int stride) {
    Frame F = frame_identity();
#pragma unroll 1
    for (int j = 0; j < R.n; ++j) fk_step(R, j, th[j * stride], F);
    return fk_flange(R, F);
}

// ----------------------------------------------------------------------------
// quaternions (w, x, y, z)

struct Q4 {
    float w;
    V3 v;
};

// Unit quaternion of the rotation with columns c0 c1 c2 (Shepperd's method:
// the largest of 4w^2, 4x^2, 4y^2, 4z^2 from the diagonal, the rest from the
// off-diagonal sums), returned with w >= 0.  The pivot is chosen first and one
// square root serves every case, so lanes with different pivots do not
// diverge; the pivot t = 4 max(w^2, x^2, y^2, z^2) is at least 1, and with
// rs = 1/sqrt(t) the pivot component is t rs / 2 and the others are sums
// times rs / 2.
__device__ __forceinline__ Q4 quat_from_frame(const Frame& E) {
    const float m00 = E.c0.x, m10 = E.c0.y, m20 = E.c0.z;
    const float m01 = E.c1.x, m11 = E.c1.y, m21 = E.c1.z;
    const float m02 = E.c2.x, m12 = E.c2.y, m22 = E.c2.z;
    const float tr = m00 + m11 + m22;
    const bool b0 = tr >= m00 && tr >= m11 && tr >= m22;
    const bool b1 = !b0 && m00 >= m11 && m00 >= m22;
    const bool b2 = !b0 && !b1 && m11 >= m22;
    const float t = b0 ? 1.0f + tr : (b1 ? 1.0f + m00 - m11 - m22 : (b2 ? 1.0f + m11 - m00 - m22 : 1.0f + m22 - m00 - m11));
    const float rs = rsqrtf(t);
    const float h = 0.5f * t * rs, r = 0.5f * rs;
    const float a = (m21 - m12) * r, bq = (m02 - m20) * r, c = (m10 - m01) * r;
    const float d = (m01 + m10) * r, e = (m02 + m20) * r, f = (m12 + m21) * r;
    const float w = b0 ? h : (b1 ? a : (b2 ? bq : c));
    const float x = b0 ? a : (b1 ? h : (b2 ? d : e));
    const float y = b0 ? bq : (b1 ? d : (b2 ? h : f));
    const float z = b0 ? c : (b1 ? e : (b2 ? f : h));
    const float sg = (w < 0.0f) ? -1.0f : 1.0f;
    return Q4{sg * w, v3(sg * x, sg * y, sg * z)};
}

__device__ __forceinline__ Q4 qmul(Q4 a, Q4 b) {
    return Q4{a.w * b.w - dot(a.v, b.v), fma3(a.w, b.v, fma3(b.w, a.v, cross(a.v, b.v)))};
}

// q_err = q_t (x) q_e^-1 with the sign chosen so that w >= 0
__device__ __forceinline__ Q4 quat_error(const TargetDesc& T, Q4 qe) {
    const Q4 qt{T.q[0], v3(T.q[1], T.q[2], T.q[3])};
    Q4 e = qmul(qt, Q4{qe.w, (-1.0f) * qe.v});
    if (e.w < 0.0f) {
        e.w = -e.w;
        e.v = (-1.0f) * e.v;
    }
    return e;
}


// Arctangent of t in [0, 1] as t P(t^2), P of degree 7: the coefficients
// minimise the largest absolute error on a dense grid of [0, 1] (a linear
// program; fit_atan.py beside this file regenerates them); |error| < 3e-8 rad
// in exact arithmetic and < 1.5e-7 rad evaluated in binary32 (checked against
// float64 over [0, 1] by the test suite, which reads these coefficients from
// this file and compares them with the script's output).
__device__ __forceinline__ float atan01(float t) {
    const float s = t * t;
    float p = -4.166443301e-03f;
    p = fmaf(p, s, 2.232482877e-02f);
    p = fmaf(p, s, -5.666722692e-02f);
    p = fmaf(p, s, 9.704074739e-02f);
    p = fmaf(p, s, -1.393516270e-01f);
    p = fmaf(p, s, 1.995220255e-01f);
    p = fmaf(p, s, -3.333036250e-01f);
    p = fmaf(p, s, 9.999994549e-01f);
    return t * p;
}

// atan2(y, x) for y >= 0, x >= 0: the ratio of the smaller to the larger
// argument in [0, 1], reflected about pi/4 when y > x
__device__ __forceinline__ float atan2_q1(float y, float x) {
    const float mx = fmaxf(x, y), mn = fminf(x, y);
    const float a = atan01(__fdividef(mn, fmaxf(mx, 1e-30f)));  // 0 at the origin
    return y > x ? 1.57079632679489662f - a : a;
}

// atan2(y, x) over all four quadrants (atan2(+-0, x < 0) = +-pi)
__device__ __forceinline__ float atan2_all(float y, float x) {
    float a = atan2_q1(fabsf(y), fabsf(x));
    if (x < 0.0f) a = 3.14159265358979324f - a;
    return copysignf(a, y);
}

// rotation angle of a (not necessarily unit-normalised) error quaternion,
// 2 atan2(|v|, |w|): the norm of omega in Eq. quat_diff
__device__ __forceinline__ float quat_angle(float w, float vv) { return 2.0f * atan2_q1(sqrt_approx(vv), fabsf(w)); }

// omega of Eq. quat_diff
__device__ __forceinline__ V3 quat_log(Q4 e) {
    const float vv = dot(e.v, e.v);
    const float rs = rsqrtf(vv);  // |v| = vv rs
    const float f = (vv > 1e-30f) ? 2.0f * atan2_q1(vv * rs, e.w) * rs : __fdividef(2.0f, e.w);  // e.w >= 0
    return f * e.v;
}

// rotate x by the unit quaternion (ch, sh * z) (rotation about unit z by 2 atan2(sh, ch))
__device__ __forceinline__ V3 rotate_half(V3 z, float sh, float ch, V3 x) {
    const V3 u = sh * z;
    const V3 t = 2.0f * cross(u, x);
    return x + fma3(ch, t, cross(u, t));
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Per-device values looked up once (host threads may launch concurrently: the
// serving scheduler and callers; a process may drive several devices).
constexpr int kMaxDevices = 64;

inline int current_device() {
    int dev = 0;
    cudaGetDevice(&dev);
    return dev;
}

// SM count of the current device.
inline int sm_count() {
    static std::atomic<int> sms[kMaxDevices];
    const int dev = current_device();
    const int i = dev >= 0 && dev < kMaxDevices ? dev : 0;
    int v = sms[i].load(std::memory_order_relaxed);
    if (v <= 0) {
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        if (v <= 0) v = 1;
        sms[i].store(v, std::memory_order_relaxed);
    }
    return v;
}

// A kernel's dynamic shared-memory limit, raised once per device, at the kernel's first launch
// there, to the most any launch of it takes (clamped to what the device allows beside the
// kernel's static shared memory).  Raising it later, when a launch first needed more than 48 KB,
// made that launch fail ("invalid argument") while smaller launches of the kernel were running
// on other streams.  Under a lock: host threads may launch concurrently.
struct SmemLimit {
    std::mutex mu;
    bool set[kMaxDevices] = {};
};

template <typename K>
inline void allow_dyn_smem(K kernel, SmemLimit& lim, size_t most) {
    const int dev = current_device();
    const int i = dev >= 0 && dev < kMaxDevices ? dev : 0;
    std::lock_guard<std::mutex> g(lim.mu);
    if (lim.set[i] && i == dev) return;
    lim.set[i] = true;
    if (most <= 48 * 1024) return;
    int optin = 0;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    cudaFuncGetAttributes(&fa, kernel);
    const size_t cap = optin > (int)fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : most;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(most < cap ? most : cap));
}

// The launches of a solve follow one another on its stream, each waiting for the one before.  Those
// of small batches are short enough for a launch's own latency to count: they are made with
// launch_next, which lets a kernel's CTAs be set up while the one before still runs.  Such a kernel
// calls grid_follow() before it touches memory: that waits until the grids before are complete and
// their writes visible, so the order is that of plain launches, and then lets the next one be set up.
// (One target, 64 seeds: 131 -> 124 us end to end; 1000 seeds and a scene, seven launches: 181 -> 170.
// The first launch of a solve and the kernels of large batches gain nothing by it.)
__device__ __forceinline__ void grid_follow() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename Arg, typename... Args>
inline void launch_next(void (*kernel)(Arg, Args...), dim3 grid, int block, size_t smem, cudaStream_t st, Arg a,
                        Args... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, a, args...);
}

// Grid for a grid-stride kernel: one thread (or warp) per item, capped at
// `per_sm` blocks per SM.

inline int grid_for(int64_t items, int per_block, int per_sm = 64) {
    int64_t b = (items + per_block - 1) / per_block;
    const int64_t cap = (int64_t)sm_count() * per_sm;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

// ----------------------------------------------------------------------------
// per-target selection.  A candidate's key is 32 bits (a non-negative score orders like its IEEE
// bit pattern; ties go to the lower candidate) and the order of the first `want` of a target's M
// keys is found by one bucket pass in shared memory: the keys' range is cut into up to kMaxBins
// equal bins, the candidates are gathered by bin, and a candidate's rank is its bin's start plus
// its rank among the few that share the bin.  The work is linear while the bins are short (a
// whole sort of 1024 keys took 55 barriers, this takes eight).  The ranked filter's time with its
// sort -> with this: one target of 1000 candidates 27 -> 21 us, 1000 targets 153 -> 119 us, 2000
// targets of 4096 candidates 1281 -> 824 us.
//
// Keys that crowd a bin would cost their square: equal scores (every seed of an invalid target scores
// infinity, so a padding row of a batch does that), a few distinct ones, or scores squeezed together by
// keys far away.  The bins therefore span the ordinary keys only (finite and non-negative; not the NaN
// of the top-K, not the ranking's class 1) where those hold every wanted rank, and where the comparisons
// within the bins that hold wanted ranks would take longer than sorting these bins' keys (crowd_limit), a radix
// sort does that.  The top quarter of 8192 scores, 600 targets: spread 445 us, all equal 268 (by their
// square 9460), 20% NaN 451.  16 targets of 8192 seeds, eight of them padding rows: a solve 5340 -> 684 us.

constexpr uint32_t kNoKey32 = 0xffffffffu;  // never ranked
constexpr int kMaxBins = 2048;

__device__ __forceinline__ uint32_t score_bits(float s) {
    return __float_as_uint(s + 0.0f);  // -0 -> +0
}

// Up to this many keys are ranked by counting, without the bucket pass' seven barriers (64 keys: the
// selection and the ranking of a solve 1.5 us less each, end to end 125 -> 122 us; the comparisons
// grow with the square, and at 256 keys they are the longer way).  COUNT = false leaves that out, for
// the collision-aware ranking, whose registers it takes past 80 and so a third CTA off each SM.
constexpr int kCountKeys = 128;
// Comparisons that take as long as the sort, which costs about 6 us and 1.7 ns a key (measured with one
// CTA per SM; a comparison takes 36 ps)
__device__ __forceinline__ uint32_t crowd_limit(int M) { return 160000u + 48u * (uint32_t)M; }
constexpr uint32_t kOrdinary = 0x7f800000u;  // keys below are finite non-negative scores (of class 0)

// bins of a pass over M keys
__host__ __device__ __forceinline__ int bucket_bins(int M) {
    int bins = 32;
    while (bins < M && bins < kMaxBins) bins <<= 1;
    return bins;
}
// Shared memory of the bucket pass for up to M keys.
__host__ __device__ __forceinline__ size_t bucket_smem_bytes(int M) {
    const size_t m = M > 0 ? M : 1;
    return sizeof(uint32_t) * (m + bucket_bins((int)m) + 36) + sizeof(uint16_t) * 2 * ((m + 1) / 2 * 2);
}
struct Bucket {
    int bins;
    uint32_t* key;    // [M]: written by the caller
    uint32_t* bin;    // [bins]
    uint32_t* tmp;    // [36]
    uint16_t* slot;   // [M]
    uint16_t* order;  // [M]: the candidates of the first `want` ranks
};
__device__ __forceinline__ Bucket bucket_of(void* smem, int M) {
    Bucket B;
    B.bins = bucket_bins(M);
    B.key = reinterpret_cast<uint32_t*>(smem);
    B.bin = B.key + M;
    B.tmp = B.bin + B.bins;
    B.slot = reinterpret_cast<uint16_t*>(B.tmp + 36);
    B.order = B.slot + (M + 1) / 2 * 2;
    return B;
}

// The crowded case of bucket_order: a radix sort of the `count` candidates whose key lies in [lo, lo + top]
// by key and then index.  Each pass takes a digit; a warp ranks its contiguous part of the
// sequence 32 at a time by matching digits, so the order is stable and the time does not depend on
// the keys.  (Digits of up to 8 bits, as the warps' counts fit the bins' memory; equal keys take one
// pass.)  Not inlined: it is rarely taken, and the callers' registers and code stay as they are.
__device__ __forceinline__ void bucket_sort(const Bucket B, int M, int count, uint32_t lo, uint32_t top) {
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, W = nth >> 5;
    int D = 8;
    while ((W << D) > 2 * B.bins || (1 << D) > nth) --D;
    const int R = 1 << D, span = 32 - __clz(top);
    uint16_t* const mine = reinterpret_cast<uint16_t*>(B.bin) + warp * R;  // [warp][digit]
    uint16_t *src = B.slot, *dst = B.order;
    int shift = 0;
    do {
        const bool first = shift == 0;  // the candidates in index order, the others left out
        const int n = first ? M : count;
        const int part = ((n + W - 1) / W + 31) & ~31, p0 = min(n, warp * part), p1 = min(n, p0 + part);
        // this lane's candidate at p and its digit (R: none)
        auto digit = [&](int p, int& cand) {
            cand = p < p1 ? (first ? p : (int)src[p]) : 0;
            const uint32_t k = p < p1 ? B.key[cand] : kNoKey32;
            return k != kNoKey32 && k - lo <= top ? (int)((k - lo) >> shift & (uint32_t)(R - 1)) : R;
        };
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < W * R; i += nth) reinterpret_cast<uint16_t*>(B.bin)[i] = 0;
        __syncthreads();
#pragma unroll 1
        for (int p = p0 + lane; p - lane < p1; p += 32) {
            int cand;
            const int d = digit(p, cand);
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            if (d < R && lane == __ffs(peers) - 1) mine[d] += (uint16_t)__popc(peers);
            __syncwarp();
        }
        __syncthreads();
        // where each warp's candidates of a digit begin
        uint16_t* const col = reinterpret_cast<uint16_t*>(B.bin) + tid;
        uint32_t sum = 0;
        if (tid < R)
#pragma unroll 1
            for (int w = 0; w < W; ++w) {
                const uint32_t v = col[w * R];
                col[w * R] = (uint16_t)sum;
                sum += v;
            }
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) B.tmp[warp] = inc;
        __syncthreads();
        uint32_t at = inc - sum;
#pragma unroll 1
        for (int w = 0; w < warp; ++w) at += B.tmp[w];
        if (tid < R)
#pragma unroll 1
            for (int w = 0; w < W; ++w) col[w * R] = (uint16_t)(col[w * R] + at);
        __syncthreads();
#pragma unroll 1
        for (int p = p0 + lane; p - lane < p1; p += 32) {
            int cand;
            const int d = digit(p, cand);
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const int to = d < R ? mine[d] + __popc(peers & ((1u << lane) - 1u)) : 0;
            __syncwarp();
            if (d < R && lane == __ffs(peers) - 1) mine[d] += (uint16_t)__popc(peers);
            if (d < R) dst[to] = (uint16_t)cand;
            __syncwarp();
        }
        uint16_t* const t = src;
        src = dst;
        dst = t;
        shift += D;
    } while (shift < span);
    __syncthreads();
    if (src != B.order) {
#pragma unroll 1
        for (int i = tid; i < count; i += nth) B.order[i] = src[i];
        __syncthreads();
    }
}

// B.order[r] for r < min(want, returned) from B.key[0, M) (visible to the whole CTA when it is
// called); returns the number of keys other than kNoKey32.  All threads of the CTA take part
// (a multiple of 32, at most 1024); ends with a barrier.
template <bool COUNT = true>
__device__ __forceinline__ int bucket_order(const Bucket& B, int M, int want) {
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5;
    if (COUNT && M <= kCountKeys) {  // every key against every other, four threads a key
        int valid = 0;
        for (int i0 = 0; i0 < max(M, 1); i0 += nth / 4) {
            const int i = i0 + tid / 4;
            const uint32_t k = i < M ? B.key[i] : kNoKey32;
            int r = 0;
            valid = 0;
            for (int j = tid & 3; j < M; j += 4) {
                const uint32_t kj = B.key[j];
                r += kj < k || (kj == k && j < i);
                valid += kj != kNoKey32;
            }
            r += __shfl_xor_sync(0xffffffffu, r, 1);
            r += __shfl_xor_sync(0xffffffffu, r, 2);
            valid += __shfl_xor_sync(0xffffffffu, valid, 1);
            valid += __shfl_xor_sync(0xffffffffu, valid, 2);
            if ((tid & 3) == 0 && k != kNoKey32 && r < want) B.order[r] = (uint16_t)i;
        }
        __syncthreads();
        return valid;
    }
    const int bins = B.bins;
    // range and number of the keys; of the ordinary ones
    uint32_t lo = kNoKey32, hi = 0, hi0 = 0, cnt = 0;  // (cnt: two halves)
    for (int i = tid; i < M; i += nth) {
        const uint32_t k = B.key[i];
        if (k != kNoKey32) {
            lo = min(lo, k);
            hi = max(hi, k);
            hi0 = k < kOrdinary ? max(hi0, k) : hi0;
            cnt += k < kOrdinary ? 0x10001u : 1u;
        }
    }
    for (int i = tid; i < bins; i += nth) B.bin[i] = 0;
    if (tid < 4) B.tmp[32 + tid] = tid == 0 ? kNoKey32 : 0u;
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    hi0 = __reduce_max_sync(0xffffffffu, hi0);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0 && cnt) {
        atomicMin(&B.tmp[32], lo);
        atomicMax(&B.tmp[33], hi);
        atomicMax(&B.tmp[34], hi0);
        atomicAdd(&B.tmp[35], cnt);
    }
    __syncthreads();
    lo = B.tmp[32];
    const int valid = (int)(B.tmp[35] & 0xffffu);
    hi = want <= (int)(B.tmp[35] >> 16) ? B.tmp[34] : B.tmp[33];  // (keys above share the last bin)
    const int span = valid ? 32 - __clz(hi - lo) : 0;  // bits of the range
    const int shift = max(0, span - (31 - __clz(bins)));
    auto bin_of = [&](uint32_t k) { return min((k - lo) >> shift, (uint32_t)bins - 1u); };
    // bin sizes, their starts (an exclusive scan: a run of bins per thread)
    for (int i = tid; i < M; i += nth) {
        const uint32_t k = B.key[i];
        if (k != kNoKey32) atomicAdd(&B.bin[bin_of(k)], 1u);
    }
    __syncthreads();
    const int per = (bins + nth - 1) / nth, b0 = min(bins, tid * per), b1 = min(bins, b0 + per);
    uint32_t sum = 0;
    for (int i = b0; i < b1; ++i) sum += B.bin[i];
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) B.tmp[warp] = inc;
    if (tid < 3) B.tmp[32 + tid] = 0;
    __syncthreads();
    uint32_t at = inc - sum;
    for (int w = 0; w < warp; ++w) at += B.tmp[w];
    uint32_t pairs = 0, last = 0, end = 0;  // comparisons in the bins with a wanted rank; the last such bin, its end
    for (int i = b0; i < b1; ++i) {
        const uint32_t v = B.bin[i];
        B.bin[i] = at;
        if (v && (int)at < want) {
            pairs += v * v;
            last = i;
            end = at + v;
        }
        at += v;
    }
    if (end) {
        atomicAdd(&B.tmp[32], pairs);
        atomicMax(&B.tmp[33], last);
        atomicMax(&B.tmp[34], end);
    }
    __syncthreads();
    if (B.tmp[32] > crowd_limit(M)) {
        last = B.tmp[33];  // (keys past the range share the last bin)
        bucket_sort(B, M, (int)B.tmp[34], lo, (int)last < bins - 1 ? ((last + 1u) << shift) - 1u : kNoKey32 - 1u - lo);
        return valid;
    }
    // the candidates by bin; a bin's entry then holds its end, which is the next one's start
    for (int i = tid; i < M; i += nth) {
        const uint32_t k = B.key[i];
        if (k != kNoKey32) B.slot[atomicAdd(&B.bin[bin_of(k)], 1u)] = (uint16_t)i;
    }
    __syncthreads();
    for (int p = tid; p < valid; p += nth) {
        const int i = B.slot[p];
        const uint32_t k = B.key[i], b = bin_of(k);
        const int s0 = b ? (int)B.bin[b - 1] : 0, s1 = (int)B.bin[b];
        if (s0 >= want) continue;
        int r = s0;
        for (int q = s0; q < s1; ++q) {
            const int j = B.slot[q];
            const uint32_t kj = B.key[j];
            r += kj < k || (kj == k && j < i);
        }
        if (r < want) B.order[r] = (uint16_t)i;
    }
    __syncthreads();
    return valid;
}

// ----------------------------------------------------------------------------
// host-side launch entry points (defined in the kernel translation units)

struct CcdArgs {
    RobotSet rs;
    const TargetDesc* tg;
    CandMap map;
    int64_t C, ld;
    const float* th_in;  // null: sample seeds
    float* th_out;
    float* th_tmp;       // cd_variant = 2: a second [n][ld] buffer
    float *score, *perr, *oerr;
    int32_t* iters;
    int k0, n_iters;  // n_iters < 0: each target's cd_iters
    hjcd_params P;
    hjcd_ccd_trace tr;
    Counters* cnt;
    int32_t block;  // threads (candidates) per CTA: 64, 128 or 256 (anything else: 128; contexts pass 64 by default)
    int32_t seed_base;  // added to each candidate's index inside its target (a shard of the seeds)
    // Iteration segments (no trace, th_out set): this launch runs iterations [seg_begin, seg_end)
    // (seg_end 0: to the cap) of every candidate, or of the candidates list_in[0 .. *n_in) whose
    // state th_out holds; a candidate still iterating at seg_end keeps its state in th_out and is
    // appended to list_out (count *n_out) instead of writing its results.
    int32_t seg_begin, seg_end;
    int32_t in_limits;  // 1: every joint vector the launch reads lies within its robot's limits
    const int32_t* list_in;
    const int32_t* n_in;
    int32_t* list_out;
    int32_t* n_out;
    // null: the items in a grid stride; else a zeroed queue head the warps take items from
    // (cd_variant 0 and 1)
    unsigned long long* queue;
};

struct LmArgs {
    RobotSet rs;
    const TargetDesc* tg;
    CandMap map;
    int64_t C, ld;
    float* th;
    float *score, *perr, *oerr;
    int32_t* iters;
    int k0, n_iters;  // n_iters < 0: each target's lm_iters
    hjcd_params P;
    hjcd_lm_trace tr;
    Counters* cnt;
    unsigned long long* queue;  // candidate queue head, zero at launch
    int32_t warps;  // warps per CTA: 2, 4 or 8 (anything else: 8, the contexts' default)
    int32_t in_limits;  // 1: every joint vector the launch reads lies within its robot's limits
    // Where a launch leaves the candidates that need more than its first iterations to the next one
    // (null: nowhere): their indices and iteration counts [C] and how many there are (zero at launch).
    // hand_at (set by launch_lm; 0: never): the iteration after which it does, at the earliest, hand_lim: how
    // many unfinished candidates it leaves at most (one lane per candidate), n_done: how many are finished
    // (zero at launch).
    int32_t* list;
    int32_t* list_k;
    int32_t* n_list;
    int32_t* n_done;
    int32_t hand_at, hand_lim;
};

struct DupArgs {
    RobotSet rs;
    const TargetDesc* tg;
    int32_t T;
    const int64_t* m_off;
    const float* score_M;
    const float* th_M;
    int64_t ld_M;
    const int64_t* b_off;
    float* th_B;
    int64_t ld_B;
    int32_t* src_B;
    int32_t ratio;
    float sigma;
};

// Where a wave's target comes from and where its results go: its pose and reference configuration
// (device or pinned host memory; null: no reference) and its blocks of the outputs (the caller's device
// memory, the workspace, or the wave's pinned buffer).
struct TargetIo {
    const float* pose;  // [7]
    const float* ref;   // [n]
    float* q;           // [top_k][n]
    float* err;         // [top_k][2]
    int32_t* count;
};

// Output of target t: to io[t], or with io null in contiguous blocks in target order (top_k rows of
// its robot's n, top_k pairs of errors); the rows past its count are filled with NaN.  With tg null
// every target takes top_k and robot 0.
struct RankArgs {
    RobotSet rs;
    const TargetDesc* tg;
    int32_t T;
    const int64_t* b_off;
    const float* th;
    int64_t ld;
    const float *score, *perr, *oerr;
    const uint8_t* hit;
    int top_k;
    const TargetIo* io;
    float* out_q;
    float* out_err;
    int32_t* out_count;
    // with q_ref set ([T][ld_ref], target t's reference configuration in row t): the candidates
    // within the target's tolerances come first, nearest to the reference (squared joint
    // distance), then the others by score
    const float* q_ref;
    int32_t ld_ref;
    // with list set: block b ranks target list[b] when b < *n_list, else nothing (the targets
    // that the bounded lazy pass left unfinished); k_rank_lazy appends those targets here
    int32_t* list;
    int32_t* n_list;
    // tolerances of every target when tg is null (with tg: each target row's own)
    float eps_pos, eps_ori;
};

// Target t's output blocks
struct RankOut {
    float* q;
    float* err;
    int32_t* count;
};
__device__ __forceinline__ RankOut rank_out(const RankArgs& A, int t, int top_k, int n) {
    if (A.io) {
        const TargetIo io = A.io[t];
        return RankOut{io.q, io.err, io.count};
    }
    return RankOut{A.out_q + (int64_t)t * top_k * n, A.out_err + (int64_t)t * top_k * 2, A.out_count + t};
}

// Ranking key of candidate i of target t (candidates [b0, b0 + B), robot DoF
// n), never for a colliding candidate (with use_hit) or a non-finite score.
// Reading c20 of Alg. 2's final step: the candidates within the target's
// tolerances (|e_p| <= eps_pos and |omega| <= eps_ori) form class 0, the rest
// class 1 (the top key bit), each class ordered by score and then index.  With
// the target's nearest flag (with tg null: whenever q_ref is set), class 0 is
// ordered by squared joint distance to the reference q_ref[t] instead
// (reading c24).  kNoKey32: not ranked.
__device__ __forceinline__ uint32_t rank_key(const RankArgs& A, int t, int64_t b0, int n, int i, bool use_hit) {
    if (use_hit && A.hit && A.hit[b0 + i]) return kNoKey32;
    const int64_t g = b0 + i;
    const float sc = A.score[g];
    if (!(sc < __int_as_float(0x7f800000))) return kNoKey32;  // finite only
    const float ep = A.tg ? A.tg[t].eps_pos : A.eps_pos, eo = A.tg ? A.tg[t].eps_ori : A.eps_ori;
    const bool conv = A.perr[g] <= ep && A.oerr[g] <= eo;
    const bool nearest = A.q_ref && (!A.tg || (A.tg[t].top_k & kNearestFlag));
    if (conv && nearest) {
        float d2 = 0.0f;
        for (int j = 0; j < n; ++j) {
            const float dj = A.th[j * A.ld + g] - A.q_ref[(int64_t)t * A.ld_ref + j];
            d2 = fmaf(dj, dj, d2);
        }
        return d2 == d2 ? score_bits(d2) : kNoKey32;
    }
    const uint32_t k = score_bits(sc);
    return conv ? k : (k | 0x80000000u);
}

// Collision filter of C candidates.  With tg null or uniform set every
// candidate is robot 0 against scene 0 (if any); otherwise candidate c belongs
// to target row map(c), whose robot and scene it uses (an invalid row: hit).  A launch with a single scene
// stages it into shared memory; with several, obstacles are read from the
// scene tables directly.
struct CollideArgs {
    RobotSet rs;
    const SceneDev* scenes;   // [n_scenes] (device)
    int32_t n_scenes;
    int32_t max_obj4;         // largest n_sph + 2 n_box over the scenes
    int32_t uniform;          // every candidate: robot 0 and scene 0 (if any) -- no per-candidate lookup
    int32_t has_grid;         // some scene of the launch carries a uniform grid
    // with uniform set: robot 0's DoF and checked body pairs, scene 0's obstacle counts (0 without a scene)
    int32_t u_n, u_pairs, u_osph, u_obox;
    const TargetDesc* tg;
    CandMap map;
    int64_t C, ld;
    const float* th;
    uint8_t* hit;
    Counters* cnt;
    int32_t* err_flag;        // set when the bounded wait for the staged tables runs out
    // polls of the first wait for the staged tables (< 0: the kernels' default limit); 0 makes
    // that wait run out at once, which only tests of the timeout path ask for
    int64_t first_wait_polls = -1;
    // with list set: only the candidates of the targets list[0 .. *n_list) whose hit entry is 2
    // are checked, item i = (list entry i / list_bmax, candidate i % list_bmax of that target's
    // b_off range)
    const int32_t* list;
    const int32_t* n_list;
    const int64_t* b_off;
    int32_t list_bmax;
};

// Per target t: the K = max(1, floor(M_full / ratio)) lowest scores of its
// candidates [off[t], off[t+1]) (ties to the lower index), written as score,
// seed index (seed_base + index in the target) and joint vector; +inf / -1
// past the candidates.  out_th [T][K][ld_n], out_s / out_i [T][K].
struct ShardTopkArgs {
    RobotSet rs;
    const TargetDesc* tg;
    int32_t T, K, seed_base;
    const int64_t* off;
    const float* score;
    const float* th;
    int64_t ld;
    float* out_s;
    int32_t* out_i;
    float* out_th;
    int32_t ld_n;
};
void launch_shard_topk(const ShardTopkArgs& A, int max_m, cudaStream_t st);

// Per target: the K best of L lists of K (score, seed index, joint vector),
// ties to the lower seed index.
struct MergeArgs {
    int32_t T, L, K, n;
    const float* in_s;   // [L][T][K]
    const int32_t* in_i; // [L][T][K]
    const float* in_th;  // [L][T][K][n]
    float* out_s;
    int32_t* out_i;
    float* out_th;       // [T][K][n]
};
void launch_topk_merge(const MergeArgs& A, cudaStream_t st);

// Alg. 2's duplication from kept seeds given per target ([T][K][n], best first):
// copy r of seed i at index r K + i, perturbed as in k_topk_dup.
struct KeptDupArgs {
    RobotSet rs;
    const TargetDesc* tg;
    int32_t T, K;
    const float* kept;   // [T][K][n]
    const int64_t* b_off;
    float* th_B;
    int64_t ld_B;
    float sigma;
};
void launch_dup_kept(const KeptDupArgs& A, cudaStream_t st);

// First launch of a wave: copies the head's image (`bytes`, a multiple of 16, both sides 16-byte
// aligned) from pinned host memory to the workspace, fills in the target rows' poses and the
// reference configurations, zeroes the wave's queue heads and error flag.
struct WaveInitArgs {
    const char* pin;  // the image
    char* ws;
    size_t bytes, o_tg, o_io, o_rp;  // the head's size; target rows, TargetIo rows and robot tables inside it
    int32_t T;
    float* ref;       // [T][ld_ref], or null
    int32_t ld_ref;
    unsigned long long* zero;  // 7 words
    int32_t* flag;
};
void launch_wave_init(const WaveInitArgs& A, cudaStream_t st);
// Target rows of [T][7] poses: tmpl with t_local counting up from its own.
void launch_pack_targets(const float* pq7, int T, const TargetDesc& tmpl, TargetDesc* out, cudaStream_t st);
void launch_fk(const RobotParams& R, int64_t C, const float* th, int64_t ld, float* out, cudaStream_t st);
void launch_sample(const RobotParams& R, uint64_t seed, CandMap map, int64_t C, float* th, int64_t ld,
                   cudaStream_t st);
void launch_ccd(const CcdArgs& A, bool trace, cudaStream_t st);
int launch_lm(const LmArgs& A, bool trace, cudaStream_t st);  // the number of launches
// What an untraced launch makes of the context's candidates per CTA / warps per CTA: 0 where it takes
// a kernel that does not use them (no pointer of A but `list` is looked at).
int ccd_block_used(const CcdArgs& A, int asked);
int lm_warps_used(const LmArgs& A, int asked);
void launch_topk_dup(const DupArgs& A, int max_m, cudaStream_t st);
void launch_rank(const RankArgs& A, int max_b, cudaStream_t st);
void launch_collide(const CollideArgs& A, cudaStream_t st);
// The ranking with the collision filter applied lazily (k_rank_lazy); false
// when it does not apply (no spheres, no target rows, or too large for shared
// memory): use launch_collide + launch_rank.  With R.list set, a target whose
// first `depth` ranked candidates hold fewer than top_k collision-free ones is
// appended to R.list instead of ranked; launch_collide and launch_rank with
// that list finish those targets.
bool launch_rank_lazy(const CollideArgs& A, const RankArgs& R, int max_b, int depth, cudaStream_t st);
void launch_contacts(const RobotParams& R, const RobotDev& rd, const SceneDev& sc, const int32_t* perm, int64_t C,
                     const float* th, int64_t ld, uint8_t* touched, cudaStream_t st);
void launch_ffma(float* sink, int iters, int blocks, cudaStream_t st);
void launch_philox(int64_t n, const uint32_t* ctr, uint64_t key, uint32_t* out, cudaStream_t st);
int ffma_flops_per_thread_iter();

}  // namespace hjcd
