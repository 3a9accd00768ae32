// k_collide.cu -- sphere collision filter (Sec. V-C), one warp per candidate, or one lane per
// candidate for large sets (k_collide_lane, below).
//
// Two levels, as in the paper's coarse-then-fine check: every body carries a
// bounding sphere of its link spheres, and a body's fine spheres are tested
// against an obstacle (or another body's spheres) only when the bounding
// spheres overlap.  The bounding radii are padded beyond binary32 rounding, so
// the verdict is the brute-force verdict over all fine pairs.
//
// Per candidate: every lane walks the kinematic chain and moves its own fine
// spheres (sphere lane + 32 q of the body-grouped table) and, on lane b, the
// bounding sphere of body b into the world frame; the warp publishes them to
// shared memory.  Self pairs: lanes over the checked body pairs for the
// bounding test; the fine sphere pairs of each overlapping body pair are
// spread over the warp.  Obstacles: lanes over obstacles (32 at a time) for
// the bounding test of one body; the overlapping obstacles are compacted into
// a list and their fine tests (list x the body's spheres) spread over the
// warp.  The warp stops at the first overlap.  When the launch has a single
// scene, its obstacles (spheres, then boxes) are staged once per CTA into
// shared memory by one bulk asynchronous copy (TMA, cp.async.bulk) completing
// on an mbarrier; a launch mixing scenes reads each candidate's obstacles from
// its scene table.  Each candidate uses its target's robot: the kinematic
// tables of the launch's robots sit in shared memory, a warp reloads its
// lanes' link spheres when its candidate's robot changes.
//
// Overlap: |c1 - c2|^2 < (r1 + r2)^2 for spheres; for a box, the squared
// distance from the centre to its clamp into the box below r^2.
#include <algorithm>

#include "hjcd_internal.cuh"

namespace hjcd {

namespace {

constexpr int kWarpsPerBlock = 8;
constexpr int kMaxStagedObj4 = 10240;  // obstacle float4s staged in shared memory (160 KB)
constexpr uint32_t kWaitLimit = 1u << 22;  // try_wait polls before the staged tables are given up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bulk global -> shared copy; both addresses 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t limit = kWaitLimit) {
    for (uint32_t i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// an obstacle: from shared memory (staged scene) or through the read-only cache
template <bool STAGED>
__device__ __forceinline__ float4 ld_obj(const float4* p, int i) {
    if (STAGED) return p[i];
    return __ldg(p + i);
}

__device__ __forceinline__ float4 to_world(const Frame& F, float4 s) {
    const V3 w = fma3(s.z, F.c2, fma3(s.y, F.c1, fma3(s.x, F.c0, F.p)));
    return make_float4(w.x, w.y, w.z, s.w);
}

// to_world by the frame of lane src
__device__ __forceinline__ float4 to_world_of(const Frame& F, int src, float4 s) {
    auto of = [&](const V3 v) {
        return v3(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src), __shfl_sync(0xffffffffu, v.z, src));
    };
    const V3 w = fma3(s.z, of(F.c2), fma3(s.y, of(F.c1), fma3(s.x, of(F.c0), of(F.p))));
    return make_float4(w.x, w.y, w.z, s.w);
}

__device__ __forceinline__ bool sph_sph(float4 a, float4 b) {
    const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z, rr = a.w + b.w;
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < rr * rr;
}

__device__ __forceinline__ bool sph_box(float4 a, float4 lo, float4 hi) {
    const float dx = a.x - clampf(a.x, lo.x, hi.x);
    const float dy = a.y - clampf(a.y, lo.y, hi.y);
    const float dz = a.z - clampf(a.z, lo.z, hi.z);
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < a.w * a.w;
}

// shared-memory layout of a CTA: staged obstacles, mbarrier, robot tables,
// then per warp the world-frame fine spheres, bounding spheres and a list
struct CollideLayout {
    uint32_t bar, robots, warp, warp_bytes, total;
};

// per warp: world fine spheres [ns], world bounding spheres [nb], the robot's
// body ranges [nb] and checked body pairs [n_pairs], a list of 32 indices
__host__ __device__ __forceinline__ CollideLayout collide_smem_layout(int n_obj4, int n_robots, int nb, int ns,
                                                                      int n_pairs) {
    CollideLayout L;
    L.bar = 16u * (uint32_t)n_obj4;
    L.robots = L.bar + 16u;
    L.warp = L.robots + (uint32_t)robots_smem_bytes(n_robots);
    L.warp_bytes = (16u * (uint32_t)(ns + nb) + 8u * (uint32_t)(nb + n_pairs) + 4u * 32u + 15u) / 16u * 16u;
    L.total = L.warp + kWarpsPerBlock * L.warp_bytes;
    return L;
}


// The warp's current robot: its lanes' link spheres (body frame) and bodies, the
// bounding sphere of body `lane`, DoF, checked pairs and the bodies that carry spheres.
template <int SPL>
struct WarpRobot {
    float4 ls[SPL];
    int lb[SPL];
    float4 lco;
    int cur, n_m, pairs_m;
    unsigned bmask;
};

// The warp's shared-memory buffers: world fine spheres, world bounding spheres,
// the robot's body ranges and checked pairs, a list of 32 indices.
struct WarpBufs {
    float4* wsph;
    float4* wco;
    int2* wrange;
    int2* wpairs;
    int* list;
};

// Makes robot rid the warp's current one.
template <int SPL>
__device__ __forceinline__ void warp_robot(const CollideArgs& A, const RobotParams* rob, WarpRobot<SPL>& W,
                                           const WarpBufs& Bf, int rid) {
    const int lane = threadIdx.x & 31;
    W.cur = rid;
    const RobotDev rd = A.rs.rd[rid];
    W.n_m = rob[rid].n;
    W.pairs_m = rd.n_pairs;
    const int ns = rd.n_sph, nbr = W.n_m + 2;
#pragma unroll
    for (int q = 0; q < SPL; ++q) {
        const int i = lane + 32 * q;
        W.lb[q] = i < ns ? __ldg(rd.body + i) : -1;
        W.ls[q] = i < ns ? __ldg(rd.sph + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    W.lco = lane < nbr ? __ldg(rd.coarse + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
    for (int i = lane; i < nbr; i += 32) Bf.wrange[i] = __ldg(rd.range + i);
    for (int i = lane; i < W.pairs_m; i += 32) Bf.wpairs[i] = __ldg(rd.pairs + i);
    __syncwarp();
    W.bmask = __ballot_sync(0xffffffffu, lane < nbr && Bf.wrange[lane].y > 0);  // bodies with spheres
}

// Collision verdict of candidate c (robot row rid, scene row sid, -1: none),
// warp-uniform; t_s / t_b accumulate the sphere and box tests.
template <int SPL, bool UNIFORM, bool GRID>
__device__ __forceinline__ bool warp_collides(const CollideArgs& A, const RobotParams* rob, const SceneDev& sc0,
                                              const float4* s_scene, WarpRobot<SPL>& W, const WarpBufs& Bf, int64_t c,
                                              int rid, int sid, unsigned long long& t_s, unsigned long long& t_b) {
    constexpr bool STAGED = UNIFORM;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    float4* const wsph = Bf.wsph;
    float4* const wco = Bf.wco;
    int2* const wrange = Bf.wrange;
    int2* const wpairs = Bf.wpairs;
    int* const list = Bf.list;
    if (rid != W.cur) warp_robot<SPL>(A, rob, W, Bf, rid);
    const RobotParams& R = rob[rid];
    const int n = UNIFORM ? A.u_n : W.n_m, nb = n + 2, n_pairs = UNIFORM ? A.u_pairs : W.pairs_m;
    // obstacles: the staged copy (shared memory) or the scene's table (global, read-only path)
    const float4* obj = s_scene;
    int n_osph = 0, n_obox = 0;
    if (UNIFORM) {
        n_osph = A.u_osph;
        n_obox = A.u_obox;
    } else if (sid >= 0) {
        const SceneDev sd = A.scenes[sid];
        obj = sd.obj;
        n_osph = sd.n_sph;
        n_obox = sd.n_box;
    }

    // world frame: body 0 is the base (identity)
    float4 ws[SPL];
#pragma unroll
    for (int q = 0; q < SPL; ++q) ws[q] = W.ls[q];
    float4 wc = W.lco;
    Frame F = frame_identity();
    // a lane loads and reduces one joint's angle; the chain then takes them in turn (a load per joint
    // inside the chain made it wait for each: ranking of 1000 targets x 1000 189 us, so 155)
    float sj = 0.0f, cj = 1.0f;
    if (lane < n) sincos_red(A.th[lane * A.ld + c] + R.off[lane], &sj, &cj);
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        fk_step_cs(R, j, __shfl_sync(0xffffffffu, cj, j), __shfl_sync(0xffffffffu, sj, j), F);
#pragma unroll
        for (int q = 0; q < SPL; ++q)
            if (W.lb[q] == j + 1) ws[q] = to_world(F, W.ls[q]);
        if (lane == j + 1) wc = to_world(F, W.lco);
    }
    const Frame E = fk_flange(R, F);
#pragma unroll
    for (int q = 0; q < SPL; ++q) {
        if (W.lb[q] == n + 1) ws[q] = to_world(E, W.ls[q]);
        if (W.lb[q] >= 0) wsph[lane + 32 * q] = ws[q];
    }
    if (lane == n + 1) wc = to_world(E, W.lco);
    if (lane < nb) wco[lane] = wc;
    __syncwarp();

    bool hit = false;

    // self-collision: bounding test per checked body pair, fine pairs spread over the warp
    for (int p0 = 0; p0 < n_pairs && !hit; p0 += 32) {
        const int p = p0 + lane;
        int2 pr = make_int2(0, 0);
        bool ch = false;
        if (p < n_pairs) {
            pr = wpairs[p];
            ch = sph_sph(wco[pr.x], wco[pr.y]);
        }
        t_s += (unsigned long long)min(32, n_pairs - p0);
        unsigned m = __ballot_sync(0xffffffffu, ch);
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1u;
            const int ba = __shfl_sync(0xffffffffu, pr.x, src), bb = __shfl_sync(0xffffffffu, pr.y, src);
            const int2 ra = wrange[ba], rb = wrange[bb];
            const int items = ra.y * rb.y;
            bool h = false;
            for (int w = lane; w < items; w += 32) {
                const int i = w / rb.y;
                h |= sph_sph(wsph[ra.x + i], wsph[rb.x + (w - i * rb.y)]);
            }
            t_s += (unsigned long long)items;
            if (__any_sync(0xffffffffu, h)) {
                hit = true;
                break;
            }
        }
    }

    // obstacle spheres of a gridded scene: per body, the lanes walk the cells within the
    // bounding sphere's radius plus the largest obstacle radius; each obstacle that
    // overlaps the bounding sphere is tested against the body's fine spheres
    const int32_t* gcell = nullptr;
    if (GRID && n_osph > 0) gcell = (UNIFORM ? sc0 : A.scenes[sid]).cell;
    if (GRID && gcell) {
        const SceneDev& G = A.scenes[UNIFORM ? 0 : sid];
        for (int b = 0; b < nb && !hit; ++b) {
            const int2 rg = wrange[b];
            if (rg.y == 0) continue;
            const float4 co = wco[b];
            const float ext = co.w + G.reach;
            const float cc[3] = {co.x, co.y, co.z};
            int i0[3], i1[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int dmax = G.dim[k] - 1;
                i0[k] = min(max((int)floorf((cc[k] - ext - G.lo[k]) * G.inv_h), 0), dmax);
                i1[k] = min(max((int)floorf((cc[k] + ext - G.lo[k]) * G.inv_h), 0), dmax);
            }
            const int nx = i1[0] - i0[0] + 1, ny = i1[1] - i0[1] + 1, nxy = nx * ny;
            const int ncell = nxy * (i1[2] - i0[2] + 1);
            bool h = false;
            unsigned tl = 0;
            for (int q = lane; q < ncell && !h; q += 32) {
                const int z = q / nxy, r = q - z * nxy, y = r / nx, x = r - y * nx;
                const int k = (i0[0] + x) + G.dim[0] * ((i0[1] + y) + G.dim[1] * (i0[2] + z));
                const int a = __ldg(gcell + k), e = __ldg(gcell + k + 1);
                for (int o = a; o < e && !h; ++o) {
                    const float4 sp = ld_obj<STAGED>(obj, o);
                    ++tl;
                    if (sph_sph(co, sp)) {
                        for (int i = 0; i < rg.y && !h; ++i) h = sph_sph(wsph[rg.x + i], sp);
                        tl += rg.y;
                    }
                }
            }
            t_s += __reduce_add_sync(0xffffffffu, tl);
            hit = __any_sync(0xffffffffu, h);
        }
    }

    // obstacle spheres, 32 at a time: each lane tests its obstacle against every body's
    // bounding sphere (a bit per body); only bodies some obstacle overlaps are visited, their
    // overlapping obstacles compacted and the fine tests spread over the warp
    const int nbs = __popc(W.bmask);
    for (int o0 = 0; o0 < n_osph && !hit && !(GRID && gcell); o0 += 32) {
        const int o = o0 + lane;
        const bool valid = o < n_osph;
        const float4 s = valid ? ld_obj<STAGED>(obj, o) : make_float4(0.f, 0.f, 0.f, 0.f);
        unsigned bm = 0;
        if (valid)
            for (unsigned bb = W.bmask; bb; bb &= bb - 1u) {
                const int b = __ffs(bb) - 1;
                if (sph_sph(wco[b], s)) bm |= 1u << b;
            }
        t_s += (unsigned long long)min(32, n_osph - o0) * nbs;
        for (unsigned todo = __reduce_or_sync(0xffffffffu, bm); todo && !hit; todo &= todo - 1u) {
            const int b = __ffs(todo) - 1;
            const int2 rg = wrange[b];
            const bool ch = (bm >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, ch);
            if (ch) list[__popc(m & lt)] = o;
            __syncwarp();
            const int items = __popc(m) * rg.y;
            bool h = false;
            for (int w = lane; w < items; w += 32) {
                const int k = w / rg.y;
                h |= sph_sph(wsph[rg.x + (w - k * rg.y)], ld_obj<STAGED>(obj, list[k]));
            }
            t_s += (unsigned long long)items;
            hit = __any_sync(0xffffffffu, h);
            __syncwarp();
        }
    }

    // obstacle boxes, the same way
    const float4* box = obj + n_osph;
    for (int o0 = 0; o0 < n_obox && !hit; o0 += 32) {
        const int o = o0 + lane;
        const bool valid = o < n_obox;
        const float4 lo = valid ? ld_obj<STAGED>(box, 2 * o) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 hi = valid ? ld_obj<STAGED>(box, 2 * o + 1) : lo;
        unsigned bm = 0;
        if (valid)
            for (unsigned bb = W.bmask; bb; bb &= bb - 1u) {
                const int b = __ffs(bb) - 1;
                if (sph_box(wco[b], lo, hi)) bm |= 1u << b;
            }
        t_b += (unsigned long long)min(32, n_obox - o0) * nbs;
        for (unsigned todo = __reduce_or_sync(0xffffffffu, bm); todo && !hit; todo &= todo - 1u) {
            const int b = __ffs(todo) - 1;
            const int2 rg = wrange[b];
            const bool ch = (bm >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, ch);
            if (ch) list[__popc(m & lt)] = o;
            __syncwarp();
            const int items = __popc(m) * rg.y;
            bool h = false;
            for (int w = lane; w < items; w += 32) {
                const int k = w / rg.y, bo = list[k];
                h |= sph_box(wsph[rg.x + (w - k * rg.y)], ld_obj<STAGED>(box, 2 * bo), ld_obj<STAGED>(box, 2 * bo + 1));
            }
            t_b += (unsigned long long)items;
            hit = __any_sync(0xffffffffu, h);
            __syncwarp();
        }
    }

    return hit;
}

// CTA prologue of the collision kernels: the obstacles of a single scene
// staged by one bulk copy (UNIFORM), the robots' kinematic tables with plain
// loads.  False (error flag set) when the staging wait ran out or the scene
// outgrew the shared memory the host sized; the CTA must return.  `meanwhile`
// runs (all threads, the robots staged) while the copy is under way.
template <bool UNIFORM, class F>
__device__ __forceinline__ bool collide_prologue(const CollideArgs& A, unsigned char* smem, const CollideLayout& L,
                                                 const SceneDev& sc0, int n_obj4, const RobotParams** rob, F&& meanwhile) {
    float4* s_scene = reinterpret_cast<float4*>(smem);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L.bar);
    const uint32_t bytes = 16u * (uint32_t)n_obj4;
    if (UNIFORM) {
        if (threadIdx.x == 0) mbar_init(bar, 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            if (bytes > 0) {
                mbar_arrive_expect_tx(bar, bytes);
                bulk_g2s(s_scene, sc0.obj, bytes, bar);
            } else {
                mbar_arrive(bar);
            }
        }
    }
    *rob = stage_robots(smem + L.robots, A.rs);
    meanwhile();
    if (UNIFORM) {
        const uint32_t polls = A.first_wait_polls < 0 ? kWaitLimit
                               : (uint32_t)(A.first_wait_polls < (int64_t)kWaitLimit ? A.first_wait_polls : kWaitLimit);
        const bool staged = mbar_wait_bounded(bar, 0, polls);
        if (__syncthreads_or(!staged)) {
            // give up: flag the error, give the copy one more bounded wait (the full limit: the
            // copy must land before the CTA's shared memory is released)
            if (threadIdx.x == 0) {
                *(volatile int32_t*)A.err_flag = 1;  // any CTA's will do (may be host memory)
                mbar_wait_bounded(bar, 0);
            }
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ WarpBufs warp_bufs(unsigned char* smem, const CollideLayout& L, const CollideArgs& A) {
    const int nb_max = A.rs.n_max + 2;
    unsigned char* wb = smem + L.warp + (threadIdx.x >> 5) * L.warp_bytes;
    WarpBufs B;
    B.wsph = reinterpret_cast<float4*>(wb);
    B.wco = B.wsph + A.rs.ns_max;
    B.wrange = reinterpret_cast<int2*>(B.wco + nb_max);
    B.wpairs = B.wrange + nb_max;
    B.list = reinterpret_cast<int*>(B.wpairs + A.rs.pairs_max);
    return B;
}

template <int SPL, bool UNIFORM, bool GRID>
__global__ void __launch_bounds__(kWarpsPerBlock * 32) k_collide(const CollideArgs A) {
    extern __shared__ __align__(128) unsigned char smem[];
    grid_follow();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const SceneDev sc0 = A.n_scenes > 0 ? A.scenes[0] : SceneDev{nullptr, 0, 0};
    const int n_obj4 = UNIFORM ? sc0.n_sph + 2 * sc0.n_box : 0;
    if (n_obj4 > (UNIFORM ? A.max_obj4 : 0)) {  // the scene outgrew the shared memory the host sized
        if (threadIdx.x == 0) *(volatile int32_t*)A.err_flag = 2;  // any CTA's will do (may be host memory)
        return;
    }
    // list mode: the candidates of the listed targets only (none listed: nothing to stage)
    const int64_t items = A.list ? (int64_t)*A.n_list * A.list_bmax : A.C;
    if (items == 0) return;
    const CollideLayout L = collide_smem_layout(n_obj4, A.rs.n, A.rs.n_max + 2, A.rs.ns_max, A.rs.pairs_max);
    const RobotParams* rob;
    if (!collide_prologue<UNIFORM>(A, smem, L, sc0, n_obj4, &rob, [] {})) return;
    const WarpBufs Bf = warp_bufs(smem, L, A);
    const float4* s_scene = reinterpret_cast<const float4*>(smem);

    WarpRobot<SPL> W;
    W.cur = -1;
    W.n_m = W.pairs_m = 0;
    W.bmask = 0;
    unsigned long long tests = 0, btests = 0, ncand = 0;
    const int64_t nwarps = (int64_t)gridDim.x * kWarpsPerBlock;
    int rid = 0, sid = 0;
    bool tvalid = true;
    for (int64_t it = (int64_t)blockIdx.x * kWarpsPerBlock + warp; it < items; it += nwarps) {
        int64_t c = it;
        if (A.list) {
            const int t = A.list[it / A.list_bmax];
            const int j = (int)(it % A.list_bmax);
            const int64_t b0 = A.b_off[t];
            if (j >= A.b_off[t + 1] - b0 || A.hit[b0 + j] != 2) continue;  // not ranked, or checked
            c = b0 + j;
        }
        if (!UNIFORM && A.tg) {
            int32_t t, s;
            tvalid = A.map.lookup(c, t, s);
            if (tvalid) {
                const TargetDesc& Td = A.tg[t];
                rid = Td.robot;
                sid = Td.scene;
                tvalid = Td.eps_pos > 0.0f;
            }
        } else if (!UNIFORM) {
            sid = A.n_scenes > 0 ? 0 : -1;
        }
        if (!tvalid) {  // no such target, or an invalid one: never ranked
            if (lane == 0) A.hit[c] = 1;
            continue;
        }
        unsigned long long t_s = 0, t_b = 0;  // tests of this candidate (uniform over the warp)
        const bool hit = warp_collides<SPL, UNIFORM, GRID>(A, rob, sc0, s_scene, W, Bf, c, rid, sid, t_s, t_b);
        if (lane == 0) {
            A.hit[c] = hit ? 1 : 0;
            tests += t_s;
            btests += t_b;
            ++ncand;
        }
        __syncwarp();
    }
    if (A.cnt && lane == 0) {
        atomicAdd(&A.cnt->v[3], tests);
        atomicAdd(&A.cnt->v[6], btests);
        atomicAdd(&A.cnt->v[4], ncand);
    }
}

// Ranking with the collision filter applied lazily (the top_k collision-free
// candidates by score are the first top_k collision-free ones in score
// order): one CTA per target orders its candidates' keys, then its warps check
// candidates in rank order, one candidate per warp and kWarpsPerBlock at a
// time, until top_k collision-free ones are found or the ranked candidates
// run out.  Same output as the collision filter over all candidates followed
// by k_rank.  A launch of few targets has CTAs of twice the warps, which check
// the next kWarpsPerBlock candidates too in case the first do not settle it; what
// they find counts only then.
// (Registers: three CTAs of 8 warps on an SM, or one of 16.)
constexpr int kRankWarps = 2 * kWarpsPerBlock;
template <int SPL, bool UNIFORM, bool GRID>
__global__ void __maxnreg__(SPL <= 2 ? 80 : 128)
    k_rank_lazy(const CollideArgs A, const RankArgs R, uint32_t keys_off, int depth) {
    extern __shared__ __align__(128) unsigned char smem[];
    grid_follow();
    __shared__ int verdict[kRankWarps];
    __shared__ int picks[HJCD_MAX_TOPK];
    __shared__ int n_found, n_checked;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x;
    const TargetDesc& T = R.tg[t];
    const SceneDev sc0 = A.n_scenes > 0 ? A.scenes[0] : SceneDev{nullptr, 0, 0};
    const int n_obj4 = UNIFORM ? sc0.n_sph + 2 * sc0.n_box : 0;
    const bool outgrown = n_obj4 > (UNIFORM ? A.max_obj4 : 0);
    if (outgrown && threadIdx.x == 0) *(volatile int32_t*)A.err_flag = 2;  // any CTA's will do (may be host memory)
    const CollideLayout L =
        collide_smem_layout(outgrown ? 0 : n_obj4, A.rs.n, A.rs.n_max + 2, A.rs.ns_max, A.rs.pairs_max);
    const RobotParams* rob;
    const int rid = T.robot, sid = UNIFORM ? 0 : T.scene;
    const int64_t b0 = R.b_off[t];
    const int B = (int)(R.b_off[t + 1] - b0);
    const Bucket S = bucket_of(smem + keys_off, B > 0 ? B : 1);
    WarpBufs Bf;
    WarpRobot<SPL> W;
    // the keys and the warps' robot load while the scene's copy is under way
    auto meanwhile = [&] {
        const int n = rob[rid].n;
        for (int i = threadIdx.x; i < B; i += blockDim.x) S.key[i] = rank_key(R, t, b0, n, i, false);
        Bf = warp_bufs(smem, L, A);
        warp_robot<SPL>(A, rob, W, Bf, rid);
    };
    if (outgrown || !collide_prologue<UNIFORM>(A, smem, L, sc0, n_obj4, &rob, meanwhile)) {
        // no verdicts: no solutions (the error flag is set)
        const int tk = T.top_k & ~kNearestFlag, nj = A.rs.rp[T.robot].n;
        const RankOut O = rank_out(R, t, tk, nj);
        for (int q = threadIdx.x; q < tk * nj; q += blockDim.x) O.q[q] = __int_as_float(0xffffffff);
        for (int q = threadIdx.x; q < tk * 2; q += blockDim.x) O.err[q] = __int_as_float(0xffffffff);
        if (threadIdx.x == 0) *O.count = 0;
        return;
    }
    const float4* s_scene = reinterpret_cast<const float4*>(smem);
    const int n = rob[rid].n;
    __syncthreads();
    // candidates with a key (finite score); the ranks that may be visited below
    const int ranked = bucket_order<false>(S, B, R.list ? depth + kWarpsPerBlock : B);
    const int top_k = T.top_k & ~kNearestFlag;

    unsigned long long tests = 0, btests = 0, ncand = 0;
    if (threadIdx.x == 0) n_found = 0;
    __syncthreads();
    int p0 = 0;
    const int warps = (int)blockDim.x >> 5, limit = R.list ? min(ranked, depth) : ranked;
    while (p0 < limit && n_found < top_k) {
        const int p = p0 + warp, g0 = p0 + warp / kWarpsPerBlock * kWarpsPerBlock;  // its group's first
        bool hit = true;
        unsigned long long t_s = 0, t_b = 0;
        if (p < ranked && g0 < limit) {
            const int64_t c = b0 + S.order[p];
            hit = warp_collides<SPL, UNIFORM, GRID>(A, rob, sc0, s_scene, W, Bf, c, rid, sid, t_s, t_b);
        }
        if (lane == 0) verdict[warp] = hit ? 1 : 0;
        __syncthreads();
        if (threadIdx.x == 0) {
            int f = n_found, g = p0;
            for (; g < p0 + warps && g < limit && f < top_k; g += kWarpsPerBlock)
                for (int q = g; q < g + kWarpsPerBlock && f < top_k; ++q)
                    if (q < ranked && !verdict[q - p0]) picks[f++] = q;
            n_found = f;
            n_checked = g;
        }
        __syncthreads();
        if (lane == 0 && p < ranked && g0 < n_checked) {
            tests += t_s;
            btests += t_b;
            ++ncand;
        }
        p0 = n_checked;
    }
    const int count = n_found;
    if (A.cnt && lane == 0) {
        atomicAdd(&A.cnt->v[3], tests);
        atomicAdd(&A.cnt->v[6], btests);
        atomicAdd(&A.cnt->v[4], ncand);
    }
    if (R.list && count < top_k && p0 < ranked) {
        // deeper than the bound: the verdicts taken so far are kept (0 free, 1 colliding), the
        // unchecked ranked candidates marked 2 for the collision filter over the listed targets,
        // which spreads them over every SM; the ranking of the listed targets follows it
        for (int i = threadIdx.x; i < B; i += blockDim.x)
            if (S.key[i] != kNoKey32) A.hit[b0 + i] = 2;
        __syncthreads();
        for (int q = threadIdx.x; q < p0; q += blockDim.x) {
            uint8_t v = 1;
            for (int r = 0; r < count; ++r) v = picks[r] == q ? 0 : v;
            A.hit[b0 + S.order[q]] = v;
        }
        if (threadIdx.x == 0) R.list[atomicAdd(R.n_list, 1)] = t;
        return;
    }
    const RankOut O = rank_out(R, t, top_k, n);
    for (int q = threadIdx.x; q < top_k * (n + 2); q += blockDim.x) {
        const int r = q / (n + 2), j = q % (n + 2);
        const bool ok = r < count;
        const int64_t g = b0 + (ok ? S.order[picks[r]] : 0);
        const float none = __int_as_float(0xffffffff);
        if (j < n) O.q[r * n + j] = ok ? R.th[j * R.ld + g] : none;
        else if (j == n) O.err[r * 2] = ok ? R.perr[g] : none;
        else O.err[r * 2 + 1] = ok ? R.oerr[g] : none;
    }
    if (threadIdx.x == 0) *O.count = count;
}

template <int SPL, bool UNIFORM, bool GRID>
bool launch_rank_lazy_t(const CollideArgs& A, const RankArgs& R, int n_obj4, int max_b, int depth, cudaStream_t st) {
    const CollideLayout L =
        collide_smem_layout(UNIFORM ? n_obj4 : 0, A.rs.n, A.rs.n_max + 2, A.rs.ns_max, A.rs.pairs_max);
    // Twice the warps while the targets leave the SMs room for them (at most two such CTAs each): a
    // cluttered target's rounds are a chain that nothing else hides.  Ranking phase, us: 97 targets x 1000
    // in 220 obstacles 87 -> 75, one target among 24 obstacles 30 -> 24; past that the SMs are full of CTAs.
    const size_t cap = 220 * 1024;
    auto keys_at = [&](int w) { return (L.total + (w - kWarpsPerBlock) * L.warp_bytes + 15u) / 16u * 16u; };
    const int64_t per_sm = (R.T + sm_count() - 1) / sm_count();
    const bool room = per_sm <= 2 && per_sm * (keys_at(kRankWarps) + bucket_smem_bytes(max_b)) <= cap;
    const int warps = room ? kRankWarps : kWarpsPerBlock;
    const uint32_t keys_off = keys_at(warps);
    const size_t smem = keys_off + bucket_smem_bytes(max_b);
    if (smem > cap) return false;
    static SmemLimit lim;
    allow_dyn_smem(k_rank_lazy<SPL, UNIFORM, GRID>, lim, cap);
    launch_next<CollideArgs, RankArgs, uint32_t, int>(k_rank_lazy<SPL, UNIFORM, GRID>, R.T, warps * 32, smem, st,
                                                      A, R, keys_off, depth);
    return true;
}

template <bool UNIFORM, bool GRID>
bool launch_rank_lazy_s(const CollideArgs& A, const RankArgs& R, int n_obj4, int max_b, int depth, cudaStream_t st) {
    const int ns = A.rs.ns_max;
    if (ns <= 32) return launch_rank_lazy_t<1, UNIFORM, GRID>(A, R, n_obj4, max_b, depth, st);
    if (ns <= 64) return launch_rank_lazy_t<2, UNIFORM, GRID>(A, R, n_obj4, max_b, depth, st);
    if (ns <= 128) return launch_rank_lazy_t<4, UNIFORM, GRID>(A, R, n_obj4, max_b, depth, st);
    return launch_rank_lazy_t<8, UNIFORM, GRID>(A, R, n_obj4, max_b, depth, st);
}

template <int SPL, bool UNIFORM, bool GRID>
void launch_collide_t(const CollideArgs& A, int n_obj4, cudaStream_t st) {
    const size_t smem =
        collide_smem_layout(UNIFORM ? n_obj4 : 0, A.rs.n, A.rs.n_max + 2, A.rs.ns_max, A.rs.pairs_max).total;
    static SmemLimit lim;
    allow_dyn_smem(k_collide<SPL, UNIFORM, GRID>, lim, 227 * 1024);
    const int g = grid_for(A.C, kWarpsPerBlock, 8);
    launch_next<CollideArgs>(k_collide<SPL, UNIFORM, GRID>, g, kWarpsPerBlock * 32, smem, st, A);
}

template <bool UNIFORM, bool GRID>
void launch_collide_s(const CollideArgs& A, int n_obj4, cudaStream_t st) {
    const int ns = A.rs.ns_max;
    if (ns <= 32) launch_collide_t<1, UNIFORM, GRID>(A, n_obj4, st);
    else if (ns <= 64) launch_collide_t<2, UNIFORM, GRID>(A, n_obj4, st);
    else if (ns <= 128) launch_collide_t<4, UNIFORM, GRID>(A, n_obj4, st);
    else launch_collide_t<8, UNIFORM, GRID>(A, n_obj4, st);
}

// ---- many candidates of one robot against one scene: a candidate per lane ----
//
// The warp-per-candidate kernel spends most of its instructions on what is the same for every
// lane (the chain, walked by all 32) or nearly always misses (every obstacle against every body's
// bounding sphere).  Here a lane walks its own candidate's chain and tests each body as its frame
// comes up, against the obstacles near it only: every CTA cuts the box that holds the obstacles,
// grown by the largest bounding radius, into 6 x 6 x 6 cells and keeps a bit per cell and obstacle,
// set where the obstacle can touch a bounding sphere centred in the cell (a margin covers the
// rounding of the cell index and of the coordinates, which may be large against a cell).  The obstacles that overlap the body's bounding sphere go to a
// lane's list and are then tested against the body's link spheres.  Pairs of bodies are tested by lane
// as well: bounding sphere against bounding sphere, the later body's link spheres against the earlier
// one's bounding sphere, and where both overlap link sphere against link sphere, for which the warp
// walks the chain again up to the earlier body (its frames would not fit shared memory): by the lanes
// that have the pair, or, where those are few, by the whole warp for one after another.  The tests that
// decide are the other kernel's, on the same spheres, so the verdicts are equal.  Bound by issue, mostly
// the walk over near obstacles, whose counts differ between lanes.  200k candidates without obstacles, us:
// a warp per candidate 228 (Panda), 612 (12 joints), 1258 (20 joints); here with the warp routine's whole self
// test for each candidate with such a pair 111, 583, 2115; with the pairs tested by lane 86, 428, 922; as it
// is 76, 301, 623.  400k Panda configurations, 60 link spheres, 220 obstacles (27% free): 294 us, where a
// warp per candidate takes 835 us.
constexpr int kCells = 6;           // per axis
constexpr int kLaneList = 12;       // overlapping obstacles a lane holds before it tests them
constexpr int64_t kLaneMinCands = 32768;
constexpr int kLaneShort = 8;       // joints up to which four CTAs per SM are taken
constexpr int kLaneMaxWords = 16;   // obstacles: 32 per word of a cell's mask, spheres and boxes in words of their own
static_assert(kCells * kCells * kCells <= kWarpsPerBlock * 32, "a cell per thread");
constexpr float kSmallBody = 0.6f;  // bounding radii up to this part of the largest have masks of their own
constexpr int kFewLanes = 4;  // candidates of a warp whose pair of bodies the whole warp tests, one after another
constexpr float kFewUlps = 4e-7f, kSomeUlps = 1e-6f;  // of a coordinate: the margins for its rounding

struct LaneLayout {
    uint32_t sph, co, range, mask, warp, warp_bytes, total;
};
constexpr int kLaneCells = kCells * kCells * kCells;
__host__ __device__ __forceinline__ LaneLayout lane_layout(uint32_t from, int ns, int nb, int words) {
    LaneLayout L;
    L.sph = (from + 15u) / 16u * 16u;
    L.co = L.sph + 16u * (uint32_t)ns;
    L.range = L.co + 16u * (uint32_t)nb;
    L.mask = L.range + 8u * (uint32_t)nb;
    L.warp = (L.mask + 4u * (uint32_t)(2 * kLaneCells * words) + 15u) / 16u * 16u;
    L.warp_bytes = 32u * (12u * (uint32_t)nb + 2u * kLaneList);
    L.total = L.warp + kWarpsPerBlock * L.warp_bytes;
    return L;
}

template <int PER_SM>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, PER_SM) k_collide_lane(const CollideArgs A) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ float s_lo[3], s_inv[3];
    __shared__ uint32_t s_pair[kMaxBodies];  // bit a of entry b: bodies a < b are checked for self-collision
    __shared__ unsigned long long s_cnt[3];  // sphere tests, box tests, candidates
    __shared__ int s_all;  // the box of the obstacles is not finite: no cells, every obstacle is near
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const SceneDev sc0 = A.n_scenes > 0 ? A.scenes[0] : SceneDev{nullptr, 0, 0};
    const int n_obj4 = sc0.n_sph + 2 * sc0.n_box;
    if (n_obj4 > A.max_obj4 || sc0.n_sph != A.u_osph || sc0.n_box != A.u_obox) {  // not the scene the host sized for
        if (tid == 0) *(volatile int32_t*)A.err_flag = 2;
        return;
    }
    const CollideLayout L = collide_smem_layout(n_obj4, A.rs.n, 0, 0, 0);
    const RobotParams* rob;
    if (!collide_prologue<true>(A, smem, L, sc0, n_obj4, &rob, [] {})) return;
    const float4* const obj = reinterpret_cast<const float4*>(smem);
    const RobotParams& R = rob[0];
    const int n = A.u_n, nb = n + 2, n_pairs = A.u_pairs, n_osph = A.u_osph, n_obox = A.u_obox;
    const int w_sph = (n_osph + 31) / 32, words = w_sph + (n_obox + 31) / 32;
    const RobotDev rd = A.rs.rd[0];
    const LaneLayout M = lane_layout(L.warp, A.rs.ns_max, nb, words);
    float4* const lsph = reinterpret_cast<float4*>(smem + M.sph);
    float4* const lco = reinterpret_cast<float4*>(smem + M.co);
    int2* const lrange = reinterpret_cast<int2*>(smem + M.range);
    uint32_t* const mask = reinterpret_cast<uint32_t*>(smem + M.mask);
    float* const cc = reinterpret_cast<float*>(smem + M.warp + warp * M.warp_bytes) + lane;  // [body][xyz][lane]
    uint16_t* const list = reinterpret_cast<uint16_t*>(smem + M.warp + warp * M.warp_bytes + 32u * 12u * nb) + lane;

    // the robot's tables
    for (int i = tid; i < rd.n_sph; i += blockDim.x) lsph[i] = __ldg(rd.sph + i);
    for (int i = tid; i < nb; i += blockDim.x) {
        lco[i] = __ldg(rd.coarse + i);
        lrange[i] = __ldg(rd.range + i);
    }
    if (tid < nb) s_pair[tid] = 0;
    if (tid < 3) s_cnt[tid] = 0;
    __syncthreads();
    for (int i = tid; i < n_pairs; i += blockDim.x) {
        const int2 pr = __ldg(rd.pairs + i);
        atomicOr(&s_pair[max(pr.x, pr.y)], 1u << min(pr.x, pr.y));
    }
    // the obstacles' box, grown by the largest bounding radius (every warp for itself)
    float rmax = 0.0f, rsmall = 0.0f;
    for (int b = 0; b < nb; ++b) rmax = fmaxf(rmax, lrange[b].y > 0 ? lco[b].w : 0.0f);
    const float r_class = kSmallBody * rmax;
    for (int b = 0; b < nb; ++b) rsmall = fmaxf(rsmall, lrange[b].y > 0 && lco[b].w <= r_class ? lco[b].w : 0.0f);
    float lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float a = __int_as_float(0x7f800000), e = -a;
        for (int o = lane; o < n_osph; o += 32) {
            const float4 v = obj[o];
            const float x = k == 0 ? v.x : (k == 1 ? v.y : v.z);
            a = fminf(a, x - v.w);
            e = fmaxf(e, x + v.w);
        }
        for (int o = lane; o < n_obox; o += 32) {
            const float4 p = obj[n_osph + 2 * o], q = obj[n_osph + 2 * o + 1];
            a = fminf(a, k == 0 ? p.x : (k == 1 ? p.y : p.z));
            e = fmaxf(e, k == 0 ? q.x : (k == 1 ? q.y : q.z));
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            a = fminf(a, __shfl_xor_sync(0xffffffffu, a, d));
            e = fmaxf(e, __shfl_xor_sync(0xffffffffu, e, d));
        }
        const float grow = rmax + 1e-3f * (e - a + rmax) + kFewUlps * fmaxf(fabsf(a), fabsf(e));
        lo[k] = a - grow;
        hi[k] = e + grow;
    }
    bool fine_box = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) fine_box = fine_box && hi[k] - lo[k] < 1e30f && hi[k] - lo[k] > 0.0f;  // (false for NaN)
    if (tid < 3) {
        const float l = tid == 0 ? lo[0] : (tid == 1 ? lo[1] : lo[2]), h = tid == 0 ? hi[0] : (tid == 1 ? hi[1] : hi[2]);
        s_lo[tid] = l;
        s_inv[tid] = (float)kCells / (h - l);
    }
    if (tid == 0) s_all = fine_box ? 0 : 1;
    // cell masks
    if (tid < kCells * kCells * kCells) {
        const int ix[3] = {tid % kCells, tid / kCells % kCells, tid / (kCells * kCells)};
        float a[3], e[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float h = (hi[k] - lo[k]) / (float)kCells;
            const float round = kFewUlps * fmaxf(fabsf(lo[k]), fabsf(hi[k]));
            a[k] = lo[k] + h * ((float)ix[k] - 1e-3f) - round;
            e[k] = lo[k] + h * ((float)ix[k] + 1.001f) + round;
        }
        for (int w = 0; w < words; ++w) {
            uint32_t m = 0, ms = 0;
            const bool sph = w < w_sph;
            const int o0 = 32 * (sph ? w : w - w_sph), cnt = min(32, (sph ? n_osph : n_obox) - o0);
#pragma unroll 4
            for (int q = 0; q < cnt; ++q) {
                const float4 p = sph ? obj[o0 + q] : obj[n_osph + 2 * (o0 + q)];
                const float4 h = sph ? p : obj[n_osph + 2 * (o0 + q) + 1];
                const float dx = fmaxf(fmaxf(a[0] - h.x, p.x - e[0]), 0.0f), dy = fmaxf(fmaxf(a[1] - h.y, p.y - e[1]), 0.0f);
                const float dz = fmaxf(fmaxf(a[2] - h.z, p.z - e[2]), 0.0f), r = sph ? p.w : 0.0f;
                const float d2 = dx * dx + dy * dy + dz * dz, rr = 1.0001f * (rmax + r), rs = 1.0001f * (rsmall + r);
                if (!fine_box || d2 <= rr * rr) m |= 1u << q;
                if (!fine_box || d2 <= rs * rs) ms |= 1u << q;
            }
            mask[tid * words + w] = m;
            mask[(kLaneCells + tid) * words + w] = ms;
        }
    }
    __syncthreads();

    const bool all = s_all != 0;
    const int64_t nwarps = (int64_t)gridDim.x * kWarpsPerBlock;
    for (int64_t c0 = 32 * ((int64_t)blockIdx.x * kWarpsPerBlock + warp); c0 < A.C; c0 += 32 * nwarps) {
        const int64_t c = c0 + lane;
        const bool have = c < A.C;
        bool hit = !have;
        unsigned t_s = 0, t_b = 0;

        // one body at frame F: its bounding sphere's centre, then the obstacles near it
        auto body = [&](int b, const Frame& F) {
            const int2 rg = lrange[b];
            const float4 co = to_world(F, lco[b]);
            cc[(3 * b) * 32] = co.x;
            cc[(3 * b + 1) * 32] = co.y;
            cc[(3 * b + 2) * 32] = co.z;
            if (rg.y == 0) return;
            const float fx = (co.x - s_lo[0]) * s_inv[0], fy = (co.y - s_lo[1]) * s_inv[1], fz = (co.z - s_lo[2]) * s_inv[2];
            const bool in = fx >= 0.0f && fx < (float)kCells && fy >= 0.0f && fy < (float)kCells && fz >= 0.0f && fz < (float)kCells;
            int cell = in && words > 0 ? (int)fx + kCells * ((int)fy + kCells * (int)fz) : -1;
            if (all && words > 0) cell = 0;  // every cell's masks are full
            if (hit) cell = -1;
            const uint32_t* const near = mask + ((lco[b].w <= r_class ? kLaneCells : 0) + max(cell, 0)) * words;
            // the set bits of mask words [w, w1), tested against the bounding sphere; those that overlap are
            // listed, and the list tested against the body's link spheres when some lane's is full and at
            // the end.  test(o) / fine(ws, o): obstacle bit o against the bounding sphere / a link sphere.
            auto walk = [&](int w, const int w1, auto test, auto fine) {
                uint32_t m = 0;
                --w;
                if (cell < 0) w = w1;  // nothing near (or already hit)
                for (;;) {
                    int k = 0;
                    while (k < kLaneList) {
                        while (m == 0 && ++w < w1) m = near[w];
                        if (m == 0) break;
                        const int o = 32 * w + __ffs(m) - 1;
                        m &= m - 1u;
                        if (test(o)) list[(k++) * 32] = (uint16_t)o;
                    }
                    __syncwarp();
                    for (int q = 0; q < k && !hit; ++q) hit = fine((int)list[q * 32]);
                    if (hit) {
                        m = 0;
                        w = w1;
                    }
                    if (!__any_sync(0xffffffffu, m != 0 || w < w1 - 1)) break;
                }
            };
            if (w_sph > 0)
                walk(0, w_sph,
                     [&](int o) {
                         ++t_s;
                         return sph_sph(co, obj[o]);
                     },
                     [&](int o) {
                         const float4 ob = obj[o];
                         bool h = false;
                         t_s += rg.y;
#pragma unroll 4
                         for (int i = rg.x; i < rg.x + rg.y; ++i) h |= sph_sph(to_world(F, lsph[i]), ob);
                         return h;
                     });
            if (words > w_sph && __any_sync(0xffffffffu, !hit)) {
                if (hit) cell = -1;
                walk(w_sph, words,
                     [&](int o) {
                         ++t_b;
                         const int x = n_osph + 2 * (o - 32 * w_sph);
                         return sph_box(co, obj[x], obj[x + 1]);
                     },
                     [&](int o) {
                         const int x = n_osph + 2 * (o - 32 * w_sph);
                         const float4 p = obj[x], h4 = obj[x + 1];
                         bool h = false;
                         t_b += rg.y;
#pragma unroll 4
                         for (int i = rg.x; i < rg.x + rg.y; ++i) h |= sph_box(to_world(F, lsph[i]), p, h4);
                         return h;
                     });
            }
            // earlier bodies whose bounding sphere overlaps this one's and one of its link spheres
            auto bound = [&](int a) {
                return make_float4(cc[(3 * a) * 32], cc[(3 * a + 1) * 32], cc[(3 * a + 2) * 32], lco[a].w);
            };
            auto widen = [](float4 s) {  // a test against it only saves work, and must not miss by rounding
                s.w += kSomeUlps * (fabsf(s.x) + fabsf(s.y) + fabsf(s.z));
                return s;
            };
            uint32_t pairs = 0;
            for (uint32_t m = s_pair[b]; m && !hit; m &= m - 1u) {
                const int a = __ffs(m) - 1;
                const float4 ca = bound(a);
                ++t_s;
                if (sph_sph(ca, co)) {
                    const float4 cw = widen(ca);
                    bool o = false;
                    t_s += rg.y;
#pragma unroll 4
                    for (int i = rg.x; i < rg.x + rg.y; ++i) o |= sph_sph(to_world(F, lsph[i]), cw);
                    pairs |= o ? 1u << a : 0u;
                }
            }
            // their link spheres against this body's: the chain is walked again up to the last of them
            uint32_t left = __reduce_or_sync(0xffffffffu, pairs);
            Frame G = frame_identity();
#pragma unroll 1
            for (int a = 0; left; ++a) {
                if (a > 0) fk_step(R, a - 1, have ? A.th[(a - 1) * A.ld + c] : 0.0f, G);
                if (!(left >> a & 1u)) continue;
                const int2 ra = lrange[a];
                unsigned who = __ballot_sync(0xffffffffu, pairs >> a & 1u);
                if (__popc(who) <= kFewLanes) {  // the warp tests one lane's spheres at a time
                    const int items = ra.y * rg.y;
                    const float per = __fdividef(1.0f, (float)rg.y);
                    for (; who; who &= who - 1u) {
                        const int src = __ffs(who) - 1;
                        bool h = false;
                        for (int w0 = 0; w0 < items; w0 += 32) {
                            const int w = min(w0 + lane, items - 1), k = (int)(((float)w + 0.5f) * per);
                            h |= sph_sph(to_world_of(G, src, lsph[ra.x + k]), to_world_of(F, src, lsph[rg.x + w - k * rg.y]));
                        }
                        h = __any_sync(0xffffffffu, h);
                        if (lane == src) {
                            hit = h;
                            t_s += items;
                        }
                    }
                } else if (pairs >> a & 1u) {
                    const float4 ca = widen(bound(a));
#pragma unroll 1
                    for (int i = rg.x; i < rg.x + rg.y && !hit; ++i) {
                        const float4 wb = to_world(F, lsph[i]);
                        if (!sph_sph(wb, ca)) continue;
                        t_s += ra.y;
#pragma unroll 4
                        for (int k = ra.x; k < ra.x + ra.y; ++k) hit |= sph_sph(to_world(G, lsph[k]), wb);
                    }
                    t_s += rg.y;
                }
                pairs = hit ? 0u : pairs & ~(1u << a);
                left = __reduce_or_sync(0xffffffffu, pairs);
            }
        };

        Frame F = frame_identity();
        float theta = have ? A.th[c] : 0.0f;  // the next joint's, loaded a body ahead
#pragma unroll 1
        for (int b = 0; b < nb; ++b) {  // (one copy of the body's code)
            if (b > n) {
                F = fk_flange(R, F);
            } else if (b > 0) {
                fk_step(R, b - 1, theta, F);
                if (b < n && have) theta = A.th[b * A.ld + c];
            }
            body(b, F);
        }
        if (have) A.hit[c] = hit ? 1 : 0;
        if (A.cnt) {  // (in shared memory: as 64-bit sums of a thread they would cost the walks registers)
            t_s = __reduce_add_sync(0xffffffffu, t_s);
            t_b = __reduce_add_sync(0xffffffffu, t_b);
            if (lane == 0) {
                atomicAdd(&s_cnt[0], (unsigned long long)t_s);
                atomicAdd(&s_cnt[1], (unsigned long long)t_b);
                atomicAdd(&s_cnt[2], (unsigned long long)min((int64_t)32, A.C - c0));
            }
        }
    }
    __syncthreads();
    if (A.cnt && tid == 0) {
        atomicAdd(&A.cnt->v[3], s_cnt[0]);
        atomicAdd(&A.cnt->v[6], s_cnt[1]);
        atomicAdd(&A.cnt->v[4], s_cnt[2]);
    }
}

template <int PER_SM>
int lane_ctas(size_t smem) {  // resident CTAs per SM
    static SmemLimit lim;
    allow_dyn_smem(k_collide_lane<PER_SM>, lim, 220 * 1024);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_collide_lane<PER_SM>, kWarpsPerBlock * 32, smem);
    return std::max(per_sm, 1);
}

bool launch_collide_lane(const CollideArgs& A, cudaStream_t st) {
    const int words = (A.u_osph + 31) / 32 + (A.u_obox + 31) / 32;
    const CollideLayout L = collide_smem_layout(A.u_osph + 2 * A.u_obox, A.rs.n, 0, 0, 0);
    const size_t smem = lane_layout(L.warp, A.rs.ns_max, A.u_n + 2, words).total;
    if (smem > 220 * 1024) return false;
    constexpr int kThreads = kWarpsPerBlock * 32;
    // Four CTAs per SM (64 registers, a few spilled) for a short chain and more candidates than three hold
    // at once, else three (80): 400k Panda configurations among 220 obstacles 353 -> 343 us, 200k of 6 joints
    // among 110 218 -> 210; 200k of 20 joints without obstacles 923 -> 1006, 65536 of 12 joints 181 -> 203
    // (before the warp took part in the pairs' tests).
    if (A.u_n <= kLaneShort && A.C > (int64_t)sm_count() * 3 * kThreads) {
        const int per_sm = lane_ctas<4>(smem);
        if (per_sm > 3) {
            k_collide_lane<4><<<grid_for(A.C, kThreads, per_sm), kThreads, smem, st>>>(A);
            return true;
        }
    }
    k_collide_lane<3><<<grid_for(A.C, kThreads, lane_ctas<3>(smem)), kThreads, smem, st>>>(A);
    return true;
}

constexpr int kContactTile = 8;  // configurations per CTA of the contact kernel

// touched[o] = 1 for every obstacle o (spheres in the caller's order, then
// boxes) that overlaps a link sphere of one of the C configurations; the
// world spheres of kContactTile configurations sit in shared memory and each
// thread tests its obstacles against all of them.
__global__ void __launch_bounds__(256) k_contacts(const RobotParams R, const RobotDev rd, const SceneDev sc,
                                                 const int32_t* perm, int64_t C, const float* th, int64_t ld,
                                                 uint8_t* touched) {
    extern __shared__ float4 wsp[];  // [kContactTile][n_sph]
    const int ns = rd.n_sph;
    const int64_t c0 = (int64_t)blockIdx.x * kContactTile;
    const int nc = (int)min((int64_t)kContactTile, C - c0);
    if (threadIdx.x < nc) {
        const int64_t c = c0 + threadIdx.x;
        float4* w = wsp + threadIdx.x * ns;
        Frame F = frame_identity();
        for (int b = 0; b <= R.n + 1; ++b) {
            if (b >= 1 && b <= R.n) fk_step(R, b - 1, th[(b - 1) * ld + c], F);
            const Frame E = b == R.n + 1 ? fk_flange(R, F) : F;
            const int2 rg = rd.range[b];
            for (int i = rg.x; i < rg.x + rg.y; ++i) w[i] = to_world(E, rd.sph[i]);
        }
    }
    __syncthreads();
    const int n_obj = sc.n_sph + sc.n_box;
    for (int o = threadIdx.x; o < n_obj; o += blockDim.x) {
        bool hit = false;
        if (o < sc.n_sph) {
            const float4 s = sc.obj[o];
            for (int i = 0; i < nc * ns && !hit; ++i) hit = sph_sph(wsp[i], s);
            if (hit) touched[perm[o]] = 1;
        } else {
            const int k = o - sc.n_sph;
            const float4 lo = sc.obj[sc.n_sph + 2 * k], hi = sc.obj[sc.n_sph + 2 * k + 1];
            for (int i = 0; i < nc * ns && !hit; ++i) hit = sph_box(wsp[i], lo, hi);
            if (hit) touched[o] = 1;
        }
    }
}

}  // namespace

void launch_contacts(const RobotParams& R, const RobotDev& rd, const SceneDev& sc, const int32_t* perm, int64_t C,
                     const float* th, int64_t ld, uint8_t* touched, cudaStream_t st) {
    if (C <= 0 || rd.n_sph <= 0 || sc.n_sph + sc.n_box <= 0) return;
    const size_t smem = sizeof(float4) * kContactTile * (size_t)rd.n_sph;
    static SmemLimit lim;
    allow_dyn_smem(k_contacts, lim, sizeof(float4) * kContactTile * (size_t)HJCD_MAX_SPHERES);
    const int64_t blocks = (C + kContactTile - 1) / kContactTile;
    k_contacts<<<(unsigned)blocks, 256, smem, st>>>(R, rd, sc, perm, C, th, ld, touched);
}

bool launch_rank_lazy(const CollideArgs& A, const RankArgs& R, int max_b, int depth, cudaStream_t st) {
    if (R.T <= 0 || A.rs.ns_max <= 0 || !R.tg || !R.io) return false;
    const bool uni = A.uniform && A.rs.n == 1 && A.n_scenes <= 1 && A.max_obj4 <= kMaxStagedObj4;
    const int n4 = A.n_scenes == 1 ? A.max_obj4 : 0;
    if (uni && A.has_grid) return launch_rank_lazy_s<true, true>(A, R, n4, max_b, depth, st);
    if (uni) return launch_rank_lazy_s<true, false>(A, R, n4, max_b, depth, st);
    if (A.has_grid) return launch_rank_lazy_s<false, true>(A, R, 0, max_b, depth, st);
    return launch_rank_lazy_s<false, false>(A, R, 0, max_b, depth, st);
}

// One robot and one scene (or none) for every candidate, with the scene small
// enough to stage: the uniform kernel (scene staged into shared memory, counts
// as launch parameters); otherwise the mixed kernel.  Launches with a gridded
// scene take the variants with the grid query.
void launch_collide(const CollideArgs& A, cudaStream_t st) {
    if (A.C <= 0 || A.rs.ns_max <= 0) return;
    const bool uni = A.uniform && A.rs.n == 1 && A.n_scenes <= 1 && A.max_obj4 <= kMaxStagedObj4;
    const int n4 = A.n_scenes == 1 ? A.max_obj4 : 0;
    // From 32768 candidates on, a candidate per lane: below, its 32 candidates per warp leave the GPU
    // underfilled.  us, by lane / by warp, 32768 candidates: Panda with 60 spheres, no obstacles 54 / 74, 110
    // obstacles 78 / 99; 6 joints, 73 spheres 55 / 92, 92 / 147; 12 joints, 127 spheres 100 / 134, 138 / 196; 20
    // joints, 197 spheres 198 / 266, 194 / 324.  (Panda among 220 obstacles, 16000: 100 / 74.)
    const int words = (A.u_osph + 31) / 32 + (A.u_obox + 31) / 32;
    if (uni && !A.has_grid && !A.list && words <= kLaneMaxWords && A.C >= kLaneMinCands && launch_collide_lane(A, st)) return;
    if (uni && A.has_grid) launch_collide_s<true, true>(A, n4, st);
    else if (uni) launch_collide_s<true, false>(A, n4, st);
    else if (A.has_grid) launch_collide_s<false, true>(A, 0, st);
    else launch_collide_s<false, false>(A, 0, st);
}

}  // namespace hjcd
