// wave.cu -- one packed solve over several requests (robots, scenes, seed
// counts and tolerances may all differ): Alg. 2 as one launch per phase over
// every target of the wave.
//
// Every target row carries its robot and scene (rows of the wave's tables),
// its request's tolerances, random-stream key and target index inside the
// request, so a request's results do not depend on what it is packed with.
//
// Device layout of a wave (one workspace):
//   head  robot kinematic tables | robot collision descriptors | scene
//         descriptors | target rows | seed offsets m_off | candidate offsets
//         b_off | each target's sources and outputs | inline obstacles
//         (written in pinned host memory, copied and completed by the first launch)
//   PO-CCD joint vectors [n_max][CM] and scores [CM]
//   PJ-IK joint vectors [n_max][CB], scores, errors, collision verdicts [CB]
//   results that the kernels cannot write in place, queue heads
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "host.h"

namespace hjcd {

hjcd_status plan_wave(hjcd_ctx* ctx, const WaveItem* items, int n_items, const hjcd_params& P, WavePlan* out) {
    WavePlan& W = *out;
    W = WavePlan{};
    W.n_items = n_items;
    W.item_robot.resize(n_items);
    W.item_scene.resize(n_items);
    W.item_t0.resize(n_items);
    W.item_q0.resize(n_items);
    W.item_e0.resize(n_items);
    W.at_tgt.resize(n_items);
    W.at_q.resize(n_items);
    W.at_e.resize(n_items);
    W.at_c.resize(n_items);
    W.at_ref.resize(n_items);
    size_t inl_bytes = 0;
    for (int i = 0; i < n_items; ++i) {
        const WaveItem& it = items[i];
        if (!it.rob) return fail(ctx, HJCD_EINVAL, "item %d: no robot", i);
        if (it.T < 0) return fail(ctx, HJCD_EINVAL, "item %d: n_targets < 0", i);
        if (it.T > 0 && (!it.targets || !it.out_q || !it.out_err || !it.out_count))
            return fail(ctx, HJCD_EINVAL, "item %d: null buffer", i);
        if (!(it.eps_pos > 0.0f) || !(it.eps_ori > 0.0f)) return fail(ctx, HJCD_EINVAL, "item %d: tolerances must be > 0", i);
        if (it.top_k < 1 || it.top_k > HJCD_MAX_TOPK) return fail(ctx, HJCD_EINVAL, "item %d: top_k outside [1, %d]", i, HJCD_MAX_TOPK);
        if (it.inl_nsph < 0 || it.inl_nbox < 0 || (it.inl_nsph > 0 && !it.inl_sph) || (it.inl_nbox > 0 && !it.inl_box))
            return fail(ctx, HJCD_EINVAL, "item %d: bad inline scene", i);
        if (it.cd_iters > 32767 || it.lm_iters > 32767) return fail(ctx, HJCD_EINVAL, "item %d: iteration caps above 32767", i);
        // robot table of the wave
        int r = -1;
        for (int k = 0; k < (int)W.robots.size(); ++k)
            if (W.robots[k] == it.rob) r = k;
        if (r < 0) {
            if ((int)W.robots.size() == kMaxLaunchRobots)
                return fail(ctx, HJCD_EINVAL, "more than %d distinct robots in one batch", kMaxLaunchRobots);
            r = (int)W.robots.size();
            W.robots.push_back(it.rob);
        }
        W.item_robot[i] = r;
        // scene table: resident scenes once each, inline scenes one per item
        int sidx = -1;
        if (it.scene) {
            for (int k = 0; k < (int)W.scenes.size(); ++k)
                if (W.scenes[k].res == it.scene) sidx = k;
            if (sidx < 0) {
                sidx = (int)W.scenes.size();
                W.scenes.push_back({it.scene, i, 0, it.scene->dev.n_sph, it.scene->dev.n_box});
            }
        } else if (it.inl_nsph + it.inl_nbox > 0) {
            for (int k = 0; k < it.inl_nsph; ++k)
                if (!(it.inl_sph[4 * k + 3] > 0.0f)) return fail(ctx, HJCD_EINVAL, "item %d: obstacle sphere %d radius must be > 0", i, k);
            for (int k = 0; k < it.inl_nbox; ++k) {
                const float* b = it.inl_box + 6 * k;
                if (!(b[0] <= b[3] && b[1] <= b[4] && b[2] <= b[5])) return fail(ctx, HJCD_EINVAL, "item %d: box %d lo > hi", i, k);
            }
            sidx = (int)W.scenes.size();
            W.scenes.push_back({nullptr, i, inl_bytes, it.inl_nsph, it.inl_nbox});
            inl_bytes += align_up(16 * (size_t)(it.inl_nsph + 2 * it.inl_nbox), 16);
        }
        W.item_scene[i] = sidx;
        const bool some = it.T > 0;
        W.at_tgt[i] = some ? pointer_reach(it.targets, ctx->device) : 0;
        W.at_q[i] = some ? pointer_reach(it.out_q, ctx->device) : 0;
        W.at_e[i] = some ? pointer_reach(it.out_err, ctx->device) : 0;
        W.at_c[i] = some ? pointer_reach(it.out_count, ctx->device) : 0;
        W.at_ref[i] = some && it.q_ref ? pointer_reach(it.q_ref, ctx->device) : 0;
        W.has_ref = W.has_ref || (some && it.q_ref);
        W.host_out = W.host_out || (some && (W.at_q[i] == 0 || W.at_e[i] == 0 || W.at_c[i] == 0));
        if (some && W.at_tgt[i] == 0) {
            for (int t = 0; t < it.T; ++t) {
                const float* q = it.targets + 7 * (size_t)t + 3;
                const float nn = q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3];
                if (!(nn > 0.0f) || !std::isfinite(nn)) return fail(ctx, HJCD_EINVAL, "item %d target %d: zero quaternion", i, t);
            }
        }
        for (int t = 0; t < it.T; ++t) {
            const int m = it.spt ? it.spt[t] : it.n_samples;
            if (m < 1 || m > HJCD_MAX_SAMPLES)
                return fail(ctx, HJCD_EINVAL, "item %d target %d: seed count %d outside [1, %d]", i, t, m, HJCD_MAX_SAMPLES);
        }
    }
    // rows, seeds and candidates, the items with the longest chains first: their candidates take longest,
    // so the kernels' queues end on short work, and candidates that share a CTA of the polish, which
    // wait for one another, are of similar length.  Eight chains of 6 to 20 joints x 40 targets in
    // ascending order 3.57 -> 3.38 ms (shortest first: 3.60); a burst of 20 served requests 1.75 -> 1.57.
    W.order.resize(n_items);
    for (int i = 0; i < n_items; ++i) W.order[i] = i;
    std::stable_sort(W.order.begin(), W.order.end(), [&](int x, int y) { return items[x].rob->P.n > items[y].rob->P.n; });
    for (int i : W.order) {
        const WaveItem& it = items[i];
        W.item_t0[i] = W.T;
        W.item_q0[i] = W.q_total;
        W.item_e0[i] = W.e_total;
        for (int t = 0; t < it.T; ++t) {
            const int m = it.spt ? it.spt[t] : it.n_samples;
            const int64_t b = dup_count(m, P.dup_ratio);
            W.CM += m;
            W.CB += b;
            W.min_m = W.CM == m ? m : std::min(W.min_m, m);
            W.max_m = std::max(W.max_m, m);
            W.max_b = std::max(W.max_b, (int)b);
        }
        if ((int64_t)W.T + it.T > (int64_t)(1 << 30)) return fail(ctx, HJCD_EINVAL, "too many targets in one batch");
        W.T += it.T;
        W.q_total += (int64_t)it.T * it.top_k * it.rob->P.n;
        W.e_total += (int64_t)it.T * it.top_k * 2;
    }
    W.NR = (int)W.robots.size();
    W.NS = (int)W.scenes.size();
    for (const RobotRec* r : W.robots) {
        W.n_max = std::max(W.n_max, r->P.n);
        W.ns_max = std::max(W.ns_max, r->P.n_sph);
        W.pairs_max = std::max(W.pairs_max, r->n_pairs);
    }
    for (const auto& e : W.scenes) W.obj4_max = std::max(W.obj4_max, e.nsph + 2 * e.nbox);

    Carve cv;
    W.o_rp = cv.take<RobotParams>(std::max(W.NR, 1));
    W.o_rd = cv.take<RobotDev>(std::max(W.NR, 1));
    W.o_sd = cv.take<SceneDev>(std::max(W.NS, 1));
    W.o_tg = cv.take<TargetDesc>(W.T);
    W.o_moff = cv.take<int64_t>((size_t)W.T + 1);
    W.o_boff = cv.take<int64_t>((size_t)W.T + 1);
    W.o_io = cv.take<TargetIo>(W.T);
    W.o_inl = cv.take<char>(inl_bytes);
    W.head = cv.off;
    bool copy_tgt = false, copy_ref = false;  // poses or references of another device, or not on 4 bytes
    for (int i = 0; i < n_items; ++i) {
        copy_tgt = copy_tgt || W.at_tgt[i] == 1;
        copy_ref = copy_ref || W.at_ref[i] == 1;
    }
    W.o_pose = cv.take<float>(copy_tgt ? 7 * (size_t)W.T : 0);
    W.o_pref = cv.take<float>(copy_ref ? (size_t)W.T * W.n_max : 0);
    W.o_ref = cv.take<float>(W.has_ref ? (size_t)W.T * W.n_max : 0);
    W.o_thM = cv.take<float>((size_t)W.n_max * W.CM);
    W.o_thM2 = cv.take<float>(P.cd_variant == 2 ? (size_t)W.n_max * W.CM : 0);  // lock-step PO-CCD's second buffer
    W.o_sM = cv.take<float>(W.CM);
    W.o_thB = cv.take<float>((size_t)W.n_max * W.CB);
    W.o_sB = cv.take<float>(W.CB);
    W.o_pB = cv.take<float>(W.CB);
    W.o_oB = cv.take<float>(W.CB);
    W.o_hB = cv.take<uint8_t>(W.CB);
    W.o_q = cv.take<float>(W.q_total);
    W.o_e = cv.take<float>(W.e_total);
    W.o_c = cv.take<int32_t>(W.T);
    W.o_ul = cv.take<int32_t>(W.T);           // targets left to the second collision pass
    W.o_sg = cv.take<int32_t>(2 * (size_t)W.CM);  // PO-CCD candidates handed between segments
    // queue head, PJ-IK's count of o_sg, count of o_ul, PO-CCD's counts of o_sg, its segments' queue heads;
    // PJ-IK's count of finished candidates
    W.o_qf = cv.take<unsigned long long>(7);
    W.bytes = cv.off;

    Carve pv;
    pv.off = W.head;
    W.p_pose = pv.take<float>(7 * (size_t)W.T);
    W.p_ref = pv.take<float>(W.has_ref ? (size_t)W.T * W.n_max : 0);
    W.staged = W.host_out && 4 * (size_t)(W.q_total + W.e_total + W.T) <= kStagedResults;
    W.p_q = pv.take<float>(W.staged ? W.q_total : 0);
    W.p_e = pv.take<float>(W.staged ? W.e_total : 0);
    W.p_c = pv.take<int32_t>(W.staged ? W.T : 0);
    W.pin_bytes = kFlagBytes + pv.off;
    return HJCD_OK;
}

void take_results(const WavePlan& W, int i, const WaveItem& it, const char* pin) {
    if (it.T == 0) return;
    pin += kFlagBytes;
    const size_t nq = (size_t)it.T * it.top_k * it.rob->P.n, ne = (size_t)it.T * it.top_k * 2;
    if (W.at_q[i] == 0) std::memcpy(it.out_q, pin + W.p_q + 4 * W.item_q0[i], sizeof(float) * nq);
    if (W.at_e[i] == 0) std::memcpy(it.out_err, pin + W.p_e + 4 * W.item_e0[i], sizeof(float) * ne);
    if (W.at_c[i] == 0) std::memcpy(it.out_count, pin + W.p_c + 4 * (size_t)W.item_t0[i], sizeof(int32_t) * (size_t)it.T);
}

hjcd_status run_wave(hjcd_ctx* ctx, const WavePlan& W, const WaveItem* items, const hjcd_params& P, char* ws,
                     char* pin, cudaStream_t s, cudaEvent_t* ev, cudaEvent_t read) {
    if (W.T == 0) return HJCD_OK;
    hjcd_status st;
    // ---- pinned image of the head ----
    int32_t* const flag = wave_flag(pin);
    pin += kFlagBytes;
    RobotParams* h_rp = reinterpret_cast<RobotParams*>(pin + W.o_rp);
    RobotDev* h_rd = reinterpret_cast<RobotDev*>(pin + W.o_rd);
    SceneDev* h_sd = reinterpret_cast<SceneDev*>(pin + W.o_sd);
    TargetDesc* h_tg = reinterpret_cast<TargetDesc*>(pin + W.o_tg);
    int64_t* h_moff = reinterpret_cast<int64_t*>(pin + W.o_moff);
    int64_t* h_boff = reinterpret_cast<int64_t*>(pin + W.o_boff);
    TargetIo* h_io = reinterpret_cast<TargetIo*>(pin + W.o_io);
    float* h_pose = reinterpret_cast<float*>(pin + W.p_pose);
    float* h_ref = reinterpret_cast<float*>(pin + W.p_ref);
    for (int r = 0; r < W.NR; ++r) {
        h_rp[r] = W.robots[r]->P;
        h_rd[r] = W.robots[r]->dev;
    }
    for (int k = 0; k < W.NS; ++k) {
        const auto& e = W.scenes[k];
        if (e.res) {
            h_sd[k] = e.res->dev;
        } else {
            const WaveItem& it = items[e.item];
            float4* o = reinterpret_cast<float4*>(pin + W.o_inl + e.off);
            for (int q = 0; q < it.inl_nsph; ++q)
                o[q] = make_float4(it.inl_sph[4 * q], it.inl_sph[4 * q + 1], it.inl_sph[4 * q + 2], it.inl_sph[4 * q + 3]);
            for (int q = 0; q < it.inl_nbox; ++q) {
                const float* b = it.inl_box + 6 * q;
                o[it.inl_nsph + 2 * q] = make_float4(b[0], b[1], b[2], 0.0f);
                o[it.inl_nsph + 2 * q + 1] = make_float4(b[3], b[4], b[5], 0.0f);
            }
            h_sd[k] = SceneDev{reinterpret_cast<const float4*>(ws + W.o_inl + e.off), e.nsph, e.nbox};
        }
    }
    h_moff[0] = h_boff[0] = 0;
    for (int i : W.order) {
        const WaveItem& it = items[i];
        const int n = it.rob->P.n;
        const int cd = it.cd_iters >= 0 ? it.cd_iters : P.cd_max_iters;
        const int lm = it.lm_iters >= 0 ? it.lm_iters : P.lm_max_iters;
        // the item's poses and references where the first launch finds them, its results where the last
        // one puts them: in place, or beside the image (host, small), or in the workspace
        const size_t t0 = W.item_t0[i], nq = (size_t)it.top_k * n;
        const float* pose = W.at_tgt[i] == 2 ? it.targets
                            : W.at_tgt[i] == 1 ? reinterpret_cast<const float*>(ws + W.o_pose) + 7 * t0 : h_pose + 7 * t0;
        const float* ref = !it.q_ref ? nullptr
                           : W.at_ref[i] == 2 ? it.q_ref
                           : W.at_ref[i] == 1 ? reinterpret_cast<const float*>(ws + W.o_pref) + t0 * W.n_max
                                              : h_ref + t0 * W.n_max;
        auto block = [&](int at, auto* user, size_t p_off, size_t o_off, size_t first) {
            using E = std::remove_reference_t<decltype(*user)>;
            if (at == 2) return user;
            return reinterpret_cast<E*>(at == 0 && W.staged ? pin + p_off : ws + o_off) + first;
        };
        float* oq = it.T ? block(W.at_q[i], it.out_q, W.p_q, W.o_q, W.item_q0[i]) : nullptr;
        float* oe = it.T ? block(W.at_e[i], it.out_err, W.p_e, W.o_e, W.item_e0[i]) : nullptr;
        int32_t* oc = it.T ? block(W.at_c[i], it.out_count, W.p_c, W.o_c, t0) : nullptr;
        for (int t = 0; t < it.T; ++t) {
            const int g = W.item_t0[i] + t;
            TargetDesc d{};
            d.eps_pos = it.eps_pos;
            d.eps_ori = it.eps_ori;
            d.key[0] = (uint32_t)(it.seed & 0xffffffffu);
            d.key[1] = (uint32_t)(it.seed >> 32);
            d.t_local = it.t_base + t;
            d.robot = W.item_robot[i];
            d.scene = W.item_scene[i];
            d.cd_iters = (int16_t)cd;
            d.lm_iters = (int16_t)lm;
            d.top_k = it.top_k | (it.q_ref ? kNearestFlag : 0);
            h_tg[g] = d;
            const int m = it.spt ? it.spt[t] : it.n_samples;
            h_moff[g + 1] = h_moff[g] + m;
            h_boff[g + 1] = h_boff[g] + dup_count(m, P.dup_ratio);
            h_io[g] = TargetIo{pose + 7 * (size_t)t, ref ? ref + (size_t)t * n : nullptr, oq + t * nq,
                               oe + (size_t)t * it.top_k * 2, oc + t};
        }
        if (W.at_tgt[i] == 0 && it.T > 0)
            std::memcpy(h_pose + 7 * t0, it.targets, sizeof(float) * 7 * (size_t)it.T);
        if (W.at_ref[i] == 0 && it.q_ref && it.T > 0)
            std::memcpy(h_ref + t0 * W.n_max, it.q_ref, sizeof(float) * (size_t)it.T * n);
    }

    // ---- what kernels cannot read in place: another device's memory, or not on 4 bytes ----
    for (int i = 0; i < W.n_items; ++i) {
        const WaveItem& it = items[i];
        if (W.at_tgt[i] == 1)
            HJCD_CUDA(ctx, cudaMemcpyAsync(ws + W.o_pose + sizeof(float) * 7 * (size_t)W.item_t0[i], it.targets,
                                           sizeof(float) * 7 * (size_t)it.T, cudaMemcpyDeviceToDevice, s));
        if (W.at_ref[i] == 1)
            HJCD_CUDA(ctx, cudaMemcpyAsync(ws + W.o_pref + sizeof(float) * (size_t)W.item_t0[i] * W.n_max, it.q_ref,
                                           sizeof(float) * (size_t)it.T * it.rob->P.n, cudaMemcpyDeviceToDevice, s));
    }

    TargetDesc* d_tg = reinterpret_cast<TargetDesc*>(ws + W.o_tg);
    const int64_t* d_moff = reinterpret_cast<const int64_t*>(ws + W.o_moff);
    const int64_t* d_boff = reinterpret_cast<const int64_t*>(ws + W.o_boff);
    float* thM = reinterpret_cast<float*>(ws + W.o_thM);
    float* sM = reinterpret_cast<float*>(ws + W.o_sM);
    float* thB = reinterpret_cast<float*>(ws + W.o_thB);
    float* sB = reinterpret_cast<float*>(ws + W.o_sB);
    float* pB = reinterpret_cast<float*>(ws + W.o_pB);
    float* oB = reinterpret_cast<float*>(ws + W.o_oB);
    uint8_t* hB = reinterpret_cast<uint8_t*>(ws + W.o_hB);
    unsigned long long* queue = reinterpret_cast<unsigned long long*>(ws + W.o_qf);
    RobotSet rs{reinterpret_cast<const RobotParams*>(ws + W.o_rp), reinterpret_cast<const RobotDev*>(ws + W.o_rd),
                W.NR, W.n_max, W.ns_max, W.pairs_max};
    rs.plain = 1;
    for (int r = 0; r < W.NR; ++r) rs.plain &= W.robots[r]->P.plain;

    if (ev) HJCD_CUDA(ctx, cudaEventRecord(ev[0], s));
    launch_wave_init(WaveInitArgs{pin, ws, W.head, W.o_tg, W.o_io, W.o_rp, W.T,
                                  W.has_ref ? reinterpret_cast<float*>(ws + W.o_ref) : nullptr, W.n_max, queue,
                                  flag},
                     s);
    if ((st = after_launch(ctx, 1, "k_wave_init"))) return st;
    if (read) HJCD_CUDA(ctx, cudaEventRecord(read, s));

    // Alg. 2: PO-CCD from uniform seeds
    CcdArgs ca{};
    ca.rs = rs;
    ca.tg = d_tg;
    const bool uni_m = W.T > 0 && W.min_m == W.max_m;  // offsets t * max_b for PJ-IK and the filter
    ca.map = CandMap{nullptr, nullptr, d_moff, W.T, 0};
    ca.C = W.CM;
    ca.ld = W.CM;
    ca.th_out = thM;
    ca.th_tmp = reinterpret_cast<float*>(ws + W.o_thM2);
    ca.score = sM;
    ca.n_iters = -1;
    ca.P = P;
    ca.cnt = ctx->cnt;
    ca.block = ctx->ccd_block;
    ca.in_limits = 1;  // seeds sampled inside the limits, every update clamped to them
    // Iteration segments: a lane whose candidate meets the coarse tolerance waits for the rest of
    // its warp, so the iterations run in three launches ([0, cap/2), [cap/2, 3 cap/4), the rest)
    // and the candidates still iterating are packed afresh into full warps for the next (the same
    // results: each candidate's state, iteration index and random streams carry over).  Only for
    // waves that fill the GPU many times over with equal seed counts: a small wave pays the extra
    // launches in latency, and the mixed eight-chain batch (unequal counts) measured slower.
    int cap_max = 0;
    for (int i = 0; i < W.n_items; ++i) cap_max = std::max(cap_max, items[i].cd_iters >= 0 ? items[i].cd_iters : P.cd_max_iters);
    const bool segments = P.cd_variant != 2 && cap_max >= 8 && W.min_m == W.max_m && W.CM >= (int64_t)sm_count() * 2048;
    if (segments) {
        int32_t* lists = reinterpret_cast<int32_t*>(ws + W.o_sg);
        int32_t* counts = reinterpret_cast<int32_t*>(ws + W.o_qf + 16);
        const int seg[3] = {0, cap_max / 2, (3 * cap_max) / 4};
        for (int g = 0; g < 3; ++g) {
            CcdArgs cg = ca;
            cg.seg_begin = seg[g];
            cg.seg_end = g < 2 ? seg[g + 1] : 0;
            cg.list_in = g > 0 ? lists + (size_t)((g - 1) & 1) * W.CM : nullptr;
            cg.n_in = g > 0 ? counts + ((g - 1) & 1) : nullptr;
            cg.list_out = g < 2 ? lists + (size_t)(g & 1) * W.CM : nullptr;
            cg.n_out = g < 2 ? counts + (g & 1) : nullptr;
            cg.queue = reinterpret_cast<unsigned long long*>(ws + W.o_qf + 24) + g;
            launch_ccd(cg, false, s);
            if ((st = after_launch(ctx, 1, "k_ccd"))) return st;
        }
    } else {
        CcdArgs c1 = ca;
        c1.queue = reinterpret_cast<unsigned long long*>(ws + W.o_qf + 24);
        launch_ccd(c1, false, s);
        if ((st = after_launch(ctx, 1, "k_ccd"))) return st;
    }
    if (ev) HJCD_CUDA(ctx, cudaEventRecord(ev[1], s));

    // top-K and perturbed duplication
    DupArgs da{rs, d_tg, W.T, d_moff, sM, thM, W.CM, d_boff, thB, W.CB, nullptr, P.dup_ratio, P.dup_sigma};
    launch_topk_dup(da, W.max_m, s);
    if ((st = after_launch(ctx, 1, "k_topk_dup"))) return st;
    if (ev) HJCD_CUDA(ctx, cudaEventRecord(ev[2], s));

    // PJ-IK
    LmArgs la{};
    la.rs = rs;
    la.tg = d_tg;
    la.map = CandMap{nullptr, nullptr, d_boff, W.T, uni_m ? W.max_b : 0};
    la.C = W.CB;
    la.ld = W.CB;
    la.th = thB;
    la.score = sB;
    la.perr = pB;
    la.oerr = oB;
    la.n_iters = -1;
    la.P = P;
    la.cnt = ctx->cnt;
    la.queue = queue;
    la.warps = ctx->lm_warps;
    la.in_limits = 1;  // PO-CCD's joint vectors and their clamped duplicates
    la.list = reinterpret_cast<int32_t*>(ws + W.o_sg);  // PO-CCD is done with its lists
    la.list_k = la.list + W.CM;
    la.n_list = reinterpret_cast<int32_t*>(ws + W.o_qf + 8);
    la.n_done = reinterpret_cast<int32_t*>(queue + 6);
    if ((st = after_launch(ctx, launch_lm(la, false, s), "k_lm"))) return st;
    if (ev) HJCD_CUDA(ctx, cudaEventRecord(ev[3], s));

    // collision filter and ranking
    const bool collide = W.ns_max > 0;
    RankArgs ra{rs, d_tg, W.T, d_boff, thB, W.CB, sB, pB, oB, collide ? hB : nullptr, 0,
                reinterpret_cast<const TargetIo*>(ws + W.o_io), nullptr, nullptr, nullptr,
                W.has_ref ? reinterpret_cast<const float*>(ws + W.o_ref) : nullptr, W.n_max};
    CollideArgs cl{};
    if (collide) {
        cl.rs = rs;
        cl.scenes = reinterpret_cast<const SceneDev*>(ws + W.o_sd);
        cl.n_scenes = W.NS;
        cl.max_obj4 = W.obj4_max;
        bool same_scene = true;  // one robot and the same scene for every request
        for (int i = 1; i < W.n_items; ++i) same_scene = same_scene && W.item_scene[i] == W.item_scene[0];
        cl.uniform = W.NR == 1 && same_scene && (W.NS == 0 || W.item_scene[0] == 0);
        if (cl.uniform) {
            cl.u_n = W.robots[0]->P.n;
            cl.u_pairs = W.robots[0]->n_pairs;
            cl.u_osph = W.NS ? W.scenes[0].nsph : 0;
            cl.u_obox = W.NS ? W.scenes[0].nbox : 0;
        }
        for (const auto& e : W.scenes) cl.has_grid = cl.has_grid || (e.res && e.res->dev.cell);
        cl.tg = d_tg;
        cl.map = CandMap{nullptr, nullptr, d_boff, W.T, uni_m ? W.max_b : 0};
        cl.C = W.CB;
        cl.ld = W.CB;
        cl.th = thB;
        cl.hit = hB;
        cl.cnt = ctx->cnt;
        cl.err_flag = flag;
        cl.first_wait_polls = ctx->first_wait_polls.load();
    }
    // the top_k collision-free candidates by score are the first top_k collision-free ones in score
    // order: check candidates in that order until they are found (same output as filtering all)
    // A target whose first kLazyDepth ranked candidates hold fewer than top_k collision-free ones
    // (a cluttered scene) would keep one CTA busy for its whole list while the other SMs idle: it
    // is listed instead, and the filter over the listed targets' candidates and their ranking
    // follow as two grid-wide launches.
    bool lazy = false;
    if (collide && ctx->collide_lazy) {
        if (ev) HJCD_CUDA(ctx, cudaEventRecord(ev[4], s));
        RankArgs rl = ra;
        rl.list = reinterpret_cast<int32_t*>(ws + W.o_ul);
        rl.n_list = reinterpret_cast<int32_t*>(ws + W.o_qf + 12);
        lazy = launch_rank_lazy(cl, rl, W.max_b, kLazyDepth, s);
        if (lazy) {
            if ((st = after_launch(ctx, 1, "k_rank_lazy"))) return st;
            CollideArgs c2 = cl;
            c2.list = rl.list;
            c2.n_list = rl.n_list;
            c2.b_off = d_boff;
            c2.list_bmax = std::max(W.max_b, 1);
            launch_collide(c2, s);
            if ((st = after_launch(ctx, 1, "k_collide (list)"))) return st;
            launch_rank(rl, W.max_b, s);
            if ((st = after_launch(ctx, 1, "k_rank (list)"))) return st;
        }
    }
    if (!lazy) {
        if (collide) {
            launch_collide(cl, s);
            if ((st = after_launch(ctx, 1, "k_collide"))) return st;
        }
        if (ev) HJCD_CUDA(ctx, cudaEventRecord(ev[4], s));
        launch_rank(ra, W.max_b, s);
        if ((st = after_launch(ctx, 1, "k_rank"))) return st;
    }
    if (ev) HJCD_CUDA(ctx, cudaEventRecord(ev[5], s));

    // results that the kernels left in the workspace
    for (int i = 0; i < W.n_items; ++i) {
        const WaveItem& it = items[i];
        if (it.T == 0) continue;
        auto out = [&](int at, void* user, const char* from, size_t bytes) -> hjcd_status {
            if (at == 2 || (at == 0 && W.staged)) return HJCD_OK;
            HJCD_CUDA(ctx, cudaMemcpyAsync(user, from, bytes, at ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
            return HJCD_OK;
        };
        const size_t nq = (size_t)it.T * it.top_k * it.rob->P.n, ne = (size_t)it.T * it.top_k * 2;
        if ((st = out(W.at_q[i], it.out_q, ws + W.o_q + 4 * W.item_q0[i], sizeof(float) * nq))) return st;
        if ((st = out(W.at_e[i], it.out_err, ws + W.o_e + 4 * W.item_e0[i], sizeof(float) * ne))) return st;
        if ((st = out(W.at_c[i], it.out_count, ws + W.o_c + 4 * (size_t)W.item_t0[i], sizeof(int32_t) * (size_t)it.T))) return st;
    }
    return HJCD_OK;
}

}  // namespace hjcd
