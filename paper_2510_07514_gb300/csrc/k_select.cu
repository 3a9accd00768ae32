// k_select.cu -- per-target selection: top-K and perturbed duplication
// (Alg. 2), ranking of the collision-free candidates (Alg. 2, final
// step), and packing of target poses.
//
// A target's candidates are ordered by one bucket pass over 32-bit keys in
// shared memory (bucket_order); ties go to the lower candidate and invalid
// entries (collisions, NaN) are not ranked.
#include <algorithm>

#include "hjcd_internal.cuh"

namespace hjcd {

namespace {

constexpr int kSelThreads = 512;

// Blocks (target, slice): each slice's CTA orders the target's seeds for itself and writes its share
// of the duplicates, one (duplicate, pair of joints) per thread at a time, so that a lone target's
// Philox draws spread over many SMs.  Bound by latency for few targets, by the draws for many.
// Time with one CTA sorting all keys and writing all duplicates -> this: one target of 1000 seeds
// 20 -> 8.8 us, of 2000 seeds and 24 joints 60 -> 11 us, 1000 targets of 1000 seeds 75 -> 51 us.
__global__ void __launch_bounds__(kSelThreads, 3) k_topk_dup(const DupArgs A) {
    extern __shared__ __align__(16) unsigned char sel_smem[];
    grid_follow();
    const int t = blockIdx.x;
    const int64_t m0 = A.m_off[t];
    const int M = (int)(A.m_off[t + 1] - m0);
    if (M <= 0) return;
    const Bucket S = bucket_of(sel_smem, M);
    for (int i = threadIdx.x; i < M; i += blockDim.x) {
        const float sc = A.score_M[m0 + i];
        S.key[i] = sc == sc ? score_bits(sc) : kNoKey32 - 1;  // NaN last, but ranked: every duplicate has a source
    }
    __syncthreads();
    const int K = max(1, M / A.ratio), copies = M / K, B = K * copies;
    bucket_order(S, M, K);

    const int64_t b0 = A.b_off[t];
    const TargetDesc T = A.tg[t];
    const RobotParams& R = A.rs.rp[T.robot];
    const int n = R.n, items = B * ((n + 1) / 2);
    for (int w = blockIdx.y * blockDim.x + threadIdx.x; w < items; w += gridDim.y * blockDim.x) {
        const int q = w / B, b = w - q * B;     // pair q of the normals of duplicate b,
        const uint32_t src = S.order[b % K];    // copy b / K of kept seed b % K
        const float2 z = normal_pair(T, (uint32_t)b, kPhaseDup, 0, q);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = 2 * q + h;
            if (j < n)
                A.th_B[j * A.ld_B + b0 + b] =
                    clampf(fmaf(A.sigma, h ? z.y : z.x, A.th_M[j * A.ld_M + m0 + src]), R.lim[j].x, R.lim[j].y);
        }
        if (q == 0 && A.src_B) A.src_B[b0 + b] = (int32_t)src;
    }
}

__global__ void __launch_bounds__(kSelThreads, 3) k_rank(const RankArgs A) {
    extern __shared__ __align__(16) unsigned char sel_smem[];
    grid_follow();
    int t = blockIdx.x;
    if (A.list) {  // the targets the bounded lazy pass left unfinished
        if (t >= *A.n_list) return;
        t = A.list[t];
    }
    const int64_t b0 = A.b_off[t];
    const int B = (int)(A.b_off[t + 1] - b0);
    const int n = A.rs.rp[A.tg ? A.tg[t].robot : 0].n;
    const int top_k = (A.tg ? A.tg[t].top_k : A.top_k) & ~kNearestFlag;
    const RankOut O = rank_out(A, t, top_k, n);
    const Bucket S = bucket_of(sel_smem, B > 0 ? B : 1);
    for (int i = threadIdx.x; i < B; i += blockDim.x) S.key[i] = rank_key(A, t, b0, n, i, true);
    __syncthreads();
    const int count = min(top_k, bucket_order(S, B, top_k));
    for (int q = threadIdx.x; q < top_k * (n + 2); q += blockDim.x) {
        const int r = q / (n + 2), j = q % (n + 2);
        const bool ok = r < count;
        const int64_t g = b0 + (ok ? S.order[r] : 0);
        const float none = __int_as_float(0xffffffff);
        if (j < n) O.q[r * n + j] = ok ? A.th[j * A.ld + g] : none;
        else if (j == n) O.err[r * 2] = ok ? A.perr[g] : none;
        else O.err[r * 2 + 1] = ok ? A.oerr[g] : none;
    }
    if (threadIdx.x == 0) *O.count = count;
}

__global__ void __launch_bounds__(kSelThreads, 4) k_shard_topk(const ShardTopkArgs A) {
    extern __shared__ __align__(16) unsigned char sel_smem[];
    const int t = blockIdx.x;
    const int64_t m0 = A.off[t];
    const int M = (int)(A.off[t + 1] - m0);
    const Bucket S = bucket_of(sel_smem, M > 0 ? M : 1);
    for (int i = threadIdx.x; i < M; i += blockDim.x) {
        const float sc = A.score[m0 + i];
        S.key[i] = sc == sc ? score_bits(sc) : kNoKey32;
    }
    __syncthreads();
    const int ranked = bucket_order(S, M, A.K);
    const int n = A.rs.rp[A.tg[t].robot].n;
    for (int q = threadIdx.x; q < A.K * (n + 2); q += blockDim.x) {
        const int r = q / (n + 2), j = q % (n + 2);
        const bool ok = r < ranked;
        const uint32_t src = ok ? S.order[r] : 0u;
        const int64_t o = (int64_t)t * A.K + r;
        if (j < n) A.out_th[o * A.ld_n + j] = ok ? A.th[j * A.ld + m0 + src] : 0.0f;
        else if (j == n) A.out_s[o] = ok ? A.score[m0 + src] : __int_as_float(0x7f800000);
        else A.out_i[o] = ok ? A.seed_base + (int32_t)src : -1;
    }
}

// 64-bit keys (score bits << 32 | seed index) of the lists' merge, sorted by a bitonic network; the
// all-ones key sorts last
constexpr uint64_t kNoKey = ~0ull;

__device__ __forceinline__ uint64_t score_key(float s, uint32_t idx) {
    return s == s ? ((uint64_t)score_bits(s) << 32) | idx : kNoKey;
}

__device__ __forceinline__ void bitonic_sort(uint64_t* keys, int N) {
    for (int size = 2; size <= N; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = threadIdx.x; i < (N >> 1); i += blockDim.x) {
                const int lo = 2 * i - (i & (stride - 1));
                const int hi = lo + stride;
                const bool up = (lo & size) == 0;
                const uint64_t a = keys[lo], b = keys[hi];
                if ((a > b) == up) {
                    keys[lo] = b;
                    keys[hi] = a;
                }
            }
            __syncthreads();
        }
    }
}

__device__ __forceinline__ int pow2_at_least(int m) {
    int N = 1;
    while (N < m) N <<= 1;
    return N;
}

__global__ void __launch_bounds__(kSelThreads) k_topk_merge(const MergeArgs A) {
    extern __shared__ uint64_t keys[];
    const int t = blockIdx.x;
    const int LK = A.L * A.K;
    const int N = pow2_at_least(LK);
    // key: score bits, then the seed index (ties to the lower index); the list slot is found again below
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        uint64_t k = kNoKey;
        if (i < LK) {
            const int l = i / A.K, r = i % A.K;
            const int64_t e = ((int64_t)l * A.T + t) * A.K + r;
            const int32_t idx = A.in_i[e];
            if (idx >= 0) k = score_key(A.in_s[e], (uint32_t)idx);
        }
        keys[i] = k;
    }
    __syncthreads();
    bitonic_sort(keys, N);
    // the i-th best: locate its list entry (seed indices are unique within a target)
    for (int r = threadIdx.x; r < A.K; r += blockDim.x) {
        const uint64_t key = keys[r];
        const int64_t o = (int64_t)t * A.K + r;
        if (key == kNoKey) {
            A.out_s[o] = __int_as_float(0x7f800000);
            A.out_i[o] = -1;
            for (int j = 0; j < A.n; ++j) A.out_th[o * A.n + j] = 0.0f;
            continue;
        }
        const int32_t idx = (int32_t)(key & 0xffffffffu);
        int64_t e = -1;
        for (int l = 0; l < A.L && e < 0; ++l)
            for (int q = 0; q < A.K; ++q) {
                const int64_t f = ((int64_t)l * A.T + t) * A.K + q;
                if (A.in_i[f] == idx) {
                    e = f;
                    break;
                }
            }
        A.out_s[o] = A.in_s[e];
        A.out_i[o] = idx;
        for (int j = 0; j < A.n; ++j) A.out_th[o * A.n + j] = A.in_th[e * A.n + j];
    }
}

__global__ void __launch_bounds__(kSelThreads) k_dup_kept(const KeptDupArgs A) {
    const int t = blockIdx.x;
    const int64_t b0 = A.b_off[t];
    const int B = (int)(A.b_off[t + 1] - b0);
    const TargetDesc T = A.tg[t];
    const RobotParams& R = A.rs.rp[T.robot];
    const int n = R.n;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        const int i = b % A.K;  // copy r = b / K of kept seed i
        const float* src = A.kept + ((int64_t)t * A.K + i) * n;
#pragma unroll 1
        for (int q = 0; 2 * q < n; ++q) {
            const float2 z = normal_pair(T, (uint32_t)b, kPhaseDup, 0, q);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = 2 * q + h;
                if (j < n) A.th_B[j * A.ld_B + b0 + b] = clampf(fmaf(A.sigma, h ? z.y : z.x, src[j]), R.lim[j].x, R.lim[j].y);
            }
        }
    }
}

// pose s (px py pz qw qx qy qz) into row d, its quaternion normalised; a zero or non-finite one marks
// the target invalid
__device__ __forceinline__ void set_pose(TargetDesc& d, const float* s) {
    const float qw = s[3], qx = s[4], qy = s[5], qz = s[6];
    const float nn = qw * qw + qx * qx + qy * qy + qz * qz;
    const bool ok = nn > 0.0f && isfinite(nn);
    const float r = ok ? rsqrtf(nn) : 0.0f;
    d.p[0] = s[0];
    d.p[1] = s[1];
    d.p[2] = s[2];
    d.q[0] = ok ? qw * r : 1.0f;
    d.q[1] = qx * r;
    d.q[2] = qy * r;
    d.q[3] = qz * r;
    if (!ok) d.eps_pos = -1.0f;
}

__global__ void k_pack_targets(const float* pq7, int T, const TargetDesc tmpl, TargetDesc* out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    TargetDesc d = tmpl;
    d.t_local = tmpl.t_local + t;  // the template holds the index of the first target
    set_pose(d, pq7 + 7 * (int64_t)t);
    out[t] = d;
}

// One launch in place of a copy of the head, copies of the poses and references, the packing of the
// poses and three fills: a small wave's time is its chain of stream operations.  The image is read
// from pinned host memory directly.  With the results written in place (or into the pinned buffer)
// instead of copied: one Panda pose of 64 seeds 148 -> 123 us, of 1000 seeds between host buffers
// 228 -> 189 us.
__global__ void __launch_bounds__(256) k_wave_init(const WaveInitArgs A) {
    const size_t tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x, nth = (size_t)gridDim.x * blockDim.x;
    if (tid < 7) A.zero[tid] = 0;
    if (tid == 7) *A.flag = 0;
    const uint4* src = reinterpret_cast<const uint4*>(A.pin);
    uint4* dst = reinterpret_cast<uint4*>(A.ws);
    const size_t g0 = A.o_tg / 16, g1 = g0 + (size_t)A.T * (sizeof(TargetDesc) / 16);  // the target rows: below
    for (size_t i = tid; i < A.bytes / 16; i += nth)
        if (i < g0 || i >= g1) dst[i] = __ldcv(src + i);
    const RobotParams* rp = reinterpret_cast<const RobotParams*>(A.pin + A.o_rp);
    for (size_t t = tid; t < (size_t)A.T; t += nth) {
        union {
            uint4 w[sizeof(TargetDesc) / 16];
            TargetDesc d;
        } row;
#pragma unroll
        for (int k = 0; k < (int)(sizeof(TargetDesc) / 16); ++k) row.w[k] = __ldcv(src + g0 + t * (sizeof(TargetDesc) / 16) + k);
        const TargetIo* io = reinterpret_cast<const TargetIo*>(A.pin + A.o_io) + t;
        set_pose(row.d, io->pose);
        reinterpret_cast<TargetDesc*>(A.ws + A.o_tg)[t] = row.d;
        if (A.ref && io->ref) {
            const int n = rp[row.d.robot].n;
            for (int j = 0; j < n; ++j) A.ref[t * A.ld_ref + j] = io->ref[j];
        }
    }
}

int smem_for(int m) {
    int N = 1;
    while (N < m) N <<= 1;
    return N * (int)sizeof(uint64_t);
}


}  // namespace

void launch_topk_dup(const DupArgs& A, int max_m, cudaStream_t st) {
    if (A.T <= 0 || max_m <= 0) return;
    static SmemLimit lim;
    allow_dyn_smem(k_topk_dup, lim, bucket_smem_bytes(HJCD_MAX_SAMPLES));
    // slices of a target: enough CTAs for two per SM, each with at least one item per thread
    const int items = max_m * ((A.rs.n_max + 1) / 2);
    const int slices = std::max(1, std::min(2 * sm_count() / A.T, (items + kSelThreads - 1) / kSelThreads));
    launch_next<DupArgs>(k_topk_dup, dim3(A.T, slices), kSelThreads, bucket_smem_bytes(max_m), st, A);
}

void launch_rank(const RankArgs& A, int max_b, cudaStream_t st) {
    if (A.T <= 0) return;
    static SmemLimit lim;
    allow_dyn_smem(k_rank, lim, bucket_smem_bytes(HJCD_MAX_SAMPLES));
    launch_next<RankArgs>(k_rank, A.T, kSelThreads, bucket_smem_bytes(max_b), st, A);
}

void launch_shard_topk(const ShardTopkArgs& A, int max_m, cudaStream_t st) {
    if (A.T <= 0) return;
    static SmemLimit lim;
    allow_dyn_smem(k_shard_topk, lim, bucket_smem_bytes(HJCD_MAX_SAMPLES));
    k_shard_topk<<<A.T, kSelThreads, bucket_smem_bytes(max_m), st>>>(A);
}

void launch_topk_merge(const MergeArgs& A, cudaStream_t st) {
    if (A.T <= 0 || A.L <= 0 || A.K <= 0) return;
    const int sm = smem_for(A.L * A.K);
    static SmemLimit lim;
    allow_dyn_smem(k_topk_merge, lim, 227 * 1024);
    k_topk_merge<<<A.T, kSelThreads, sm, st>>>(A);
}

void launch_dup_kept(const KeptDupArgs& A, cudaStream_t st) {
    if (A.T <= 0) return;
    k_dup_kept<<<A.T, kSelThreads, 0, st>>>(A);
}

void launch_pack_targets(const float* pq7, int T, const TargetDesc& tmpl, TargetDesc* out, cudaStream_t st) {
    if (T <= 0) return;
    k_pack_targets<<<(T + 127) / 128, 128, 0, st>>>(pq7, T, tmpl, out);
}

void launch_wave_init(const WaveInitArgs& A, cudaStream_t st) {
    k_wave_init<<<grid_for(std::max<int64_t>(A.T, (int64_t)(A.bytes / 16)), 256, 8), 256, 0, st>>>(A);
}

}  // namespace hjcd
