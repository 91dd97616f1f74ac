// Keep the k highest-entropy tokens of every segment (ties -> lower index) and build the
// gather/scatter index lists.
//
// One CTA per segment. The segment's keys (at most 16384) live in the registers of its threads as
// order-preserving unsigned integers. The k-th largest key T, and how many keys equal to T must still be taken,
// come from a most-significant-digit radix select on digits of 11 bits that starts at the highest bit in which any two
// keys differ; when at most 32 keys are left in the chosen bin, they are ranked directly. A final ordered pass
// (warp ballots + a sum over the warps' totals) writes kept and pruned indices in ascending order.
// What bounds it: latency, mostly of barriers and shared-memory atomics. Entropies differ little in their exponents,
// so the first 8-bit digit of a four-pass select over keys in shared memory put most keys in two or three bins, one atomic
// after the other, and each pass cost three barriers. Launches back to back, us: 2 segments of 256 keys 5.8 -> 2.4, 2 x 1024
// 6.4 -> 2.7, 32 x 1600 8.2 -> 4.4, 128 x 4096 12.9 -> 8.9, 1 x 16384 16.8 -> 12.7.
#include "common.cuh"

namespace {

constexpr int kDigitBits = 11;
constexpr int kBins = 1 << kDigitBits;
constexpr int kDirect = 32;            // candidates ranked directly, one per lane
constexpr int kMaxSegPerLaunch = 256;

struct SegParams {
    int32_t k[kMaxSegPerLaunch];
};

__device__ __forceinline__ uint32_t order_key(float f)
{
    uint32_t u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0;                       // -0 and +0 are the same key
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u); // larger float <=> larger key
}

// group == 0: the launch's segments form one list (cu_keep [S+1], kept and pruned lists concatenated
// over all segments). group > 0: every `group` consecutive segments (the images of one layer) form a
// list of their own: cumulative counts restart, group g writes cu_keep[g*(group+1) ...] and its index
// lists start at g*group*N. A launch then holds whole groups.
template <int THREADS, int KEYS>
__global__ void __launch_bounds__(THREADS)
select_topk_kernel(const float* __restrict__ ent, int N, int seg0, int cu0, SegParams sp,
                   const int32_t* __restrict__ k_dev, int32_t* __restrict__ keep_idx, int32_t* __restrict__ prune_idx,
                   int32_t* __restrict__ cu_keep, int32_t* __restrict__ pos, int group)
{
    constexpr int kWarps = THREADS / 32, kBinsPer = kBins / THREADS;
    __shared__ uint32_t hist[kBins], cand[kDirect], warp_a[kWarps], warp_b[kWarps];
    __shared__ uint32_t sh_digit, sh_need, sh_count, sh_cand;

    pdl_launch_dependents();               // (everything before an ordinary launch has ended)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int seg_local = blockIdx.x;
    const int seg = seg0 + seg_local;
    // warp w owns the indices [w * 32 * KEYS, (w + 1) * 32 * KEYS), lane-interleaved
    const int i0 = warp * 32 * KEYS + lane;
    const float* e = ent + (long)seg * N;
    uint32_t key[KEYS];
#pragma unroll
    for (int j = 0; j < KEYS; ++j) key[j] = i0 + j * 32 < N ? order_key(e[i0 + j * 32]) : 0u;

    const int grp = group > 0 ? seg / group : 0;
    const int seg_in = group > 0 ? seg - grp * group : seg;          // position within its list
    const int list_first = seg - seg_in;                             // first segment of the list
    __shared__ int sh_cu;
    int k, cu;
    if (k_dev) {
        // keep counts written by an earlier kernel: clamp to [0, N]; cu = sum over the list's segments before
        if (tid == 0) sh_cu = 0;
        __syncthreads();
        int part = 0;
        for (int s = list_first + tid; s < seg; s += THREADS) part += min(max(k_dev[s], 0), N);
        part = __reduce_add_sync(0xffffffffu, part);
        if (lane == 0 && part) atomicAdd(&sh_cu, part);
        __syncthreads();
        cu = sh_cu;
        k = min(max(k_dev[seg], 0), N);
    } else {
        k = sp.k[seg_local];
        cu = group > 0 ? 0 : cu0;
        for (int s = group > 0 ? seg_local - seg_in : 0; s < seg_local; ++s) cu += sp.k[s];
    }
    if (tid == 0) {
        int32_t* cu_out = cu_keep + (group > 0 ? (long)grp * (group + 1) : 0);
        cu_out[seg_in] = cu;
        // last segment of a list (or of this launch: the next launch overwrites with the same value)
        if (group > 0 ? seg_in == group - 1 : seg_local == (int)gridDim.x - 1) cu_out[seg_in + 1] = cu + k;
    }

    // ---- kept: every key > T, and the first `need` of those equal to T.
    // (k <= 0: keep nothing; k >= N: keep everything)
    const bool keep_all = (k >= N), keep_none = (k <= 0);
    uint32_t T = 0, need = (uint32_t)k;
    if (!keep_all && !keep_none) {
        uint32_t lo = 0xffffffffu, hi = 0;
#pragma unroll
        for (int j = 0; j < KEYS; ++j)
            if (i0 + j * 32 < N) { lo = min(lo, key[j]); hi = max(hi, key[j]); }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) { warp_a[warp] = lo; warp_b[warp] = hi; }
#pragma unroll
        for (int j = 0; j < kBinsPer; ++j) hist[tid + j * THREADS] = 0;
        if (tid == 0) sh_cand = 0;
        __syncthreads();
        lo = __reduce_min_sync(0xffffffffu, lane < kWarps ? warp_a[lane] : 0xffffffffu);
        hi = __reduce_max_sync(0xffffffffu, lane < kWarps ? warp_b[lane] : 0u);
        // Only the low `bits` bits are still open; above them T is known and `in_play` keys agree with it.
        int bits = 32 - __clz((int)(lo ^ hi));
        auto in_play = [&](int j) { return i0 + j * 32 < N && (bits >= 32 || ((key[j] ^ T) >> bits) == 0); };
        T = bits >= 32 ? 0u : hi & (0xffffffffu << bits);
        while (bits > 0) {
            const int shift = max(bits - kDigitBits, 0);
            const uint32_t digit_mask = (1u << (bits - shift)) - 1u;
#pragma unroll
            for (int j = 0; j < KEYS; ++j)
                if (in_play(j)) atomicAdd(&hist[(key[j] >> shift) & digit_mask], 1u);
            __syncthreads();
            // thread t owns the bins kBins - 1 - t * kBinsPer and down; how many keys lie above them?
            uint32_t c[kBinsPer], tot = 0;
#pragma unroll
            for (int j = 0; j < kBinsPer; ++j) { c[j] = hist[kBins - 1 - tid * kBinsPer - j]; tot += c[j]; }
            uint32_t incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane == 31) warp_a[warp] = incl;
            __syncthreads();
            uint32_t above = __reduce_add_sync(0xffffffffu, lane < warp ? warp_a[lane] : 0u) + incl - tot;
            if (above < need && need <= above + tot) {
                bool found = false;
#pragma unroll
                for (int j = 0; j < kBinsPer; ++j) {
                    if (!found && need <= above + c[j]) {
                        sh_digit = (uint32_t)(kBins - 1 - tid * kBinsPer - j);
                        sh_need = need - above;
                        sh_count = c[j];
                        found = true;
                    }
                    above += c[j];
                }
            }
#pragma unroll
            for (int j = 0; j < kBinsPer; ++j) hist[kBins - 1 - tid * kBinsPer - j] = 0;      // for the next digit
            __syncthreads();
            T |= sh_digit << shift;
            need = sh_need;
            bits = shift;
            const uint32_t count = sh_count;
            if (bits == 0) break;
            if (count == need) {           // the whole bin is kept: T is its lowest possible key
                need = (uint32_t)N;
                break;
            }
            if (count <= kDirect) {
#pragma unroll
                for (int j = 0; j < KEYS; ++j)
                    if (in_play(j)) cand[atomicAdd(&sh_cand, 1u)] = key[j];
                __syncthreads();
                const uint32_t mine = lane < (int)count ? cand[lane] : 0u;
                uint32_t gt = 0, eq = 0;
                for (int j = 0; j < (int)count; ++j) {
                    const uint32_t v = __shfl_sync(0xffffffffu, mine, j);
                    gt += v > mine;
                    eq += v == mine;
                }
                const uint32_t hit = __ballot_sync(0xffffffffu, lane < (int)count && gt < need && need <= gt + eq);
                const int at = __ffs((int)hit) - 1;
                T = __shfl_sync(0xffffffffu, mine, at);
                need -= __shfl_sync(0xffffffffu, gt, at);
                break;
            }
        }
    }

    // ---- ordered emit
    uint32_t n_gt = 0, n_eq = 0;
    auto is_gt = [&](int j) { return i0 + j * 32 < N && (keep_all || (!keep_none && key[j] > T)); };
    auto is_eq = [&](int j) { return i0 + j * 32 < N && !keep_all && !keep_none && key[j] == T; };
#pragma unroll
    for (int j = 0; j < KEYS; ++j) {
        n_gt += __popc(__ballot_sync(0xffffffffu, is_gt(j)));
        n_eq += __popc(__ballot_sync(0xffffffffu, is_eq(j)));
    }
    __syncthreads();                       // (warp_a and warp_b are free)
    if (lane == 0) { warp_a[warp] = n_gt; warp_b[warp] = n_eq; }
    __syncthreads();
    uint32_t gt_before = __reduce_add_sync(0xffffffffu, lane < warp ? warp_a[lane] : 0u);
    uint32_t eq_before = __reduce_add_sync(0xffffffffu, lane < warp ? warp_b[lane] : 0u);

    const long list_base = (long)list_first * N;         // 0 unless grouped
    int32_t* keep_out = keep_idx + list_base + cu;
    int32_t* prune_out = prune_idx + list_base + ((long)seg_in * N - cu);
    int32_t* pos_out = pos ? pos + (long)seg * N : nullptr;
    const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < KEYS; ++j) {
        const int i = i0 + j * 32;
        const bool gt = is_gt(j), eq = is_eq(j);
        const uint32_t bg = __ballot_sync(0xffffffffu, gt);
        const uint32_t be = __ballot_sync(0xffffffffu, eq);
        const uint32_t my_gt = gt_before + __popc(bg & lt_mask);
        const uint32_t my_eq = eq_before + __popc(be & lt_mask);
        if (i < N) {
            const bool kept = gt || (eq && my_eq < need);
            const uint32_t kept_before = my_gt + min(my_eq, need);
            if (kept) {
                keep_out[kept_before] = i;
                if (pos_out) pos_out[i] = (int32_t)kept_before;
            } else {
                prune_out[(uint32_t)i - kept_before] = i;
                if (pos_out) pos_out[i] = -1;
            }
        }
        gt_before += __popc(bg);
        eq_before += __popc(be);
    }
}

// As few threads as hold the segment with at most two keys each, up to 1024 threads of up to 16.
template <class... A>
void launch_select(int segments, int N, cudaStream_t st, A... args)
{
    if (N <= 512) select_topk_kernel<256, 2><<<segments, 256, 0, st>>>(args...);
    else if (N <= 1024) select_topk_kernel<512, 2><<<segments, 512, 0, st>>>(args...);
    else if (N <= 2048) select_topk_kernel<1024, 2><<<segments, 1024, 0, st>>>(args...);
    else if (N <= 4096) select_topk_kernel<1024, 4><<<segments, 1024, 0, st>>>(args...);
    else if (N <= 8192) select_topk_kernel<1024, 8><<<segments, 1024, 0, st>>>(args...);
    else select_topk_kernel<1024, 16><<<segments, 1024, 0, st>>>(args...);
}

}  // namespace

extern "C" nova_status nova_select_topk(nova_ctx* ctx, const float* ent, int S, int N,
                                        const int32_t* k, int32_t* keep_idx, int32_t* prune_idx,
                                        int32_t* cu_keep, int32_t* pos, void* stream)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (S < 0 || N < 0) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk: negative size");
    if (N > 16384) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_select_topk: N > 16384");
    if (!cu_keep) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk: null cu_keep");
    NOVA_DEVICE_GUARD(ctx, "nova_select_topk");
    cudaStream_t st = (cudaStream_t)stream;
    if (S == 0 || N == 0) {
        NOVA_CUDA_CHECK(ctx, cudaMemsetAsync(cu_keep, 0, sizeof(int32_t) * (size_t)(S + 1), st));
        return NOVA_OK;
    }
    if (!ent || !k) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk: null pointer");
    long total_keep = 0;
    for (int s = 0; s < S; ++s) {
        if (k[s] < 0 || k[s] > N) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk: k outside [0, N]");
        total_keep += k[s];
    }
    if ((total_keep > 0 && !keep_idx) || (total_keep < (long)S * N && !prune_idx))
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk: null index output");

    int cu = 0;
    for (int s0 = 0; s0 < S; s0 += kMaxSegPerLaunch) {
        const int n = (S - s0 < kMaxSegPerLaunch) ? (S - s0) : kMaxSegPerLaunch;
        SegParams sp;
        memset(&sp, 0, sizeof(sp));
        for (int s = 0; s < n; ++s) sp.k[s] = k[s0 + s];
        {
            nova_launch_scope scope(ctx, NOVA_K_SELECT, st);
            launch_select(n, N, st, ent, N, s0, cu, sp, nullptr, keep_idx, prune_idx, cu_keep, pos, 0);
        }
        for (int s = 0; s < n; ++s) cu += k[s0 + s];
    }
    NOVA_CUDA_CHECK(ctx, cudaGetLastError());
    return NOVA_OK;
}

// The same selection with the keep counts in device memory (written by nova_keep_ratios_device):
// no host value depends on them, so the call needs no synchronisation and can be captured.
extern "C" nova_status nova_select_topk_device(nova_ctx* ctx, const float* ent, int S, int N,
                                               const int32_t* k_dev, int32_t* keep_idx, int32_t* prune_idx,
                                               int32_t* cu_keep, int32_t* pos, void* stream)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (S < 0 || N < 0) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_device: negative size");
    if (N > 16384) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_select_topk_device: N > 16384");
    if (S > 65535) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_select_topk_device: S > 65535");
    if (!cu_keep) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_device: null cu_keep");
    NOVA_DEVICE_GUARD(ctx, "nova_select_topk_device");
    cudaStream_t st = (cudaStream_t)stream;
    if (S == 0 || N == 0) {
        NOVA_CUDA_CHECK(ctx, cudaMemsetAsync(cu_keep, 0, sizeof(int32_t) * (size_t)(S + 1), st));
        return NOVA_OK;
    }
    if (!ent || !k_dev || !keep_idx || !prune_idx)
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_device: null pointer");
    SegParams sp;
    memset(&sp, 0, sizeof(sp));
    {
        nova_launch_scope scope(ctx, NOVA_K_SELECT, st);
        launch_select(S, N, st, ent, N, 0, 0, sp, k_dev, keep_idx, prune_idx, cu_keep, pos, 0);
    }
    NOVA_CUDA_CHECK(ctx, cudaGetLastError());
    return NOVA_OK;
}

// Selection for all layers of a scale at once: G lists (layers) of S segments (images) each.
static nova_status select_grouped(nova_ctx* ctx, const float* ent, int G, int S, int N, const int32_t* k_host,
                                  const int32_t* k_dev, int32_t* keep_idx, int32_t* prune_idx, int32_t* cu_keep,
                                  int32_t* pos, void* stream, const char* who)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (G < 0 || S < 0 || N < 0) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_grouped: negative size");
    if (N > 16384) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_select_topk_grouped: N > 16384");
    if (S > kMaxSegPerLaunch) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_select_topk_grouped: more than 256 segments per list");
    if ((long)G * S > 0x7fffffffL / (N > 0 ? N : 1)) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_select_topk_grouped: too many tokens");
    if (G == 0) return NOVA_OK;
    if (!cu_keep) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_grouped: null cu_keep");
    NOVA_DEVICE_GUARD(ctx, who);
    cudaStream_t st = (cudaStream_t)stream;
    if (S == 0 || N == 0) {
        NOVA_CUDA_CHECK(ctx, cudaMemsetAsync(cu_keep, 0, sizeof(int32_t) * (size_t)G * (S + 1), st));
        return NOVA_OK;
    }
    if (!ent || (!k_host && !k_dev) || !keep_idx || !prune_idx)
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_grouped: null pointer");
    if (k_host)
        for (long i = 0; i < (long)G * S; ++i)
            if (k_host[i] < 0 || k_host[i] > N)
                return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_grouped: k outside [0, N]");
    SegParams sp;
    memset(&sp, 0, sizeof(sp));
    if (k_dev) {
        nova_launch_scope scope(ctx, NOVA_K_SELECT, st);
        launch_select(G * S, N, st, ent, N, 0, 0, sp, k_dev, keep_idx, prune_idx, cu_keep, pos, S);
    } else {
        // the host's counts travel as kernel parameters, 256 per launch: whole lists per launch
        const int lists_per_launch = kMaxSegPerLaunch / S;
        for (int g0 = 0; g0 < G; g0 += lists_per_launch) {
            const int ng = (G - g0 < lists_per_launch) ? (G - g0) : lists_per_launch;
            for (int i = 0; i < ng * S; ++i) sp.k[i] = k_host[(long)g0 * S + i];
            nova_launch_scope scope(ctx, NOVA_K_SELECT, st);
            launch_select(ng * S, N, st, ent, N, g0 * S, 0, sp, nullptr, keep_idx, prune_idx,
                                                                      cu_keep, pos, S);
        }
    }
    NOVA_CUDA_CHECK(ctx, cudaGetLastError());
    return NOVA_OK;
}

extern "C" nova_status nova_select_topk_grouped(nova_ctx* ctx, const float* ent, int G, int S, int N, const int32_t* k,
                                                int32_t* keep_idx, int32_t* prune_idx, int32_t* cu_keep,
                                                int32_t* pos, void* stream)
{
    if (ctx && G > 0 && S > 0 && N > 0 && !k) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_grouped: null k");
    return select_grouped(ctx, ent, G, S, N, k, nullptr, keep_idx, prune_idx, cu_keep, pos, stream, "nova_select_topk_grouped");
}

extern "C" nova_status nova_select_topk_grouped_device(nova_ctx* ctx, const float* ent, int G, int S, int N,
                                                       const int32_t* k_dev, int32_t* keep_idx, int32_t* prune_idx,
                                                       int32_t* cu_keep, int32_t* pos, void* stream)
{
    if (ctx && G > 0 && S > 0 && N > 0 && !k_dev) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_select_topk_grouped_device: null k");
    return select_grouped(ctx, ent, G, S, N, nullptr, k_dev, keep_idx, prune_idx, cu_keep, pos, stream,
                          "nova_select_topk_grouped_device");
}
