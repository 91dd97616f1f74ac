// Eq. 14 on the kept tokens: gather + LayerNorm, QKV projection with K/V cache append,
// attention, output projection + residual, LayerNorm, MLP with tanh-GELU + residual.
// This file holds the small memory-bound kernels (row maps, LayerNorm, kv_len update), the
// workspace layout and the launch sequence; the contractions live in gemm.cu / attention.cu.
#include "common.cuh"

namespace {

// ---- row maps ---------------------------------------------------------------------------
// src_row[r] = b*N + keep_idx[r]            row of x_in feeding compacted row r
// kv_row[r]  = b*Lmax + kv_len[b] + (r - cu_keep[b])   cache row receiving r's k and v
//              (-1 and a SHAPE flag if the image's cache would overflow)
// Both are produced by the first LayerNorm on its way: it needs
// src_row to gather its input anyway.
struct RowMapArgs {
    const int32_t* keep_idx;
    const int32_t* cu_keep;
    const int32_t* kv_len;
    int B, N, Lmax;
    int32_t* src_row;
    int32_t* kv_row;
    int32_t* img_row;     // image of compacted row r
    unsigned int* status;
};

// Per-image modulation of a LayerNorm's output (adaptive LayerNorm): out * (1 + scale[b]) + shift[b].
// scale / shift: [B, C] bf16 or NULL; img_row gives b for the kernels that do not build the maps.
struct LnModArgs {
    const uint4* scale;
    const uint4* shift;
    const int32_t* img_row;
};

// ---- LayerNorm ----------------------------------------------------------------------------
// A row (C <= 64 * 8 * VEC bf16, or half of that with one warp) is the work of one or two warps, in persistent blocks that go
// through the rows in turn. x is read once and out written once; in between the row stays in registers.
// The sums of a row are made in an order that depends on its width alone, so that a token's result is the same to the last bit in any
// launch: 32 partial sums, of the 128-bit pieces l, l + 32, l + 64, ..., the even and the odd features apart, the even added to
// the odd ones, then a butterfly. One warp does that as packed pairs. Of two warps one has the row's even features and the other its odd
// ones: they load alternate pieces, hand each other through shared memory the half that the other needs, and meet again for the
// one addition per lane.
// What bounds it: HBM and L2 at many rows, and instructions close behind; at few the chain list -> row -> two reductions -> store, so
// a thread has little to do and all its loads go out first, gain and bias too. Two warps, in blocks of their own, while all their rows
// run at once with some room left for the next launch (7 of the 8 rows per SM: 1024 rows of 2048 in 3.6 us, with one warp 4.3), and
// where a row is too wide for one warp's registers; else one, which saves the exchange, eight rows to a block: two blocks per SM that load
// their next row before they work on the present one, or three that do not where only those take all rows at once (3277 rows of 2048 over
// inputs larger than L2 6.5 us instead of 7.8; with blocks of two rows 8.4).
// us, one warp per row in blocks of eight rows that end with them -> this, back to back over warm inputs: 256 rows x 1024 2.5 -> 1.8,
// 300 x 2048 4.0 -> 2.4, 1600 x 2048 4.9 -> 4.5, 2252 x 1920 5.1 -> 4.5, 4096 x 2048 8.6 -> 6.6, 8192 x 2048 11.4 -> 10.9, 2048 x 4096
// 13.5 -> 8.2, 2048 x 8192 50 -> 20; over inputs larger than L2 2252 x 1920 5.8 -> 5.3, 4096 x 2048 10.1 -> 8.3, 8192 x 2048
// 15.0 -> 13.6 (4.9 TB/s), 8192 x 1024 8.0 -> 7.8. With two warps that each add up their own pieces 1.9, 2.3, 4.4, 4.9, 6.7, 10.4, 7.8, 15 and
// 5.9, 7.9, 13.3, 8.9, but other last bits.
constexpr int kLnThreads = 64;         // two warps per row
constexpr int kLnBlocksPerSm = 8;
constexpr int kLnOneThreads = 256;     // one warp per row
constexpr int kLnOneRows = kLnOneThreads / 32;
constexpr int kLnOneVec = 8;           // widest row of one warp: 8 pieces per lane, C = 2048

__device__ __forceinline__ uint4 ld_stream(const uint4* p)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// A row's sum from its two warps' halves: lane by lane, then over the lanes. Two slots of 64 floats in turn: all have read one when
// they meet at the other's barrier.
__device__ __forceinline__ float row_sum(float half, float* slot)
{
    slot[threadIdx.x] = half;
    __syncthreads();
    return warp_sum(half + slot[threadIdx.x ^ 32]);
}

__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float lo_f32(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_f32(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ uint64_t bf16x2_f32x2(uint32_t w) { return pack_f32x2(lo_f32(w), hi_f32(w)); }

// VEC: 128-bit pieces per thread. AHEAD: the next row is loaded before the present one is worked on. (Two warps seldom have a second
// one, only with a bound on a device-side count: without the code for it 300 rows of 2048 take 2.4 us instead of 2.8, and 4096 rows
// 7.5 instead of 8.1.)
template <int VEC, int WARPS, bool AHEAD, bool MAPS, bool MOD>
__global__ void __launch_bounds__(WARPS == 1 ? kLnOneThreads : kLnThreads, WARPS == 2 ? kLnBlocksPerSm : AHEAD ? 2 : 3)
layernorm_rows(const uint4* x, const uint4* gamma, const uint4* beta, float eps, int M, const int32_t* m_dev, int vec_per_row,
               uint4* __restrict__ out, const RowMapArgs maps, const LnModArgs mod)
{
    constexpr int T = 32 * WARPS, kRows = WARPS == 1 ? kLnOneRows : 1;      // threads of a row, rows of a block
    constexpr bool kGainAhead = WARPS == 2 && VEC <= 4;      // gain and bias are loaded early where there are registers for them
    __shared__ uint2 given[WARPS == 2 ? VEC * kLnThreads : 1];
    __shared__ float part[2 * kLnThreads];
    pdl_launch_dependents();
    const int tid = threadIdx.x & (T - 1);
    // Gain and bias come from HBM (each layer has its own): brought to L2 while the launch before this one ends. A
    // prefetch hands nothing to this kernel, so whoever still writes them does no harm. With few
    // rows the launch is a chain of latencies, of which this takes one off: a 16-layer 256x256 generation 9412 ->
    // 9316 us, a 20x20 scale of one image 3097 -> 3058.
    for (int c = threadIdx.x * 8; c < vec_per_row; c += T * kRows * 8) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(gamma + c));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(beta + c));
    }
    pdl_wait();
    if (m_dev) M = min(M, *m_dev);      // the host knows only an upper bound
    // row r of the launch: its row of x and its image
    auto locate = [&](int r, long& src, int& img) {
        src = r;
        img = MOD && !MAPS ? mod.img_row[r] : 0;
        if (MAPS) {
            const int token = maps.keep_idx[r];
            int lo = 0, hi = maps.B;        // largest b with cu_keep[b] <= r
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (maps.cu_keep[mid] <= r) lo = mid; else hi = mid;
            }
            src = (long)lo * maps.N + token;
            img = lo;
        }
    };
    auto load = [&](long src, uint4 (&d)[VEC]) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const int c = i * T + tid;
            d[i] = (c < vec_per_row) ? ld_stream(x + src * vec_per_row + c) : make_uint4(0, 0, 0, 0);
        }
    };
    int r = blockIdx.x * kRows + (WARPS == 1 ? threadIdx.x / T : 0);
    if (r >= M) return;
    long src, src_next = 0;
    int img, img_next = 0;
    uint4 raw[VEC], next[VEC], g[VEC], bt[VEC];
    locate(r, src, img);
    load(src, raw);
    if (kGainAhead) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const int c = i * T + tid;
            if (c < vec_per_row) { g[i] = gamma[c]; bt[i] = beta[c]; }
        }
    }
    const float n = (float)(vec_per_row * 8);
    while (true) {
        const int r_next = r + (int)gridDim.x * kRows;
        if (r_next < M) {
            locate(r_next, src_next, img_next);
            if (AHEAD) load(src_next, next);
        }
        if (MAPS && tid == 0) {
            const int c0 = maps.cu_keep[img], k_b = maps.cu_keep[img + 1] - c0, len = maps.kv_len[img];
            maps.src_row[r] = (int32_t)src;
            maps.img_row[r] = img;
            if (len + k_b > maps.Lmax) {
                maps.kv_row[r] = -1;
                atomicOr(maps.status, NOVA_DEV_SHAPE);
            } else {
                maps.kv_row[r] = img * maps.Lmax + len + (r - c0);
            }
        }
        float mean, rstd;
        uint2 f[WARPS == 2 ? 2 * VEC : 1];
        const bool odd = WARPS == 2 && tid >= 32;
        if constexpr (WARPS == 1) {
            uint64_t sum = pack_f32x2(0.f, 0.f), sq = sum;
            float even_f, odd_f;
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
#pragma unroll
                for (int q = 0; q < 4; ++q) sum = add_f32x2(sum, bf16x2_f32x2(w[q]));
            }
            unpack_f32x2(sum, even_f, odd_f);
            mean = warp_sum(even_f + odd_f) / n;
            const uint64_t neg_mean = pack_f32x2(-mean, -mean);
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                if (i * T + tid < vec_per_row) {
                    const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint64_t d = add_f32x2(bf16x2_f32x2(w[q]), neg_mean);
                        sq = fma_f32x2(d, d, sq);
                    }
                }
            }
            unpack_f32x2(sq, even_f, odd_f);
            rstd = rsqrtf(warp_sum(even_f + odd_f) / n + eps);
        } else {
            // f: this warp's features of the whole row, two to a word
            const uint32_t keep = odd ? 0x7632 : 0x5410, give = odd ? 0x5410 : 0x7632;
#pragma unroll
            for (int i = 0; i < VEC; ++i)
                given[i * T + tid] = make_uint2(__byte_perm(raw[i].x, raw[i].y, give), __byte_perm(raw[i].z, raw[i].w, give));
            __syncthreads();
            float sum = 0.f, sq = 0.f;
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                const uint2 kept = make_uint2(__byte_perm(raw[i].x, raw[i].y, keep), __byte_perm(raw[i].z, raw[i].w, keep));
                const uint2 got = given[i * T + (tid ^ 32)];
                f[2 * i] = odd ? got : kept;
                f[2 * i + 1] = odd ? kept : got;
#pragma unroll
                for (int j = 2 * i; j < 2 * i + 2; ++j) {
                    sum += lo_f32(f[j].x);
                    sum += hi_f32(f[j].x);
                    sum += lo_f32(f[j].y);
                    sum += hi_f32(f[j].y);
                }
            }
            mean = row_sum(sum, part) / n;
#pragma unroll
            for (int j = 0; j < 2 * VEC; ++j) {
                if (j * 32 + (tid & 31) < vec_per_row) {
                    const float d0 = lo_f32(f[j].x) - mean, d1 = hi_f32(f[j].x) - mean, d2 = lo_f32(f[j].y) - mean, d3 = hi_f32(f[j].y) - mean;
                    sq = fmaf(d0, d0, sq);
                    sq = fmaf(d1, d1, sq);
                    sq = fmaf(d2, d2, sq);
                    sq = fmaf(d3, d3, sq);
                }
            }
            rstd = rsqrtf(row_sum(sq, part + kLnThreads) / n + eps);
        }
        // (x - mean) * rstd = x * rstd + shift
        const float shift = -mean * rstd;
        const uint64_t rstd2 = pack_f32x2(rstd, rstd), shift2 = pack_f32x2(shift, shift);
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const int c = i * T + tid;
            if (c < vec_per_row) {
                if (!kGainAhead) { g[i] = gamma[c]; bt[i] = beta[c]; }
                uint64_t v[4];
                if constexpr (WARPS == 1) {
                    const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q] = bf16x2_f32x2(w[q]);
                } else {
                    // the piece from the two halves (the one that was given away is still in shared memory)
                    const uint2 kept = odd ? f[2 * i + 1] : f[2 * i], gave = given[i * T + tid];
                    const uint2 ev = odd ? gave : kept, od = odd ? kept : gave;
                    v[0] = pack_f32x2(lo_f32(ev.x), lo_f32(od.x));
                    v[1] = pack_f32x2(hi_f32(ev.x), hi_f32(od.x));
                    v[2] = pack_f32x2(lo_f32(ev.y), lo_f32(od.y));
                    v[3] = pack_f32x2(hi_f32(ev.y), hi_f32(od.y));
                }
                const uint32_t gw[4] = {g[i].x, g[i].y, g[i].z, g[i].w}, bw[4] = {bt[i].x, bt[i].y, bt[i].z, bt[i].w};
                uint32_t o[4];
                uint32_t sc[4] = {0, 0, 0, 0}, sh[4] = {0, 0, 0, 0};        // bf16 zeros: no modulation
                if (MOD && mod.scale) { const uint4 t = mod.scale[(long)img * vec_per_row + c]; sc[0] = t.x; sc[1] = t.y; sc[2] = t.z; sc[3] = t.w; }
                if (MOD && mod.shift) { const uint4 t = mod.shift[(long)img * vec_per_row + c]; sh[0] = t.x; sh[1] = t.y; sh[2] = t.z; sh[3] = t.w; }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float y0, y1;
                    unpack_f32x2(fma_f32x2(fma_f32x2(v[q], rstd2, shift2), bf16x2_f32x2(gw[q]), bf16x2_f32x2(bw[q])), y0, y1);
                    if (MOD) {
                        y0 = fmaf(y0, 1.f + lo_f32(sc[q]), lo_f32(sh[q]));
                        y1 = fmaf(y1, 1.f + hi_f32(sc[q]), hi_f32(sh[q]));
                    }
                    __nv_bfloat162 t = __floats2bfloat162_rn(y0, y1);
                    o[q] = *reinterpret_cast<uint32_t*>(&t);
                }
                out[(long)r * vec_per_row + c] = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
        if (r_next >= M) return;
        r = r_next;
        src = src_next;
        img = img_next;
        if (AHEAD) {
#pragma unroll
            for (int i = 0; i < VEC; ++i) raw[i] = next[i];
        } else {
            load(src, raw);
        }
    }
}

// ---- query/key normalisation and rotary embedding -----------------------------------------------
// After the QKV projection, per kept row r and head: q (in the q buffer) and the row's new key (in
// its cache row) are, in place, scaled to unit L2 norm times a per-channel gain, then rotated pair by
// pair by the angle of the token's position in the scale. One warp per (row, head); a lane holds DH / 32
// consecutive channels, i.e. whole pairs.
template <int DH>
__global__ void __launch_bounds__(256)
qk_transform_kernel(__nv_bfloat16* __restrict__ q, __nv_bfloat16* __restrict__ k_cache, const int32_t* kv_row,
                    const int32_t* keep_idx, int M, const int32_t* m_dev, int C, int n_heads,
                    const __nv_bfloat16* gain_q, const __nv_bfloat16* gain_k, float eps,
                    const float* rope_cos, const float* rope_sin)
{
    pdl_launch_dependents();
    pdl_wait();
    constexpr int PER = DH / 32;          // 2 or 4 channels per lane
    const int lane = threadIdx.x & 31;
    const long wid = (long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (m_dev) M = min(M, *m_dev);
    if (wid >= (long)M * n_heads) return;
    const int r = (int)(wid / n_heads), hd = (int)(wid - (long)r * n_heads);
    const int pos = keep_idx[r];
    const int ch = hd * DH + lane * PER;
    float cs[PER / 2], sn[PER / 2];
    if (rope_cos) {
#pragma unroll
        for (int i = 0; i < PER / 2; ++i) {
            cs[i] = rope_cos[(long)pos * (DH / 2) + lane * (PER / 2) + i];
            sn[i] = rope_sin[(long)pos * (DH / 2) + lane * (PER / 2) + i];
        }
    }
    auto transform = [&](__nv_bfloat16* row, const __nv_bfloat16* gain) {
        float v[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) v[i] = __bfloat162float(row[ch + i]);
        if (gain) {
            float ss = 0.f;
#pragma unroll
            for (int i = 0; i < PER; ++i) ss = fmaf(v[i], v[i], ss);
            ss = warp_sum(ss);
            const float inv = 1.f / fmaxf(sqrtf(ss), eps);
#pragma unroll
            for (int i = 0; i < PER; ++i) v[i] = v[i] * inv * __bfloat162float(gain[ch + i]);
        }
        if (rope_cos) {
#pragma unroll
            for (int i = 0; i < PER / 2; ++i) {
                const float a = v[2 * i], b = v[2 * i + 1];
                v[2 * i] = a * cs[i] - b * sn[i];
                v[2 * i + 1] = a * sn[i] + b * cs[i];
            }
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) row[ch + i] = __float2bfloat16_rn(v[i]);
    };
    transform(q + (long)r * C, gain_q);
    const int kr = kv_row[r];
    if (kr >= 0) transform(k_cache + (long)kr * C, gain_k);      // a row of an overflowing image has no cache row
}

struct Workspace {
    int32_t* src_row;
    int32_t* kv_row;
    int32_t* img_row;
    __nv_bfloat16 *h, *q, *o, *x1, *f;
    size_t bytes;
};

inline size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

Workspace carve(void* base, int M, int C, int F)
{
    Workspace w;
    size_t off = 0;
    auto take = [&](size_t bytes) { void* p = base ? (char*)base + off : nullptr; off += align_up(bytes); return p; };
    const size_t Mp = (size_t)((M + 127) / 128) * 128;   // whole 128-row tiles
    w.src_row = (int32_t*)take(Mp * 4);
    w.kv_row = (int32_t*)take(Mp * 4);
    w.h = (__nv_bfloat16*)take(Mp * C * 2);
    w.q = (__nv_bfloat16*)take(Mp * C * 2);
    w.o = (__nv_bfloat16*)take(Mp * C * 2);
    w.x1 = (__nv_bfloat16*)take(Mp * C * 2);
    w.f = (__nv_bfloat16*)take(Mp * (size_t)F * 2);
    w.img_row = (int32_t*)take(Mp * 4);
    w.bytes = off;
    return w;
}

bool shape_ok(const nova_block_shape* s)
{
    if (!s || s->B < 1 || s->N < 1 || s->C < 64 || s->n_heads < 1 || s->F < 64 || s->Lmax < 1 || s->M < 0) return false;
    if (s->C % 64 || s->F % 64 || s->C % s->n_heads) return false;
    const int dh = s->C / s->n_heads;
    if (dh != 64 && dh != 128) return false;
    if (s->C > 8192) return false;
    if ((long)s->M > (long)s->B * s->N) return false;
    return true;
}

}  // namespace

static nova_status launch_ln(nova_ctx* ctx, const __nv_bfloat16* x, const RowMapArgs* maps, const LnModArgs& mod,
                             const __nv_bfloat16* g, const __nv_bfloat16* b, float eps, int M, const int32_t* m_dev,
                             int C, __nv_bfloat16* out, cudaStream_t st)
{
    if (M <= 0) return NOVA_OK;
    const int vec = C / 8;
    const int fit = ctx->num_sms * kLnBlocksPerSm;
    // (of a bound on a device-side count a quarter: a last scale keeps about that)
    const bool one = (m_dev ? M / 4 : M) > fit - fit / 8 && vec <= 32 * kLnOneVec;
    const int one_blocks = (M + kLnOneRows - 1) / kLnOneRows;
    const bool ahead = m_dev || one_blocks <= 2 * ctx->num_sms || one_blocks > 3 * ctx->num_sms;
    const dim3 grid(one ? min(one_blocks, (ahead ? 2 : 3) * ctx->num_sms) : min(M, fit)), block(one ? kLnOneThreads : kLnThreads);
    RowMapArgs none;
    memset(&none, 0, sizeof(none));
    cudaError_t le = cudaSuccess;
    nova_launch_scope scope(ctx, NOVA_K_LAYERNORM, st);
#define NOVA_LN_LAUNCH(V, W, AHEAD, MAPS, MOD, MAPARG)                                                                     \
    le = nova_launch_pdl(layernorm_rows<V, W, AHEAD, MAPS, MOD>, grid, block, 0, st, 0, (const uint4*)x, (const uint4*)g, (const uint4*)b, eps, M, m_dev, vec, (uint4*)out, MAPARG, mod)
#define NOVA_LN_CASE(V, W, AHEAD)                                                                                          \
    do {                                                                                                         \
        if (maps && modulated) NOVA_LN_LAUNCH(V, W, AHEAD, true, true, *maps);                                             \
        else if (maps) NOVA_LN_LAUNCH(V, W, AHEAD, true, false, *maps);                                                    \
        else if (modulated) NOVA_LN_LAUNCH(V, W, AHEAD, false, true, none);                                                \
        else NOVA_LN_LAUNCH(V, W, AHEAD, false, false, none);                                                              \
    } while (0)
    const bool modulated = mod.scale || mod.shift;
    if (one && ahead && vec <= 32 * 4) NOVA_LN_CASE(4, 1, true);
    else if (one && ahead && vec <= 32 * 6) NOVA_LN_CASE(6, 1, true);
    else if (one && ahead) NOVA_LN_CASE(kLnOneVec, 1, true);
    else if (one && vec <= 32 * 4) NOVA_LN_CASE(4, 1, false);
    else if (one && vec <= 32 * 6) NOVA_LN_CASE(6, 1, false);
    else if (one) NOVA_LN_CASE(kLnOneVec, 1, false);
    else if (vec <= 64 * 2) NOVA_LN_CASE(2, 2, false);
    else if (vec <= 64 * 3) NOVA_LN_CASE(3, 2, false);
    else if (vec <= 64 * 4) NOVA_LN_CASE(4, 2, false);
    else if (vec <= 64 * 8) NOVA_LN_CASE(8, 2, false);
    else if (vec <= 64 * 16) NOVA_LN_CASE(16, 2, false);
    else return nova_fail(ctx, NOVA_ERR_SHAPE, "layernorm: C > 8192");
#undef NOVA_LN_LAUNCH
#undef NOVA_LN_CASE
    NOVA_CUDA_CHECK(ctx, le);
    return NOVA_OK;
}

extern "C" size_t nova_block_workspace_bytes(const nova_block_shape* s)
{
    if (!shape_ok(s)) return 0;
    return carve(nullptr, s->M, s->C, s->F).bytes;
}

// Where the block's output goes when the last GEMM scatters it straight into the token map (Eq. 15-16
// on the kept rows) instead of writing the compacted y_kept.
struct ScatterOut {
    void* x_out;        // [B, N, C]: kept rows receive the layer output
    void* cache_out;    // [B, N, C] or NULL: kept rows receive output - input
    // the pruned rows of both, from the previous scale's residual cache
    const int32_t* prune_idx;
    const void* cache_prev;
    int hp, wp, h, w;
};

// m_on_device: s->M is only an upper bound of the kept rows (it sizes grids, tensor maps and the
// workspace); every kernel takes the true count from cu_keep[B] on the device.
static nova_status block_forward(nova_ctx* ctx, const nova_block_weights* w, const nova_block_modulation* mod,
                                 const nova_block_shape* s, const void* x_in,
                                 const int32_t* keep_idx, const int32_t* cu_keep,
                                 void* k_cache, void* v_cache, int32_t* kv_len,
                                 int append_kv, void* y_kept, void* stream, bool m_on_device,
                                 const ScatterOut* scatter = nullptr, const nova_block_extras* ext = nullptr)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (!w || !s) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_block_forward: null weights or shape");
    if (!shape_ok(s)) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_pruned_block_forward: unsupported shape");
    if (s->M == 0) return NOVA_OK;
    if (!x_in || !keep_idx || !cu_keep || !k_cache || !v_cache || !kv_len || (!y_kept && !scatter))
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_block_forward: null tensor");
    const void* wp[] = {w->ln1_g, w->ln1_b, w->w_qkv, w->b_qkv, w->w_o, w->b_o,
                        w->ln2_g, w->ln2_b, w->w_fc1, w->b_fc1, w->w_fc2, w->b_fc2};
    for (const void* ptr : wp) {
        if (!ptr) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_block_forward: null weight");
        if (!nova_aligned16(ptr)) return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_pruned_block_forward: weight not 16-byte aligned");
    }
    if (!nova_aligned16(x_in) || !nova_aligned16(k_cache) || !nova_aligned16(v_cache) || !nova_aligned16(y_kept))
        return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_pruned_block_forward: tensor not 16-byte aligned");
    Workspace ws = carve(ctx->workspace, s->M, s->C, s->F);
    if (!ctx->workspace || ctx->workspace_bytes < ws.bytes)
        return nova_fail(ctx, NOVA_ERR_WORKSPACE, "nova_pruned_block_forward: workspace missing or too small");
    const bool rope = ext && (ext->rope_cos || ext->rope_sin);
    const bool qk_norm = ext && (ext->qk_gain_q || ext->qk_gain_k);
    const bool cross = ext && ext->w_q2;
    if (rope && (!ext->rope_cos || !ext->rope_sin)) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_block_forward_ext: rope_cos and rope_sin go together");
    if (qk_norm && (!ext->qk_gain_q || !ext->qk_gain_k)) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_block_forward_ext: qk_gain_q and qk_gain_k go together");
    if (cross) {
        const void* cp[] = {ext->lnc_g, ext->lnc_b, ext->w_q2, ext->b_q2, ext->w_o2, ext->b_o2, ext->cond_k, ext->cond_v, ext->cond_len};
        for (const void* ptr : cp)
            if (!ptr) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_block_forward_ext: incomplete cross-attention weights");
        if (ext->Lc_max < 1) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_block_forward_ext: Lc_max < 1");
    }
    if (ext) {
        const void* ep[] = {ext->rope_cos, ext->rope_sin, ext->qk_gain_q, ext->qk_gain_k, ext->lnc_g, ext->lnc_b, ext->w_q2,
                            ext->b_q2, ext->w_o2, ext->b_o2, ext->cond_k, ext->cond_v};
        for (const void* ptr : ep)
            if (!nova_aligned16(ptr)) return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_pruned_block_forward_ext: tensor not 16-byte aligned");
    }
    NOVA_DEVICE_GUARD(ctx, "nova_pruned_block_forward");

    cudaStream_t st = (cudaStream_t)stream;
    {
        const nova_status chk = nova_debug_check_lists(ctx, "nova_pruned_block_forward", keep_idx, nullptr, cu_keep,
                                                       s->B, s->N, s->M, !m_on_device, st);
        if (chk != NOVA_OK) return chk;
    }
    const int M = s->M, C = s->C, F = s->F;
    typedef const __nv_bfloat16* cbf;
    typedef __nv_bfloat16* bf;

    const int32_t* m_dev = m_on_device ? cu_keep + s->B : nullptr;
    nova_block_modulation md;
    memset(&md, 0, sizeof(md));
    if (mod) md = *mod;
    const void* mp[] = {md.shift1, md.scale1, md.gate1, md.shift2, md.scale2, md.gate2};
    for (const void* ptr : mp)
        if (!nova_aligned16(ptr)) return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_pruned_block_forward: modulation not 16-byte aligned");
    LnModArgs ln1_mod = {(const uint4*)md.scale1, (const uint4*)md.shift1, ws.img_row};
    LnModArgs ln2_mod = {(const uint4*)md.scale2, (const uint4*)md.shift2, ws.img_row};
    nova_status rc;
    // h = LN1(gathered rows); the same kernel writes the row maps the GEMM epilogues use
    RowMapArgs maps;
    maps.keep_idx = keep_idx; maps.cu_keep = cu_keep; maps.kv_len = kv_len; maps.B = s->B; maps.N = s->N;
    maps.Lmax = s->Lmax; maps.src_row = ws.src_row; maps.kv_row = ws.kv_row; maps.img_row = ws.img_row; maps.status = ctx->dev_status;
    rc = launch_ln(ctx, (cbf)x_in, &maps, ln1_mod, (cbf)w->ln1_g, (cbf)w->ln1_b, w->eps, M, m_dev, C, ws.h, st);
    if (rc) return rc;
    // [q | k | v] = h W_qkv^T + b; k, v go straight to their cache rows
    nova_gemm_args g;
    memset(&g, 0, sizeof(g));
    g.A = ws.h; g.W = (cbf)w->w_qkv; g.bias = (cbf)w->b_qkv; g.M = M; g.m_dev = m_dev; g.N = 3 * C; g.K = C;
    // (count_settled only for the GEMMs after this one: LN1 lets this one in before its own wait, and the kernel that writes
    // the counts may be the one before LN1)
    g.epilogue = NOVA_EPI_QKV; g.cat = NOVA_K_GEMM_QKV; g.out = ws.q; g.C = C; g.k_cache = (bf)k_cache; g.v_cache = (bf)v_cache; g.kv_row = ws.kv_row;
    rc = nova_launch_gemm(ctx, g, st);
    if (rc) return rc;
    if (rope || qk_norm) {
        // q and the new keys, in place: unit norm times gain, then the rotation of the token's position
        const long warps = (long)M * s->n_heads;
        const unsigned blocks = (unsigned)((warps + 7) / 8);
        typedef const float* cfl;
        cudaError_t qe;
        nova_launch_scope scope(ctx, NOVA_K_LAYERNORM, st);
        if (C / s->n_heads == 64)
            qe = nova_launch_pdl(qk_transform_kernel<64>, dim3(blocks), dim3(256), 0, st, 0, ws.q, (bf)k_cache, ws.kv_row, keep_idx, M, m_dev, C, s->n_heads,
                                                          (cbf)ext->qk_gain_q, (cbf)ext->qk_gain_k, ext->qk_eps,
                                                          (cfl)ext->rope_cos, (cfl)ext->rope_sin);
        else
            qe = nova_launch_pdl(qk_transform_kernel<128>, dim3(blocks), dim3(256), 0, st, 0, ws.q, (bf)k_cache, ws.kv_row, keep_idx, M, m_dev, C, s->n_heads,
                                                           (cbf)ext->qk_gain_q, (cbf)ext->qk_gain_k, ext->qk_eps,
                                                           (cfl)ext->rope_cos, (cfl)ext->rope_sin);
        NOVA_CUDA_CHECK(ctx, qe);
    }
    // o = softmax(q K^T / sqrt(dh)) V
    nova_attn_args a;
    a.q = ws.q; a.k_cache = (cbf)k_cache; a.v_cache = (cbf)v_cache; a.cu_keep = cu_keep; a.kv_len = kv_len;
    a.o = ws.o; a.B = s->B; a.C = C; a.n_heads = s->n_heads; a.Lmax = s->Lmax; a.M = M;
    // neither the projection's output buffer nor the MLP's hidden buffer is in use yet, and they lie
    // next to each other: together they hold the partial results of a key-split last wave
    a.scratch = ws.x1;
    a.scratch_bytes = (size_t)((char*)ws.f - (char*)ws.x1) + (size_t)((M + 127) / 128) * 128 * (size_t)F * 2;
    a.cache_only = false;
    rc = nova_launch_attention(ctx, a, st);
    if (rc) return rc;
    // x1 = Xc + o W_o^T + b_o
    memset(&g, 0, sizeof(g));
    g.A = ws.o; g.W = (cbf)w->w_o; g.bias = (cbf)w->b_o; g.M = M; g.m_dev = m_dev; g.N = C; g.K = C;
    g.epilogue = NOVA_EPI_BIAS_RES; g.cat = NOVA_K_GEMM_PROJ; g.out = ws.x1; g.res = (cbf)x_in; g.res_row = ws.src_row;
    g.count_settled = true;
    g.gate = (cbf)md.gate1; g.img_row = ws.img_row;
    rc = nova_launch_gemm(ctx, g, st);
    if (rc) return rc;
    if (cross) {
        // x1 <- x1 + softmax(q2 Kc^T / sqrt(dh)) Vc W_o2^T + b_o2 with q2 = LN(x1) W_q2^T + b_q2: the same
        // kernels once more, on buffers that are free at this point (h, q, o), the keys and values being
        // the image's condition tokens and nothing else
        LnModArgs none_mod = {nullptr, nullptr, ws.img_row};
        rc = launch_ln(ctx, ws.x1, nullptr, none_mod, (cbf)ext->lnc_g, (cbf)ext->lnc_b, w->eps, M, m_dev, C, ws.h, st);
        if (rc) return rc;
        memset(&g, 0, sizeof(g));
        g.A = ws.h; g.W = (cbf)ext->w_q2; g.bias = (cbf)ext->b_q2; g.M = M; g.m_dev = m_dev; g.N = C; g.K = C;
        g.epilogue = NOVA_EPI_QKV; g.cat = NOVA_K_GEMM_QKV; g.out = ws.q; g.C = C; g.kv_row = ws.kv_row;   // all columns are q
        g.count_settled = true;
        rc = nova_launch_gemm(ctx, g, st);
        if (rc) return rc;
        nova_attn_args ca;
        ca.q = ws.q; ca.k_cache = (cbf)ext->cond_k; ca.v_cache = (cbf)ext->cond_v; ca.cu_keep = cu_keep; ca.kv_len = ext->cond_len;
        ca.o = ws.o; ca.B = s->B; ca.C = C; ca.n_heads = s->n_heads; ca.Lmax = ext->Lc_max; ca.M = M;
        ca.scratch = nullptr; ca.scratch_bytes = 0;      // x1 is live: no room for a key-split wave
        ca.cache_only = true;
        rc = nova_launch_attention(ctx, ca, st);
        if (rc) return rc;
        memset(&g, 0, sizeof(g));
        g.A = ws.o; g.W = (cbf)ext->w_o2; g.bias = (cbf)ext->b_o2; g.M = M; g.m_dev = m_dev; g.N = C; g.K = C;
        g.epilogue = NOVA_EPI_BIAS_RES; g.cat = NOVA_K_GEMM_PROJ; g.out = ws.x1; g.res = ws.x1; g.res_row = nullptr;   // in place
        g.count_settled = true;
        rc = nova_launch_gemm(ctx, g, st);
        if (rc) return rc;
    }
    // h = LN2(x1)
    rc = launch_ln(ctx, ws.x1, nullptr, ln2_mod, (cbf)w->ln2_g, (cbf)w->ln2_b, w->eps, M, m_dev, C, ws.h, st);
    if (rc) return rc;
    // The pruned rows depend on nothing that the block computes. With `beside` FC1 lets their kernel in as soon as it has
    // passed its wait, when everything up to LN2 has ended; FC1 itself neither writes what it reads nor reads what it
    // writes. It then runs in the registers and the memory bandwidth that FC1 leaves, one block per SM, which is worth it
    // where FC1 takes longer than that: about 110 rows of 2048 a microsecond against 2 M F C / 1.3e15 s, even at M F = 2885 pruned
    // rows, and a few per cent more here. Otherwise, and
    // where the kept count is not known here, it follows the last GEMM. us after -> beside: a 20x20 scale of one image, 32 layers
    // of 2048, 2923 -> 2681, a 32x32 scale of four, 30 layers of 1920, 8843 -> 8750, a 16-layer 256x256 generation 9070 -> 8840;
    // with 3072 pruned rows for 1024 kept, 64x64 tokens (M F = 2731 pruned), 6674 -> 7087, with 13107 for 3277 (2048) 33.8 -> 34.4 ms; the
    // first two have M F = 24600 and 9400 pruned. With 8192 kept rows, where the GEMMs run at the power limit, it makes no
    // difference (39.7 ms either way); between that and the largest that was timed, 3277, the line at 4096 is a choice.
    // Not with event brackets around either of the two: events keep launches apart, and one block per SM alone is slow (a bracketed 64x64
    // scale of one image, 2048 kept, 11.7 -> 12.4 ms).
    const long pruned = (long)s->B * s->N - M;
    const bool apart = ctx->profiling && (ctx->prof_mask & (1ull << NOVA_K_GEMM_FC1 | 1ull << NOVA_K_RESTORE));
    const bool beside = scatter && !m_on_device && !apart && pruned > 0 && M <= 4096 && pruned * 3072 < (long)M * F;
    auto restore = [&](bool wait_last) {
        return nova_restore_pruned_rows(ctx, x_in, scatter->prune_idx, cu_keep, scatter->cache_prev, scatter->hp, scatter->wp,
                                        scatter->h, scatter->w, C, s->B, M, m_on_device, scatter->x_out, scatter->cache_out, stream, wait_last);
    };
    // f = GELU(h W_fc1^T + b_fc1)
    memset(&g, 0, sizeof(g));
    g.A = ws.h; g.W = (cbf)w->w_fc1; g.bias = (cbf)w->b_fc1; g.M = M; g.m_dev = m_dev; g.N = F; g.K = C;
    g.epilogue = NOVA_EPI_BIAS_GELU; g.cat = NOVA_K_GEMM_FC1; g.out = ws.f;
    g.count_settled = true;
    g.early_trigger = beside;
    rc = nova_launch_gemm(ctx, g, st);
    if (rc) return rc;
    if (beside) {
        rc = restore(true);
        if (rc) return rc;
    }
    // y = x1 + f W_fc2^T + b_fc2
    memset(&g, 0, sizeof(g));
    g.A = ws.f; g.W = (cbf)w->w_fc2; g.bias = (cbf)w->b_fc2; g.M = M; g.m_dev = m_dev; g.N = C; g.K = F;
    g.epilogue = NOVA_EPI_BIAS_RES; g.cat = NOVA_K_GEMM_FC2; g.out = (bf)y_kept; g.res = ws.x1; g.res_row = nullptr;
    g.count_settled = true;
    g.gate = (cbf)md.gate2; g.img_row = ws.img_row;
    if (scatter) {
        // kept row r is token src_row[r] of the map: x_out[token] = y, cache_out[token] = y - x_in[token]
        g.out = (bf)scatter->x_out; g.out_row = ws.src_row;
        g.diff_in = (cbf)x_in; g.diff_out = (bf)scatter->cache_out;
    }
    if (append_kv) {
        // the last kernel of the block also advances kv_len: every reader of the old lengths (row
        // maps, attention) ran in an earlier kernel of this call
        g.adv_cu_keep = cu_keep; g.adv_kv_len = kv_len; g.adv_B = s->B; g.adv_Lmax = s->Lmax;
    }
    rc = nova_launch_gemm(ctx, g, st);
    if (rc) return rc;
    if (scatter && !beside) return restore(false);
    return NOVA_OK;
}

extern "C" nova_status nova_pruned_block_forward(nova_ctx* ctx, const nova_block_weights* w,
                                                 const nova_block_shape* s, const void* x_in,
                                                 const int32_t* keep_idx, const int32_t* cu_keep,
                                                 void* k_cache, void* v_cache, int32_t* kv_len,
                                                 int append_kv, void* y_kept, void* stream)
{
    return block_forward(ctx, w, nullptr, s, x_in, keep_idx, cu_keep, k_cache, v_cache, kv_len, append_kv, y_kept, stream, false);
}

extern "C" nova_status nova_pruned_block_forward_device(nova_ctx* ctx, const nova_block_weights* w,
                                                        const nova_block_shape* s, const void* x_in,
                                                        const int32_t* keep_idx, const int32_t* cu_keep,
                                                        void* k_cache, void* v_cache, int32_t* kv_len,
                                                        int append_kv, void* y_kept, void* stream)
{
    return block_forward(ctx, w, nullptr, s, x_in, keep_idx, cu_keep, k_cache, v_cache, kv_len, append_kv, y_kept, stream, true);
}

extern "C" nova_status nova_pruned_block_forward_adaln(nova_ctx* ctx, const nova_block_weights* w,
                                                       const nova_block_modulation* mod,
                                                       const nova_block_shape* s, const void* x_in,
                                                       const int32_t* keep_idx, const int32_t* cu_keep,
                                                       void* k_cache, void* v_cache, int32_t* kv_len,
                                                       int append_kv, void* y_kept, int m_on_device, void* stream)
{
    return block_forward(ctx, w, mod, s, x_in, keep_idx, cu_keep, k_cache, v_cache, kv_len, append_kv, y_kept, stream,
                         m_on_device != 0);
}

extern "C" nova_status nova_pruned_block_forward_ext(nova_ctx* ctx, const nova_block_weights* w,
                                                     const nova_block_modulation* mod, const nova_block_extras* ext,
                                                     const nova_block_shape* s, const void* x_in,
                                                     const int32_t* keep_idx, const int32_t* cu_keep,
                                                     void* k_cache, void* v_cache, int32_t* kv_len,
                                                     int append_kv, void* y_kept, int m_on_device, void* stream)
{
    return block_forward(ctx, w, mod, s, x_in, keep_idx, cu_keep, k_cache, v_cache, kv_len, append_kv, y_kept, stream,
                         m_on_device != 0, nullptr, ext);
}

// Eq. 14 followed by Eq. 15-16 for one layer: the block on the kept rows with its last GEMM writing
// the kept rows of x_out / cache_out directly, then the pruned rows from the upsampled cache.
extern "C" nova_status nova_pruned_layer_forward(nova_ctx* ctx, const nova_block_weights* w,
                                                 const nova_block_modulation* mod, const nova_block_shape* s,
                                                 const void* x_in, const int32_t* keep_idx, const int32_t* prune_idx,
                                                 const int32_t* cu_keep, void* k_cache, void* v_cache, int32_t* kv_len,
                                                 int append_kv, const void* cache_prev, int hp, int wp, int h, int w_,
                                                 void* x_out, void* cache_out, int m_on_device, void* stream)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (!s) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_layer_forward: null shape");
    if (!shape_ok(s)) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_pruned_layer_forward: unsupported shape");
    if ((long)h * w_ != (long)s->N) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_layer_forward: h * w must equal N");
    if (!x_in || !x_out || !cu_keep) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_layer_forward: null tensor");
    if (x_out == x_in) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_layer_forward: x_out aliases x_in");
    if (!nova_aligned16(x_out) || !nova_aligned16(cache_out))
        return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_pruned_layer_forward: tensors must be 16-byte aligned");
    const long total = (long)s->B * s->N;
    if (total > 0x7fffffffL) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_pruned_layer_forward: too many rows");
    const bool on_dev = m_on_device != 0;
    if ((s->M < total || on_dev) && (!prune_idx || !cache_prev || hp < 1 || wp < 1))
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_layer_forward: pruned rows need prune_idx and cache_prev");
    if (total > 0 && !nova_aligned16(cache_prev))       // the restore would refuse it too, with half of the layer done
        return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_pruned_layer_forward: tensors must be 16-byte aligned");
    NOVA_DEVICE_GUARD(ctx, "nova_pruned_layer_forward");
    {   // debug mode: both lists are checked before the block's first kernel, so that a bad pruned list leaves no half-done layer
        const nova_status chk = nova_debug_check_lists(ctx, "nova_pruned_layer_forward", keep_idx, prune_idx, cu_keep,
                                                       s->B, s->N, s->M, !on_dev, (cudaStream_t)stream);
        if (chk != NOVA_OK) return chk;
    }
    const ScatterOut sc = {x_out, cache_out, prune_idx, cache_prev, hp, wp, h, w_};
    const nova_status rc = block_forward(ctx, w, mod, s, x_in, keep_idx, cu_keep, k_cache, v_cache, kv_len, append_kv, nullptr,
                                         stream, on_dev, &sc);
    if (rc != NOVA_OK || s->M > 0) return rc;
    // nothing kept: the block launched nothing
    return nova_restore_pruned_rows(ctx, x_in, prune_idx, cu_keep, cache_prev, hp, wp, h, w_, s->C, s->B, 0, on_dev,
                                    x_out, cache_out, stream, false);
}

// ---- block forward for callers that cannot allocate device memory --------------------------
// The scratch that nova_pruned_block_forward normally takes from the caller's workspace lives
// here, in a fixed array that is part of the library image: every GPU that loads the library
// holds these bytes until the process exits.
#define NOVA_STATIC_SCRATCH_BYTES (6u << 20)
static __device__ __align__(256) unsigned char g_static_scratch[NOVA_STATIC_SCRATCH_BYTES];

// Device address of g_static_scratch per CUDA device ordinal. In host code the array's name is
// only a handle for the runtime, not an address a kernel can use; the real address is looked up
// once per device with that device current.
static void* g_static_scratch_addr[64];

extern "C" size_t nova_static_scratch_bytes(void) { return NOVA_STATIC_SCRATCH_BYTES; }

extern "C" nova_status nova_pruned_block_forward_static(nova_ctx* ctx, const nova_block_weights* w,
                                                        const nova_block_shape* s, const void* x_in,
                                                        const int32_t* keep_idx, const int32_t* cu_keep,
                                                        void* k_cache, void* v_cache, int32_t* kv_len,
                                                        int append_kv, void* y_kept, void* stream)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (!s) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_block_forward_static: null shape");
    if (ctx->profiling)
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG,
                         "nova_pruned_block_forward_static: not available inside a profiling window (event creation may allocate)");
    if (!shape_ok(s)) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_pruned_block_forward_static: unsupported shape");
    if (s->M == 0) return NOVA_OK;      // nothing kept: a no-op, as for the ordinary entry point
    const size_t need = nova_block_workspace_bytes(s);
    if (need > NOVA_STATIC_SCRATCH_BYTES) {
        snprintf(ctx->err, sizeof(ctx->err),
                 "nova_pruned_block_forward_static: shape needs %zu bytes of scratch, the built-in array holds %u",
                 need, (unsigned)NOVA_STATIC_SCRATCH_BYTES);
        return NOVA_ERR_WORKSPACE;
    }
    int cur = -1;
    NOVA_CUDA_CHECK(ctx, cudaGetDevice(&cur));
    if (cur != ctx->device || cur < 0 || cur >= 64)
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG,
                         "nova_pruned_block_forward_static: the context's device must be the current device");
    if (!g_static_scratch_addr[cur]) {
        void* addr = nullptr;
        NOVA_CUDA_CHECK(ctx, cudaGetSymbolAddress(&addr, g_static_scratch));
        g_static_scratch_addr[cur] = addr;
    }
    // Run the ordinary path with the built-in array standing in for the caller's workspace.
    void* saved_ws = ctx->workspace;
    const size_t saved_bytes = ctx->workspace_bytes;
    ctx->workspace = g_static_scratch_addr[cur];
    ctx->workspace_bytes = NOVA_STATIC_SCRATCH_BYTES;
    const nova_status rc = nova_pruned_block_forward(ctx, w, s, x_in, keep_idx, cu_keep, k_cache, v_cache, kv_len,
                                                     append_kv, y_kept, stream);
    ctx->workspace = saved_ws;
    ctx->workspace_bytes = saved_bytes;
    return rc;
}
