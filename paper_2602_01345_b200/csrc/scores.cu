// Alternative per-token selection scores of the paper's selection-metric ablation (the table that
// compares entropy with an attention-based and an MSE-based criterion). Either score feeds the same
// nova_select_topk as the entropy does.
#include "tc_common.cuh"

namespace {

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ void unpack2(uint32_t w, float& lo, float& hi)
{
    lo = __uint_as_float(w << 16);
    hi = __uint_as_float(w & 0xffff0000u);
}

// ---- MSE score: mean over channels of (x - bilinear resize of the previous scale's map)^2 -----------
constexpr int kMseWarps = 8;

__global__ void __launch_bounds__(kMseWarps * 32)
score_mse_kernel(const uint4* x, const uint4* ref, int B, int hp, int wp, int h, int w,
                 int vec_per_row, float* __restrict__ score)
{
    const int lane = threadIdx.x & 31;
    const long r = (long)blockIdx.x * kMseWarps + (threadIdx.x >> 5);
    const int N = h * w;
    if (r >= (long)B * N) return;
    const int b = (int)(r / N), i = (int)(r - (long)b * N);
    const int oy = i / w, ox = i - oy * w;
    float sy = ((float)oy + 0.5f) * ((float)hp / (float)h) - 0.5f;
    float sx = ((float)ox + 0.5f) * ((float)wp / (float)w) - 0.5f;
    sy = fmaxf(sy, 0.f);
    sx = fmaxf(sx, 0.f);
    const int y0 = min((int)sy, hp - 1), x0 = min((int)sx, wp - 1);
    const int y1 = min(y0 + 1, hp - 1), x1 = min(x0 + 1, wp - 1);
    const float fy = sy - (float)y0, fx = sx - (float)x0;
    const float w00 = (1.f - fy) * (1.f - fx), w01 = (1.f - fy) * fx, w10 = fy * (1.f - fx), w11 = fy * fx;
    const uint4* c00 = ref + (((long)b * hp + y0) * wp + x0) * vec_per_row;
    const uint4* c01 = ref + (((long)b * hp + y0) * wp + x1) * vec_per_row;
    const uint4* c10 = ref + (((long)b * hp + y1) * wp + x0) * vec_per_row;
    const uint4* c11 = ref + (((long)b * hp + y1) * wp + x1) * vec_per_row;
    const uint4* xr = x + r * vec_per_row;
    float acc = 0.f;
    for (int v = lane; v < vec_per_row; v += 32) {
        const uint4 xv = xr[v], a = c00[v], bq = c01[v], c = c10[v], d = c11[v];
        const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
        const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {bq.x, bq.y, bq.z, bq.w};
        const uint32_t cw[4] = {c.x, c.y, c.z, c.w}, dw[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float xl, xh, al, ah, bl, bh, cl, ch, dl, dh;
            unpack2(xw[q], xl, xh);
            unpack2(aw[q], al, ah);
            unpack2(bw[q], bl, bh);
            unpack2(cw[q], cl, ch);
            unpack2(dw[q], dl, dh);
            const float d0 = xl - (w00 * al + w01 * bl + w10 * cl + w11 * dl);
            const float d1 = xh - (w00 * ah + w01 * bh + w10 * ch + w11 * dh);
            acc = fmaf(d0, d0, acc);
            acc = fmaf(d1, d1, acc);
        }
    }
    acc = warp_sum(acc);
    if (lane == 0) score[r] = acc / (float)(vec_per_row * 8);
}

// ---- attention mass ------------------------------------------------------------------------------
// Two passes over S = q K^T / sqrt(dh) per (image, head), both as 128 x 128 tiles on the tensor cores:
//   pass 1  rows: A = 128 queries, B = the key tiles (cache rows, then the scale's own keys);
//           lse[b, h, q] = log2-domain log-sum-exp of row q over all keys
//   pass 2  columns, transposed so that a thread's row is a key: A = 128 own keys, B = the query tiles of
//           one head after the other; score[key] = sum of 2^(s - lse) over queries and heads
// What bounds both is the special-function unit: one exponential per score, 16 per clock and SM, 44 us
// for the 201 M scores of two images of 1024 tokens, 30 heads and 1216 prior keys. The rest is arranged
// around keeping it busy: one thread per row of S reads its row from tensor memory 64 scores at a
// time, two warpgroups take the tiles in turn, each with its own S buffer (256 columns of tensor memory),
// and at head size 64 two CTAs share an SM. In small calls a row's work is spread over a cluster of 1 to 8 CTAs
// (pass 1: key tiles, pass 2: heads; the size that leaves the least of the last wave idle), whose
// partial results are merged through distributed shared memory in a fixed order; in large ones, where a quarter of the time
// went into starting and merging those and another into the last wave, the launch's tiles are divided evenly (attn_mass_ranges).
// Either way results are reproducible bit for bit. Both passes of that shape: 105 us in clusters, 87 in ranges, 1876
// with warp-level matrix fragments and the scores staged through shared memory.
constexpr int kAmThreads = 320;        // producer warp, MMA warp, two warpgroups of row threads
constexpr int kAmTile = 128;
constexpr int kAmSlab = 128 * 128;     // [128 rows][64 bf16]

template <int DH>
struct AmSmem {
    static constexpr int kTileBytes = (DH / 64) * kAmSlab;
    static constexpr int kStages = (DH == 64) ? 3 : 4;
    static constexpr int kAOff = 0;                                    // two A tiles
    static constexpr int kBOff = 2 * kTileBytes;
    static constexpr int kLseOff = kBOff + kStages * kTileBytes;       // [8 warps][2][128] fp32 (pass 2)
    static constexpr int kStatOff = kLseOff + 8 * 2 * kAmTile * 4;     // [2 in turn][2 warpgroups][128] float2
    static constexpr int kBarOff = kStatOff + 2 * 2 * kAmTile * 8;
    static constexpr int kTotal = kBarOff + 256 + 1024;
};

struct AmParams {
    const int32_t* kv_len;
    int N, Lmax, n_heads;
    float scale_log2e;
    int B;
    float* lse;
    float* score;
    float2* part;                // [CTA][first or last of its rows][128]
    unsigned int* tickets;       // one per CTA: of the row that starts in its range and does not end there
    unsigned int* status;
};

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
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
__device__ __forceinline__ float2 ld_dsmem2(uint32_t cluster_addr)
{
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(cluster_addr) : "memory");
    return v;
}

// State of one row of S across its tiles, and one tile: the thread's row of S from tensor memory, 64 scores at a time, then the
// buffer is released. Pass 1: `valid` columns count. Pass 2: neg_lse holds -lse of the tile's columns.
struct AmRow {
    float c, m2, l;              // score scale in the log2 domain; pass 1: running maximum (log2 domain) and sum
    uint64_t c2, acc[2];         // pass 2: sums
    __device__ __forceinline__ void reset()
    {
        m2 = -1e30f;
        l = 0.f;
        acc[0] = acc[1] = pack_f32x2(0.f, 0.f);
    }
    // what is left of the row: (maximum, sum), or (0, sum)
    template <int PASS>
    __device__ __forceinline__ float2 result() const
    {
        if (PASS == 1) return make_float2(m2, l);
        float s0, s1;
        unpack_f32x2(add_f32x2(acc[0], acc[1]), s0, s1);
        return make_float2(0.f, s0 + s1);
    }
};
template <int PASS>
__device__ __forceinline__ void am_tile(AmRow& s, uint32_t s_addr, uint64_t* s_empty, int lane, int valid, const float* neg_lse)
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t sv[64];
        tc::tmem_ld32(s_addr + h * 64, *reinterpret_cast<uint32_t(*)[32]>(&sv[0]));
        tc::tmem_ld32(s_addr + h * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&sv[32]));
        tc::tmem_ld_wait();
        if (h == 1) {            // the tile now lives in registers: the tensor core may have the buffer
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(s_empty);
        }
        if (PASS == 1) {
            if (valid < (h + 1) * 64) {
#pragma unroll
                for (int j = 0; j < 64; ++j)
                    if (h * 64 + j >= valid) sv[j] = 0xff800000u;        // -inf: past the last key of the tile
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int j = 0; j < 64; ++j) mx[j & 3] = fmaxf(mx[j & 3], __uint_as_float(sv[j]));
            const float t2 = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * s.c;
            const float m_new = fmaxf(s.m2, t2);
            const uint64_t nm2 = pack_f32x2(-m_new, -m_new);
            uint64_t part[2] = {pack_f32x2(0.f, 0.f), pack_f32x2(0.f, 0.f)};
#pragma unroll
            for (int j = 0; j < 64; j += 2) {
                float d0, d1;
                unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1])), s.c2, nm2), d0, d1);
                part[(j >> 1) & 1] = add_f32x2(part[(j >> 1) & 1], pack_f32x2(ex2(d0), ex2(d1)));
            }
            float s0, s1;
            unpack_f32x2(add_f32x2(part[0], part[1]), s0, s1);
            s.l = s.l * ex2(s.m2 - m_new) + (s0 + s1);
            s.m2 = m_new;
        } else {
            const ulonglong2* e2 = (const ulonglong2*)(neg_lse + h * 64);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const ulonglong2 e = e2[j];        // four -lse values, the same address in every lane
                float d0, d1, d2, d3;
                unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sv[4 * j]), __uint_as_float(sv[4 * j + 1])), s.c2, e.x), d0, d1);
                unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sv[4 * j + 2]), __uint_as_float(sv[4 * j + 3])), s.c2, e.y), d2, d3);
                s.acc[0] = add_f32x2(s.acc[0], pack_f32x2(ex2(d0), ex2(d1)));
                s.acc[1] = add_f32x2(s.acc[1], pack_f32x2(ex2(d2), ex2(d3)));
            }
        }
    }
}

// PASS 1: blockIdx.y = head, .z = image, cluster index along x = query tile.
// PASS 2: blockIdx.z = image, cluster index along x = key tile; the cluster's CTAs share the heads.
template <int DH, int PASS>
__global__ void __launch_bounds__(kAmThreads, DH == 64 ? 2 : 1)
attn_mass(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
          const __grid_constant__ CUtensorMap tmap_cache, const AmParams p, const int cs)
{
    using namespace tc;
    using L = AmSmem<DH>;
    constexpr int kStages = L::kStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* a_full = (uint64_t*)(smem + L::kBarOff);     // 2
    uint64_t* a_empty = a_full + 2;                        // 2
    uint64_t* b_full = a_empty + 2;                        // kStages
    uint64_t* b_empty = b_full + kStages;                  // kStages
    uint64_t* s_full = b_empty + kStages;                  // 2
    uint64_t* s_empty = s_full + 2;                        // 2, one arrival per warp of the warpgroup
    uint32_t* tmem_slot = (uint32_t*)(s_empty + 2);
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank();
    const int row_tile = blockIdx.x / cs, b = blockIdx.z;
    const int n_old = (PASS == 1 && p.kv_len) ? min(max(p.kv_len[b], 0), p.Lmax) : 0;
    const int tiles_own = (p.N + kAmTile - 1) / kAmTile, tiles_old = (n_old + kAmTile - 1) / kAmTile;
    // this CTA's work: groups (one A tile each) of `per_group` B tiles
    int group0 = 0, groups = 1, tile0 = 0, per_group = tiles_own;
    if (PASS == 1) {
        const int tiles = tiles_old + tiles_own;
        tile0 = rank * tiles / cs;
        per_group = (rank + 1) * tiles / cs - tile0;
        if (per_group == 0) groups = 0;
    } else {
        group0 = rank * p.n_heads / cs;
        groups = (rank + 1) * p.n_heads / cs - group0;
    }
    const int total = groups * per_group;

    if (threadIdx.x == 0) {
        abort_flag_s = 0;
        for (int i = 0; i < 2; ++i) {
            mbar_init(&a_full[i], 1);
            mbar_init(&a_empty[i], 1);
            mbar_init(&s_full[i], 1);
            mbar_init(&s_empty[i], 4);
        }
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&b_full[i], 1);
            mbar_init(&b_empty[i], 1);
        }
        fence_barrier_init();
        prefetch_tmap(&tmap_q);
        prefetch_tmap(&tmap_k);
        if (PASS == 1) prefetch_tmap(&tmap_cache);
    }
    if (warp == 1) tmem_alloc(tmem_slot, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (elect_one()) {
            bool ok = true;
            int i = 0, groups_issued = 0;
            for (int g = 0; g < groups && ok; ++g) {
                const int head = (PASS == 1) ? (int)blockIdx.y : group0 + g;
                if (g >= 2) ok = mbar_wait(&a_empty[g & 1], (uint32_t)((g >> 1) - 1) & 1u, abort_flag, p.status);
                if (!ok) break;
                mbar_arrive_expect_tx(&a_full[g & 1], L::kTileBytes);
                for (int sl = 0; sl < DH / 64; ++sl)
                    tma_load_3d(smem + L::kAOff + (g & 1) * L::kTileBytes + sl * kAmSlab, PASS == 1 ? &tmap_q : &tmap_k,
                                &a_full[g & 1], head * DH + sl * 64, row_tile * kAmTile, b);
                groups_issued = g + 1;
                for (int t = 0; t < per_group; ++t, ++i) {
                    const int st = i % kStages;
                    if (i >= kStages) ok = mbar_wait(&b_empty[st], (uint32_t)((i / kStages) - 1) & 1u, abort_flag, p.status);
                    if (!ok) break;
                    const CUtensorMap* map = PASS == 1 ? &tmap_k : &tmap_q;
                    int tile = tile0 + t;
                    if (PASS == 1) {
                        if (tile < tiles_old) map = &tmap_cache;
                        else tile -= tiles_old;
                    }
                    mbar_arrive_expect_tx(&b_full[st], L::kTileBytes);
                    for (int sl = 0; sl < DH / 64; ++sl)
                        tma_load_3d(smem + L::kBOff + st * L::kTileBytes + sl * kAmSlab, map, &b_full[st], head * DH + sl * 64,
                                    tile * kAmTile, b);
                }
            }
            if (*abort_flag) {       // let the copies in flight land before shared memory is released
                for (int g = max(0, groups_issued - 2); g < groups_issued; ++g) mbar_drain(&a_full[g & 1], (uint32_t)(g >> 1) & 1u);
                for (int j = max(0, i - kStages); j < i; ++j) mbar_drain(&b_full[j % kStages], (uint32_t)(j / kStages) & 1u);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            constexpr uint32_t idesc = idesc_bf16_f32(kAmTile, kAmTile, 0);
            const uint64_t a_desc = smem_desc_sw128(smem_u32(smem + L::kAOff), 16, 1024);
            const uint64_t b_desc = smem_desc_sw128(smem_u32(smem + L::kBOff), 16, 1024);
            bool ok = true;
            int i = 0;
            for (int g = 0; g < groups && ok; ++g) {
                ok = mbar_wait(&a_full[g & 1], (uint32_t)(g >> 1) & 1u, abort_flag, p.status);
                for (int t = 0; t < per_group && ok; ++t, ++i) {
                    const int st = i % kStages;
                    ok = mbar_wait(&b_full[st], (uint32_t)(i / kStages) & 1u, abort_flag, p.status);
                    if (ok && i >= 2) ok = mbar_wait(&s_empty[i & 1], (uint32_t)((i >> 1) - 1) & 1u, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t ad = a_desc + (uint32_t)((g & 1) * (L::kTileBytes >> 4));
                    const uint64_t bd = b_desc + (uint32_t)(st * (L::kTileBytes >> 4));
#pragma unroll
                    for (int kk = 0; kk < DH / 16; ++kk) {
                        const uint32_t off = (kk >> 2) * (kAmSlab >> 4) + (kk & 3) * 2;
                        mma_bf16_ss(tmem_base + 128u * (i & 1), ad + off, bd + off, idesc, kk ? 1u : 0u);
                    }
                    mma_commit(&s_full[i & 1]);
                    mma_commit(&b_empty[st]);
                }
                if (ok) mma_commit(&a_empty[g & 1]);
            }
        }
    } else {
        const int wg = (warp - 2) >> 2, q = warp & 3, row = q * 32 + lane;
        const uint32_t s_addr = tmem_base + ((uint32_t)(q * 32) << 16) + 128u * wg;
        float* lse_s = (float*)(smem + L::kLseOff) + (warp - 2) * 2 * kAmTile;
        AmRow s;
        s.c = p.scale_log2e;
        s.c2 = pack_f32x2(s.c, s.c);
        s.reset();
        for (int i = wg; i < total; i += 2) {
            int valid = kAmTile;
            if (PASS == 1) {
                const int tile = tile0 + i;
                valid = tile < tiles_old ? n_old - tile * kAmTile : p.N - (tile - tiles_old) * kAmTile;
            } else {
                // -lse of the tile's queries, a copy per warp (no barrier between warps); -inf past the last query
                const int g = i / per_group, q0 = (i - g * per_group) * kAmTile;
                const float* src = p.lse + ((long)b * p.n_heads + group0 + g) * p.N;
                float* dst = lse_s + ((i >> 1) & 1) * kAmTile;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int qi = q0 + j * 32 + lane;
                    dst[j * 32 + lane] = qi < p.N ? -src[qi] : -INFINITY;
                }
                __syncwarp();
            }
            if (!mbar_wait_warp(&s_full[wg], (uint32_t)(i >> 1) & 1u, abort_flag, p.status)) break;
            tc_fence_after();
            am_tile<PASS>(s, s_addr, &s_empty[wg], lane, valid, lse_s + ((i >> 1) & 1) * kAmTile);
        }
        float2 mine = s.result<PASS>();
        if (PASS == 2) mine = make_float2(mine.y, 0.f);
        ((float2*)(smem + L::kStatOff))[wg * kAmTile + row] = mine;
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();              // every CTA's partial results are in place
    if (rank == 0 && warp >= 2 && warp < 6) {
        // merged in the order (CTA 0: warpgroup 0, 1), (CTA 1: 0, 1), ...
        const int row = (warp & 3) * 32 + lane, i = row_tile * kAmTile + row;
        const uint32_t at = smem_u32(smem + L::kStatOff) + (uint32_t)row * 8u;
        float m = -1e30f, sum = 0.f;
        if (PASS == 1)
            for (int r = 0; r < cs; ++r)
                for (int w = 0; w < 2; ++w) m = fmaxf(m, ld_dsmem2(map_to_cta(at + w * kAmTile * 8, (uint32_t)r)).x);
        for (int r = 0; r < cs; ++r)
            for (int w = 0; w < 2; ++w) {
                const float2 v = ld_dsmem2(map_to_cta(at + w * kAmTile * 8, (uint32_t)r));
                sum += (PASS == 1) ? v.y * exp2f(v.x - m) : v.x;
            }
        if (i < p.N) {
            if (PASS == 1) p.lse[((long)b * p.n_heads + blockIdx.y) * p.N + i] = m + log2f(sum);
            else p.score[(long)b * p.N + i] = sum / ((float)p.n_heads * (float)p.N);
        }
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 256);
    }
    __syncwarp();
    cluster_sync_all();              // nobody's shared memory goes while it is read
}

// The same for launches in which a CTA gets many tiles: the launch's tiles, in the order of their rows, are divided evenly over as
// many CTAs as run at once. Rows that lie in the ranges of several CTAs are merged through memory by the CTA that finishes its part
// last, in the order of the CTAs: reproducible bit for bit.
// Where a CTA is in the launch's tiles. Pass 1: rows = (image, head, query tile), T = the image's key tiles. Pass 2: rows =
// (image, key tile), T = query tiles of all heads.
template <int PASS>
struct AmWalk {
    int b = 0, item, t, T;
    long row0;                   // first tile of the present row, counted over the launch
    __device__ __forceinline__ static int tiles_of(const AmParams& p) { return (p.N + kAmTile - 1) / kAmTile; }
    __device__ __forceinline__ static int old_keys(const AmParams& p, int b) { return PASS == 1 && p.kv_len ? min(max(p.kv_len[b], 0), p.Lmax) : 0; }
    __device__ __forceinline__ static int row_tiles(const AmParams& p, int b)
    {
        return PASS == 1 ? tiles_of(p) + (old_keys(p, b) + kAmTile - 1) / kAmTile : tiles_of(p) * p.n_heads;
    }
    // The launch's tiles, and the place of one of them; by whole warps, 32 images at a time (with one after the other a launch of 60000
    // images of 16 tokens took 11.2 ms, 3.0 of them for its tiles), or a few one after the other (two images: 0.7 us of a call of 106).
    static constexpr int kFewImages = 4;
    __device__ __forceinline__ long image_tiles(const AmParams& p, int b) const { return b < p.B ? (long)rows_of(p) * row_tiles(p, b) : 0; }
    __device__ __forceinline__ explicit AmWalk(const AmParams&) {}
    __device__ __forceinline__ static int rows_of(const AmParams& p) { return PASS == 1 ? tiles_of(p) * p.n_heads : tiles_of(p); }
    __device__ __forceinline__ long total(const AmParams& p) const
    {
        long n = 0;
        if (p.B <= kFewImages) {
            for (int i = 0; i < p.B; ++i) n += image_tiles(p, i);
            return n;
        }
        for (int b0 = threadIdx.x & 31; b0 < p.B; b0 += 32) n += image_tiles(p, b0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
        return n;
    }
    __device__ __forceinline__ void find(const AmParams& p, long at)
    {
        const int lane = threadIdx.x & 31;
        row0 = 0;
        if (p.B <= kFewImages) {
            for (; b < p.B - 1 && at >= row0 + image_tiles(p, b); ++b) row0 += image_tiles(p, b);
        } else for (int b0 = 0; b0 < p.B; b0 += 32) {
            const long mine = image_tiles(p, b0 + lane);
            long incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const uint32_t past = __ballot_sync(0xffffffffu, at < row0 + incl);
            if (past) {
                const int at_lane = __ffs(past) - 1;
                row0 += __shfl_sync(0xffffffffu, incl - mine, at_lane);
                b = b0 + at_lane;
                break;
            }
            row0 += __shfl_sync(0xffffffffu, incl, 31);
        }
        T = row_tiles(p, b);
        item = (int)((at - row0) / T);
        row0 += (long)item * T;
        t = (int)(at - row0);
    }
    __device__ __forceinline__ void next(const AmParams& p)
    {
        if (++t < T) return;
        t = 0;
        row0 += T;
        if (++item < rows_of(p)) return;
        item = 0;
        if (++b < p.B) T = row_tiles(p, b);
    }
    __device__ __forceinline__ int head(const AmParams& p) const { return PASS == 1 ? item / tiles_of(p) : t / tiles_of(p); }
    __device__ __forceinline__ int row_tile(const AmParams& p) const { return PASS == 1 ? item % tiles_of(p) : item; }
    // does this tile need another A tile than the one before?
    __device__ __forceinline__ bool new_a(const AmParams& p) const { return PASS == 1 ? t == 0 : t % tiles_of(p) == 0; }
};
__device__ __forceinline__ long am_start(long cta, long ctas, long total) { return cta * total / ctas; }
__device__ __forceinline__ int am_owner(long tile, long ctas, long total) { return (int)(((tile + 1) * ctas - 1) / total); }

template <int DH, int PASS>
__global__ void __launch_bounds__(kAmThreads, DH == 64 ? 2 : 1)
attn_mass_ranges(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
          const __grid_constant__ CUtensorMap tmap_cache, const AmParams p)
{
    using namespace tc;
    using L = AmSmem<DH>;
    using Walk = AmWalk<PASS>;
    constexpr int kStages = L::kStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* a_full = (uint64_t*)(smem + L::kBarOff);     // 2
    uint64_t* a_empty = a_full + 2;                        // 2
    uint64_t* b_full = a_empty + 2;                        // kStages
    uint64_t* b_empty = b_full + kStages;                  // kStages
    uint64_t* s_full = b_empty + kStages;                  // 2
    uint64_t* s_empty = s_full + 2;                        // 2, one arrival per warp of the warpgroup
    uint32_t* tmem_slot = (uint32_t*)(s_empty + 2);
    __shared__ int abort_flag_s, ticket_s;
    volatile int* abort_flag = &abort_flag_s;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        abort_flag_s = 0;
        for (int i = 0; i < 2; ++i) {
            mbar_init(&a_full[i], 1);
            mbar_init(&a_empty[i], 1);
            mbar_init(&s_full[i], 1);
            mbar_init(&s_empty[i], 4);
        }
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&b_full[i], 1);
            mbar_init(&b_empty[i], 1);
        }
        fence_barrier_init();
        prefetch_tmap(&tmap_q);
        prefetch_tmap(&tmap_k);
        if (PASS == 1) prefetch_tmap(&tmap_cache);
    }
    if (warp == 1) tmem_alloc(tmem_slot, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_launch_dependents();
    pdl_wait();
    Walk w(p);
    const long all = w.total(p), begin = am_start(blockIdx.x, gridDim.x, all);
    const int total = (int)(am_start(blockIdx.x + 1, gridDim.x, all) - begin);
    if (total > 0) w.find(p, begin);

    if (warp == 0) {
        if (elect_one() && total > 0) {
            bool ok = true;
            int i = 0, groups = 0;
            for (; i < total && ok; ++i, w.next(p)) {
                const int head = w.head(p);
                if (i == 0 || w.new_a(p)) {
                    const int g = groups & 1;
                    if (groups >= 2) ok = mbar_wait(&a_empty[g], (uint32_t)((groups >> 1) - 1) & 1u, abort_flag, p.status);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&a_full[g], L::kTileBytes);
                    for (int sl = 0; sl < DH / 64; ++sl)
                        tma_load_3d(smem + L::kAOff + g * L::kTileBytes + sl * kAmSlab, PASS == 1 ? &tmap_q : &tmap_k,
                                    &a_full[g], head * DH + sl * 64, w.row_tile(p) * kAmTile, w.b);
                    ++groups;
                }
                const int st = i % kStages;
                if (i >= kStages) ok = mbar_wait(&b_empty[st], (uint32_t)((i / kStages) - 1) & 1u, abort_flag, p.status);
                if (!ok) break;
                const CUtensorMap* map = PASS == 1 ? &tmap_k : &tmap_q;
                int tile = PASS == 1 ? w.t : w.t % Walk::tiles_of(p);
                if (PASS == 1) {
                    const int tiles_old = w.T - Walk::tiles_of(p);
                    if (tile < tiles_old) map = &tmap_cache;
                    else tile -= tiles_old;
                }
                mbar_arrive_expect_tx(&b_full[st], L::kTileBytes);
                for (int sl = 0; sl < DH / 64; ++sl)
                    tma_load_3d(smem + L::kBOff + st * L::kTileBytes + sl * kAmSlab, map, &b_full[st], head * DH + sl * 64,
                                tile * kAmTile, w.b);
            }
            if (*abort_flag) {       // let the copies in flight land before shared memory is released
                for (int g = max(0, groups - 2); g < groups; ++g) mbar_drain(&a_full[g & 1], (uint32_t)(g >> 1) & 1u);
                for (int j = max(0, i - kStages); j < i; ++j) mbar_drain(&b_full[j % kStages], (uint32_t)(j / kStages) & 1u);
            }
        }
    } else if (warp == 1) {
        if (elect_one() && total > 0) {
            constexpr uint32_t idesc = idesc_bf16_f32(kAmTile, kAmTile, 0);
            const uint64_t a_desc = smem_desc_sw128(smem_u32(smem + L::kAOff), 16, 1024);
            const uint64_t b_desc = smem_desc_sw128(smem_u32(smem + L::kBOff), 16, 1024);
            bool ok = true;
            int groups = 0;
            for (int i = 0; i < total && ok; ++i) {
                if (i == 0 || w.new_a(p)) {
                    ok = mbar_wait(&a_full[groups & 1], (uint32_t)(groups >> 1) & 1u, abort_flag, p.status);
                    ++groups;
                }
                const int g = (groups - 1) & 1, st = i % kStages;
                if (ok) ok = mbar_wait(&b_full[st], (uint32_t)(i / kStages) & 1u, abort_flag, p.status);
                if (ok && i >= 2) ok = mbar_wait(&s_empty[i & 1], (uint32_t)((i >> 1) - 1) & 1u, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                const uint64_t ad = a_desc + (uint32_t)(g * (L::kTileBytes >> 4));
                const uint64_t bd = b_desc + (uint32_t)(st * (L::kTileBytes >> 4));
#pragma unroll
                for (int kk = 0; kk < DH / 16; ++kk) {
                    const uint32_t off = (kk >> 2) * (kAmSlab >> 4) + (kk & 3) * 2;
                    mma_bf16_ss(tmem_base + 128u * (i & 1), ad + off, bd + off, idesc, kk ? 1u : 0u);
                }
                mma_commit(&s_full[i & 1]);
                mma_commit(&b_empty[st]);
                w.next(p);
                if (i + 1 < total && w.new_a(p)) mma_commit(&a_empty[g]);
            }
        }
    } else {
        const int wg = (warp - 2) >> 2, q = warp & 3, row = q * 32 + lane;
        const uint32_t s_addr = tmem_base + ((uint32_t)(q * 32) << 16) + 128u * wg;
        float* lse_s = (float*)(smem + L::kLseOff) + (warp - 2) * 2 * kAmTile;
        AmRow s;
        s.c = p.scale_log2e;
        s.c2 = pack_f32x2(s.c, s.c);
        s.reset();
        bool ok = true;                                // after a failed wait only the barriers are kept up: the status word says so
        int ends = 0;                                  // rows finished so far, by this CTA's part of them
        for (int i = 0; i < total; ++i) {
            if ((i & 1) == wg && ok) {
                int valid = kAmTile;
                if (PASS == 1) {
                    const int tiles_old = w.T - Walk::tiles_of(p);
                    valid = w.t < tiles_old ? Walk::old_keys(p, w.b) - w.t * kAmTile : p.N - (w.t - tiles_old) * kAmTile;
                } else {
                    // -lse of the tile's queries, a copy per warp (no barrier between warps); -inf past the last query
                    const int q0 = (w.t % Walk::tiles_of(p)) * kAmTile;
                    const float* src = p.lse + ((long)w.b * p.n_heads + w.head(p)) * p.N;
                    float* dst = lse_s + ((i >> 1) & 1) * kAmTile;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int qi = q0 + j * 32 + lane;
                        dst[j * 32 + lane] = qi < p.N ? -src[qi] : -INFINITY;
                    }
                    __syncwarp();
                }
                ok = mbar_wait_warp(&s_full[wg], (uint32_t)(i >> 1) & 1u, abort_flag, p.status);
                tc_fence_after();
                am_tile<PASS>(s, s_addr, &s_empty[wg], lane, valid, lse_s + ((i >> 1) & 1) * kAmTile);
            }
            if (w.t == w.T - 1 || i == total - 1) {
                // the end of this CTA's part of the row: warpgroup 1 hands its half to warpgroup 0
                float2* stat = (float2*)(smem + L::kStatOff) + (ends & 1) * 2 * kAmTile;
                const float2 mine = s.result<PASS>();
                s.reset();
                ++ends;
                if (wg == 1) stat[row] = mine;
                asm volatile("bar.sync 1, 256;" ::: "memory");
                if (wg == 0) {
                    auto merge = [](float2 x, float2 y) {
                        if (PASS == 2) return make_float2(0.f, x.y + y.y);
                        const float m = fmaxf(x.x, y.x);
                        return make_float2(m, x.y * exp2f(x.x - m) + y.y * exp2f(y.x - m));
                    };
                    float2 sum = merge(mine, stat[row]);
                    const int first = am_owner(w.row0, gridDim.x, all), last = am_owner(w.row0 + w.T - 1, gridDim.x, all);
                    bool write = true;
                    if (first != last) {
                        // a CTA's parts: of its first row, and of another that is its last
                        auto slot = [&](int of) {
                            return p.part + (of * 2 + (am_start(of, gridDim.x, all) < w.row0 ? 1 : 0)) * kAmTile + row;
                        };
                        __stcg(slot(blockIdx.x), sum);
                        __threadfence();
                        asm volatile("bar.sync 2, 128;" ::: "memory");
                        if (threadIdx.x == 64) {
                            const unsigned int drawn = atomicAdd(p.tickets + first, 1u);
                            if ((int)drawn == last - first) p.tickets[first] = 0;       // ready for the next launch
                            ticket_s = (int)drawn;
                            __threadfence();
                        }
                        asm volatile("bar.sync 2, 128;" ::: "memory");
                        write = ticket_s == last - first;                              // everybody else has published
                        if (write) {
                            sum = __ldcg(slot(first));
                            for (int of = first + 1; of <= last; ++of) sum = merge(sum, __ldcg(slot(of)));
                        }
                    }
                    const int at = w.row_tile(p) * kAmTile + row;
                    if (write && at < p.N) {
                        if (PASS == 1) p.lse[((long)w.b * p.n_heads + w.head(p)) * p.N + at] = sum.x + log2f(sum.y);
                        else p.score[(long)w.b * p.N + at] = sum.y / ((float)p.n_heads * (float)p.N);
                    }
                }
            }
            w.next(p);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 256);
    }
}

// Cluster size 1, 2, 4 or 8 for `items` rows of tiles of `steps` steps that can be split `ways` ways: the one
// with the shortest schedule, a CTA's start-up and merge counted as two steps.
int am_cluster(long items, long steps, int ways, int num_sms)
{
    int best = 1;
    long best_cost = 0;
    for (int cs = 1; cs <= 8 && cs <= ways; cs *= 2) {
        const long cost = ((items * cs + num_sms - 1) / num_sms) * ((steps + cs - 1) / cs + 2);
        if (cs == 1 || cost < best_cost) { best = cs; best_cost = cost; }
    }
    return best;
}

template <int DH>
nova_status launch_mass(nova_ctx* ctx, const void* q, const void* k, const void* k_cache, const int32_t* kv_len,
                        int B, int N, int C, int n_heads, int Lmax, float* lse, float* score, cudaStream_t st)
{
    using L = AmSmem<DH>;
    static bool attr_done[64];
    if (ctx->device >= 64 || !attr_done[ctx->device]) {
        NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(attn_mass<DH, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kTotal));
        NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(attn_mass<DH, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kTotal));
        NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(attn_mass_ranges<DH, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kTotal));
        NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(attn_mass_ranges<DH, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kTotal));
        if (ctx->device < 64) attr_done[ctx->device] = true;
    }
    CUtensorMap tq, tk, tcache;
    const uint64_t dn[3] = {(uint64_t)C, (uint64_t)N, (uint64_t)B}, sn[2] = {(uint64_t)C * 2, (uint64_t)N * C * 2};
    const bool cached = kv_len && Lmax > 0;
    const uint64_t dl[3] = {(uint64_t)C, (uint64_t)Lmax, (uint64_t)B}, sl[2] = {(uint64_t)C * 2, (uint64_t)Lmax * C * 2};
    if (!tc::make_tmap_bf16(ctx, &tq, q, 3, dn, sn, kAmTile) || !tc::make_tmap_bf16(ctx, &tk, k, 3, dn, sn, kAmTile) ||
        !(cached ? tc::make_tmap_bf16(ctx, &tcache, k_cache, 3, dl, sl, kAmTile) : tc::make_tmap_bf16(ctx, &tcache, k, 3, dn, sn, kAmTile)))
        return nova_fail(ctx, NOVA_ERR_CUDA, "nova_score_attention_mass: cuTensorMapEncodeTiled failed");
    AmParams p;
    p.kv_len = cached ? kv_len : nullptr; p.N = N; p.Lmax = Lmax; p.n_heads = n_heads;
    p.scale_log2e = (float)((1.0 / sqrt((double)DH)) * 1.4426950408889634);
    p.lse = lse; p.score = score; p.status = ctx->dev_status; p.B = B;
    p.tickets = ctx->dev_status + NOVA_STATUS_WORDS + NOVA_MEAN_MAX_SEGMENTS * 2;
    p.part = (float2*)(p.tickets + NOVA_TICKETS);
    const int tiles = (N + kAmTile - 1) / kAmTile;
    const int steps1 = tiles + (cached ? (Lmax + kAmTile - 1) / kAmTile : 0);
    // Ranges where a CTA gets at least so many tiles of the second pass; with fewer, merging rows through memory costs more
    // than clusters do. us, clusters -> ranges, at tiles per CTA; head size 64: 2.6 33 -> 40, 5.1 56 -> 51, 6.5 70 -> 61, 8.6 78 -> 65,
    // 13 104 -> 87, 27 180 -> 148; head size 128: 3.5 25 -> 31, 6.9 42 -> 44 and 46 -> 40, 13.8 78 -> 64, 73 287 -> 247.
    // At head size 64, where two CTAs share an SM and hide each other's start, clusters again with many rows of more than five key tiles:
    // 16 images of 1024 tokens, 13 rows per CTA, 542 -> 559, 32 such 1039 -> 1125; 12 such, 10 rows, 434 -> 424; 256 images of 100
    // tokens, 14 rows of three tiles, 139 -> 122. At 128 ranges throughout: 512 images of 256 tokens 1283 -> 905.
    const long slots = min((long)ctx->num_sms * (DH == 64 ? 2 : 1), (long)NOVA_TICKETS), tiles2 = (long)tiles * tiles * n_heads * B;
    const long rows1 = (long)tiles * n_heads * B;
    if (tiles2 >= (DH == 64 ? 5 : 8) * slots && (DH == 128 || rows1 <= 10 * slots || steps1 <= 5)) {
        {
            nova_launch_scope scope(ctx, NOVA_K_SCORE, st);
            NOVA_CUDA_CHECK(ctx, nova_launch_pdl(attn_mass_ranges<DH, 1>, dim3((unsigned)slots), dim3(kAmThreads), L::kTotal, st, 0, tq, tk, tcache, p));
        }
        nova_launch_scope scope(ctx, NOVA_K_SCORE, st);
        NOVA_CUDA_CHECK(ctx, nova_launch_pdl(attn_mass_ranges<DH, 2>, dim3((unsigned)slots), dim3(kAmThreads), L::kTotal, st, 0, tq, tk, tcache, p));
        return NOVA_OK;
    }
    const int cs1 = am_cluster((long)tiles * n_heads * B, steps1, steps1, ctx->num_sms);
    const int cs2 = am_cluster((long)tiles * B, (long)n_heads * tiles, n_heads, ctx->num_sms);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(kAmThreads); cfg.dynamicSmemBytes = L::kTotal; cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 1;
    {
        nova_launch_scope scope(ctx, NOVA_K_SCORE, st);
        attr[0].val.clusterDim.x = cs1;
        cfg.gridDim = dim3(tiles * cs1, n_heads, B);
        NOVA_CUDA_CHECK(ctx, cudaLaunchKernelEx(&cfg, attn_mass<DH, 1>, tq, tk, tcache, p, (int)cs1));
    }
    {
        nova_launch_scope scope(ctx, NOVA_K_SCORE, st);
        attr[0].val.clusterDim.x = cs2;
        cfg.gridDim = dim3(tiles * cs2, 1, B);
        NOVA_CUDA_CHECK(ctx, cudaLaunchKernelEx(&cfg, attn_mass<DH, 2>, tq, tk, tcache, p, (int)cs2));
    }
    NOVA_CUDA_CHECK(ctx, cudaGetLastError());
    return NOVA_OK;
}

}  // namespace

extern "C" nova_status nova_score_mse(nova_ctx* ctx, const void* x, const void* ref_prev, int B, int hp, int wp,
                                      int h, int w, int C, float* score, void* stream)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (B < 0 || h < 0 || w < 0 || C < 1) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_score_mse: bad sizes");
    const long total = (long)B * h * w;
    if (total == 0) return NOVA_OK;
    if (total > 0x7fffffffL) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_score_mse: too many tokens");
    if (C % 8) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_score_mse: C must be a multiple of 8");
    if (!x || !ref_prev || !score || hp < 1 || wp < 1) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_score_mse: null pointer or empty reference map");
    if (!nova_aligned16(x) || !nova_aligned16(ref_prev)) return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_score_mse: tensors must be 16-byte aligned");
    NOVA_DEVICE_GUARD(ctx, "nova_score_mse");
    const unsigned blocks = (unsigned)((total + kMseWarps - 1) / kMseWarps);
    nova_launch_scope scope(ctx, NOVA_K_SCORE, (cudaStream_t)stream);
    score_mse_kernel<<<blocks, kMseWarps * 32, 0, (cudaStream_t)stream>>>((const uint4*)x, (const uint4*)ref_prev, B, hp, wp, h, w,
                                                                         C / 8, score);
    NOVA_CUDA_CHECK(ctx, cudaGetLastError());
    return NOVA_OK;
}

extern "C" nova_status nova_score_attention_mass(nova_ctx* ctx, const void* q, const void* k, const void* k_cache,
                                                 const int32_t* kv_len, int B, int N, int C, int n_heads, int Lmax,
                                                 float* lse_scratch, float* score, void* stream)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (B < 0 || N < 0 || C < 1 || n_heads < 1 || Lmax < 0) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_score_attention_mass: bad sizes");
    if ((long)B * N == 0) return NOVA_OK;
    if (C % n_heads || (C / n_heads != 64 && C / n_heads != 128))
        return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_score_attention_mass: head size must be 64 or 128");
    if (B > 65535 || n_heads > 65535) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_score_attention_mass: too many images or heads");
    if (!q || !k || !score || !lse_scratch || (kv_len && !k_cache))
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_score_attention_mass: null pointer");
    if (!nova_aligned16(q) || !nova_aligned16(k) || !nova_aligned16(k_cache))
        return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_score_attention_mass: tensors must be 16-byte aligned");
    NOVA_DEVICE_GUARD(ctx, "nova_score_attention_mass");
    cudaStream_t st = (cudaStream_t)stream;
    if (C / n_heads == 64) return launch_mass<64>(ctx, q, k, k_cache, kv_len, B, N, C, n_heads, Lmax, lse_scratch, score, st);
    return launch_mass<128>(ctx, q, k, k_cache, kv_len, B, N, C, n_heads, Lmax, lse_scratch, score, st);
}
