// out[M, N] = epilogue(A[M, K] * W[N, K]^T + bias) on the sm_100a tensor cores.
//
// Both operands are K-major bf16, so one TMA box of 64 K-elements (128 bytes, 128-byte swizzle) per row
// feeds tcgen05.mma directly. Two kernels, both of CTA pairs (tcgen05 cta_group::2: per instruction each
// CTA supplies only half of the operand rows, which halves the shared-memory and L2 traffic per flop)
// with the same warp roles:
//   warp 0      TMA producer: fills a ring of {A tile, W tile} stages
//   warp 1      allocates TMEM, issues tcgen05.mma (one elected thread of the leader CTA), commits to mbarriers
//   warps 2-9   epilogue: the fp32 accumulator from tensor memory, bias, GELU / residual / QKV routing, bf16
// gemm_bf16_tn_pair takes the larger problems: a persistent grid
// whose accumulator is double buffered in tensor memory, so that the epilogue of tile i overlaps the main
// loop of tile i+1, with two epilogue warps per tensor-memory lane quarter (alternate column chunks), which
// keep the epilogue shorter than the main loop even with GELU. gemm_bf16_split takes the smaller ones.
// Every mbarrier wait is bounded; on expiry the CTA records a timeout and tears down.
#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int BK = 64;

__device__ __forceinline__ float gelu_tanh(float x)
{
    // 0.5 x (1 + tanh(c (x + 0.044715 x^3))) with the hardware tanh (relative error 2^-11, an order
    // of magnitude below the bf16 rounding of the result): six instructions per element. The FC1
    // epilogue is bound by its instruction count, not by memory.
    const float c = 0.7978845608028654f;
    const float inner = x * fmaf(x * x, 0.044715f * c, c);
    float t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(inner));
    const float hx = 0.5f * x;
    return fmaf(hx, t, hx);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&t);
}

struct GemmParams {
    const __nv_bfloat16* bias;
    int M, N, K;
    __nv_bfloat16* out;
    const __nv_bfloat16* res;
    const int32_t* res_row;
    int C;
    __nv_bfloat16* k_cache;
    __nv_bfloat16* v_cache;
    const int32_t* kv_row;
    unsigned int* status;
    const int32_t* adv_cu_keep;
    int32_t* adv_kv_len;
    int adv_B, adv_Lmax;
    float* ent;
    float* head_part;
    unsigned int* head_tickets;
    const int32_t* m_dev;
    const __nv_bfloat16* gate;
    const int32_t* img_row;
    const int32_t* out_row;
    const __nv_bfloat16* diff_in;
    __nv_bfloat16* diff_out;
    int early_trigger, count_settled;
};

// Rows of this launch: p.M, or the device-side count when the host only knows an upper bound.
__device__ __forceinline__ int true_rows(const GemmParams& p)
{
    return p.m_dev ? min(max(*p.m_dev, 0), p.M) : p.M;
}

// Is the row count known before the wait? A device-side count is an earlier launch's, of one that has ended already if count_settled says so.
__device__ __forceinline__ bool count_known(const GemmParams& p) { return !p.m_dev || p.count_settled; }
// The end of the kernel, of the two that are launched with a device-side count, that the problem does not belong to. One CTA
// waits, so that the launch ends after the one before it; the others make room for the next launch at once. With all of
// them waiting, and the count read only then, the last 64x64 scale in a graph, three such launches in each of 32 layers, takes
// 6786 us instead of 6722.
__device__ __forceinline__ void leave_to_other(const GemmParams& p)
{
    pdl_launch_dependents();
    if (blockIdx.x == 0) pdl_wait();
}

// Advance of the K/V cache lengths, done by one warp-sized loop of the launch's first CTA.
__device__ __forceinline__ void advance_kv_len(const GemmParams& p)
{
    if (!p.adv_kv_len) return;
    for (int b = threadIdx.x; b < p.adv_B; b += blockDim.x) {
        const int k_b = p.adv_cu_keep[b + 1] - p.adv_cu_keep[b];
        if (p.adv_kv_len[b] + k_b <= p.adv_Lmax) p.adv_kv_len[b] += k_b;
    }
}


// ---- epilogue: four consecutive features of eight rows per lane ---------------------------------------
// Both kernels turn their accumulators round in shared memory so that the lanes of a warp hold
// consecutive features of a few rows: every access to global memory then covers whole sectors of one
// row, where the tensor-memory layout (one row per thread) would touch 32 rows with every instruction.
// The eight rows of a lane are worked on together, without a branch between them: one after the other,
// each row's chain of dependent instructions cost a warp about 400 clocks, and the epilogue of a 256 x 256
// tile 8.4 us; so it takes 4.0, and a launch of 4096 x 2048 x 2048 27 us instead of 35.
__device__ __forceinline__ void unpack_bf16x4(uint2 w, float (&v)[4])
{
    v[0] = __uint_as_float(w.x << 16);
    v[1] = __uint_as_float(w.x & 0xffff0000u);
    v[2] = __uint_as_float(w.y << 16);
    v[3] = __uint_as_float(w.y & 0xffff0000u);
}

// Rows row0 + STEP * i: where each reads its residual (in) and writes (out; -1: nothing to write).
template <int EPI>
struct EpiRows {
    int in[8], out[8];
    int img;        // image of all eight (rows are sorted by image), or -1 if there are several (only looked up with a gate)
    // rows past the last one (row_end) stand in for it when reading and are not written
    template <int STEP>
    __device__ __forceinline__ void load(const GemmParams& p, int row0, int row_end)
    {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = min(row0 + STEP * i, row_end - 1);
            in[i] = out[i] = row;
            if (EPI == NOVA_EPI_BIAS_RES) {
                if (p.res_row) in[i] = p.res_row[row];
                if (p.out_row) out[i] = p.out_row[row];
            }
            if (EPI == NOVA_EPI_QKV) out[i] = p.kv_row[row];      // -1: cache overflow, flagged when the row map was built
        }
        if (EPI == NOVA_EPI_BIAS_RES && p.gate) {
            img = p.img_row[min(row0, row_end - 1)];
            if (p.img_row[min(row0 + STEP * 7, row_end - 1)] != img) img = -1;
        }
    }
};
// What the epilogue reads of four features of those rows, fetched before the accumulator is ready. DIFF: with a second output
// (if there is none all the same, diff_out says so).
template <int EPI, bool DIFF>
struct EpiData {
    uint2 res[8], diff[8], gate;
    __device__ __forceinline__ void fetch(const GemmParams& p, const EpiRows<EPI>& r, int col)
    {
        if (EPI != NOVA_EPI_BIAS_RES) return;
#pragma unroll
        for (int i = 0; i < 8; ++i) res[i] = *(const uint2*)(p.res + (long)r.in[i] * p.N + col);
        if (DIFF && p.diff_out) {
#pragma unroll
            for (int i = 0; i < 8; ++i) diff[i] = *(const uint2*)(p.diff_in + (long)r.out[i] * p.N + col);
        }
        if (p.gate && r.img >= 0) gate = *(const uint2*)(p.gate + (long)r.img * p.N + col);
    }
};
// v = accumulators; + bias, then GELU / residual / QKV routing, rounded to bf16. Features col .. col + 3 of
// rows row0 + STEP * (FROM + i) < row_end, four of the eight at a time (registers).
template <int EPI, int STEP, int FROM, bool DIFF>
__device__ __forceinline__ void epi_store(const GemmParams& p, int row0, int row_end, const EpiRows<EPI>& r, int col, uint2 bias,
                                          const EpiData<EPI, DIFF>& d, float (&v)[4][4])
{
    float t[4];
    unpack_bf16x4(bias, t);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) v[i][j] += t[j];
    uint2 y[4];
    if (EPI == NOVA_EPI_BIAS_GELU) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) v[i][j] = gelu_tanh(v[i][j]);
    }
    if (EPI == NOVA_EPI_BIAS_RES) {
        if (p.gate) {
            // per-image gate of the branch: out = residual + gate * (acc + bias)
            uint2 g[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) g[i] = d.gate;
            if (r.img < 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    g[i] = *(const uint2*)(p.gate + (long)p.img_row[min(row0 + STEP * (FROM + i), row_end - 1)] * p.N + col);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                unpack_bf16x4(g[i], t);
#pragma unroll
                for (int j = 0; j < 4; ++j) v[i][j] *= t[j];
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            unpack_bf16x4(d.res[FROM + i], t);
#pragma unroll
            for (int j = 0; j < 4; ++j) v[i][j] += t[j];
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) y[i] = make_uint2(pack_bf16(v[i][0], v[i][1]), pack_bf16(v[i][2], v[i][3]));
    if (EPI == NOVA_EPI_QKV) {
        const int which = col / p.C, cc = col - which * p.C;      // C % 4 == 0: the four lie in one of q, k, v
        __nv_bfloat16* base = (which == 0 ? p.out : which == 1 ? p.k_cache : p.v_cache) + cc;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = row0 + STEP * (FROM + i), dst = which == 0 ? row : r.out[FROM + i];
            if (row < row_end && dst >= 0) *(uint2*)(base + (long)dst * p.C) = y[i];
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (row0 + STEP * (FROM + i) < row_end) *(uint2*)(p.out + (long)r.out[FROM + i] * p.N + col) = y[i];
    if (EPI == NOVA_EPI_BIAS_RES && DIFF && p.diff_out) {
        // second output: the stored (bf16-rounded) value minus diff_in's row, i.e. what a separate pass over
        // the stored output would compute
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float s[4];
            unpack_bf16x4(d.diff[FROM + i], t);
            unpack_bf16x4(y[i], s);
            if (row0 + STEP * (FROM + i) < row_end)
                *(uint2*)(p.diff_out + (long)r.out[FROM + i] * p.N + col) =
                    make_uint2(pack_bf16(s[0] - t[0], s[1] - t[1]), pack_bf16(s[2] - t[2], s[3] - t[3]));
        }
    }
}

GemmParams make_params(nova_ctx* ctx, const nova_gemm_args& a)
{
    GemmParams p;
    p.bias = a.bias; p.M = a.M; p.N = a.N; p.K = a.K; p.out = a.out;
    p.res = a.res; p.res_row = a.res_row; p.C = a.C; p.k_cache = a.k_cache; p.v_cache = a.v_cache;
    p.kv_row = a.kv_row; p.status = ctx->dev_status;
    p.adv_cu_keep = a.adv_cu_keep; p.adv_kv_len = a.adv_kv_len; p.adv_B = a.adv_B; p.adv_Lmax = a.adv_Lmax;
    p.head_tickets = ctx->dev_status + NOVA_STATUS_WORDS + NOVA_MEAN_MAX_SEGMENTS * 2;
    p.head_part = (float*)(p.head_tickets + NOVA_TICKETS);
    p.ent = a.ent; p.m_dev = a.m_dev; p.gate = a.gate; p.img_row = a.img_row;
    p.out_row = a.out_row; p.diff_in = a.diff_in; p.diff_out = a.diff_out; p.early_trigger = a.early_trigger;
    p.count_settled = a.count_settled;
    return p;
}

// ---- which of the two kernels, and how ---------------------------------------------------------------
// Clusters of 2 and of 4 CTAs that the plan counts on running at the same time. They follow from the SM count and not
// from what the driver says fits: that depends on how the SMs left on a chip are spread over its eight GPCs, and with it
// would the plan, the order of the sums and the last bits of the results. Clusters of 4 are taken to lose two SMs in every
// GPC: 33 on 148 SMs, which is also what the driver said there. On a chip that holds fewer, a few tiles
// would run after the others; no cluster waits for another.
struct SplitCaps {
    int c[2];
};
inline SplitCaps split_caps(int num_sms)
{
    SplitCaps caps = {{num_sms / 2, num_sms > 20 ? (num_sms - 16) / 4 : 1}};
    return caps;
}
struct SplitPlan {
    int ls, nt;      // s = 1 << ls
    bool takes;      // false: the problem is the pair kernel's
};
// The plan follows from the true M, N, K and the SM count alone, on the host and in the kernel alike, so that a launch
// whose row count only the device knows adds in the same order as one whose row count the host knows.
// For each s, nt is the smallest token tile with which all tiles run at once; the cheaper s by estimated
// clocks wins. The constants are fits to launches of 8 to 1600 tokens, 1024 to 8192 features and K from 1024
// to 8192: a k-block takes its tensor time (2 nt clocks) or the 305 clocks at which a full ring of loads
// comes in, exchange and epilogue take 40 clocks a token. A four-way split was within 3 % of the two-way
// one or slower everywhere but at 256 x 1024 x 4096 (10.8 against 11.8 us).
// Where K need not be split and the token tile would be wider than 192, and where one round of tiles is not
// enough, the persistent kernel is the faster one (2250 x 1920 x 7680: 43.3 us against 46.3; with tiles
// of 192 at 1600 x 2048 x 8192 it is 45.3 against 39.0).
__host__ __device__ inline SplitPlan split_plan(int M, int N, int num_kb, const SplitCaps& caps)
{
    const int tiles_n = (N + 255) / 256;
    SplitPlan best = {0, 256, false};
    int best_cost = 0;
    for (int ls = 0; ls < 2 && (1 << ls) <= num_kb; ++ls) {
        const int tiles_t = caps.c[ls] / tiles_n;
        if (tiles_t < 1) continue;
        const int nt = ((M + tiles_t - 1) / tiles_t + 31) & ~31;
        if (nt > (ls ? 256 : 192)) continue;
        const int per_kb = 2 * nt > 305 ? 2 * nt : 305;
        const int cost = ((num_kb + (1 << ls) - 1) >> ls) * per_kb + 40 * nt;
        if (!best.takes || cost < best_cost) { best.ls = ls; best.nt = nt; best.takes = true; best_cost = cost; }
    }
    return best;
}

// ---- CTA-pair kernel ------------------------------------------------------------------------
constexpr int kPairBM = 256;           // rows of one pair tile (128 per CTA)
constexpr int kPairThreads = 320;      // producer warp, MMA warp, eight epilogue warps

template <int BN, int STAGES>
struct PairSmem {
    static constexpr int kABytes = 128 * BK * 2;           // this CTA's 128 rows of A
    static constexpr int kBBytes = (BN / 2) * BK * 2;      // this CTA's half of the W rows
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kTurnOff = STAGES * kStageBytes;  // per epilogue warp: 32 rows x 32 fp32, for the turn-round
    static constexpr int kBarOff = kTurnOff + 8 * 4096;
    static constexpr int kTotal = kBarOff + 256 + 1024 /*alignment slack*/;
};

// Work list of one launch: entries [0, tiles_full) are whole 256 x BN tiles in column-major tile
// order; the tiles after those, which would otherwise leave most pairs idle in a last partial wave,
// are each split into two 256 x BN/2 halves (entries tiles_full, tiles_full + 1, ...).
struct PairTile {
    int m0;     // first row of the pair tile
    int n0;     // first column
    int bn;     // columns: BN or BN / 2
};
// `span` > 0: tile index = m_tile + tiles_m * n_tile with span = tiles_m (tiles that run at the same
// time share few W rows and sweep all of A); span < 0: index = n_tile + tiles_n * m_tile with
// -span = tiles_n (they sweep all of W and share few A rows). The launcher picks the order whose
// swept operand is the smaller one, so that the larger one is fetched from HBM only once.
template <int BN>
__device__ __forceinline__ PairTile decode_tile(int entry, int span, int tiles_full)
{
    PairTile t;
    int whole = entry, half = -1;
    if (entry >= tiles_full) {
        const int h = entry - tiles_full;
        whole = tiles_full + (h >> 1);
        half = h & 1;
    }
    const int mt = span > 0 ? whole % span : whole / (-span);
    const int nt = span > 0 ? whole / span : whole % (-span);
    t.m0 = mt * kPairBM;
    t.n0 = nt * BN + (half > 0 ? BN / 2 : 0);
    t.bn = half >= 0 ? BN / 2 : BN;
    return t;
}

// Entry of the work list that pair `pair` handles as its `local`-th tile, or -1 past the end.
// group == 0: entries pair, pair + num_pairs, ... (any tile to any pair). Otherwise (entropy epilogue, |group| = tiles along N,
// N-fastest order) the epilogue threads carry a row's softmax state along its row block, and a pair takes
//   group > 0  whole row blocks, all their column tiles in turn;
//   group < 0  as many consecutive tiles as any other, or one less. A row block that lies in the ranges of several pairs is
//              merged by the one that finishes its part last (EntropyState::publish).
// Ranges where they take at most five sixths of the rounds: 16384 rows of 2048 against 4096 codes, 64 blocks on 74 pairs, take
// 178 us as whole blocks, in 16 rounds in which all pairs read the same column tile, and 188 us as ranges of 14 tiles.
// Fewer rows, us as whole blocks -> as ranges: 130 rows 150 -> 24, 4096 151 -> 54, 8192 152 -> 85, 12288 155 -> 129.
__device__ __forceinline__ int range_start(int pair, int num_pairs, int num_tiles) { return (int)((long)pair * num_tiles / num_pairs); }
__device__ __forceinline__ int range_owner(int tile, int num_pairs, int num_tiles)
{
    return (int)(((long)(tile + 1) * num_pairs - 1) / num_tiles);
}
__device__ __forceinline__ int pair_entry(int local, int pair, int num_pairs, int num_tiles, int group)
{
    if (group < 0) {
        const int e = range_start(pair, num_pairs, num_tiles) + local;
        return e < range_start(pair + 1, num_pairs, num_tiles) ? e : -1;
    }
    const int e = group == 0 ? pair + local * num_pairs : (pair + (local / group) * num_pairs) * group + local % group;
    return e < num_tiles ? e : -1;
}

// ---- entropy epilogue: running softmax-entropy state of one output row ----------------------
// m = reference maximum, s = sum e^{z-m}, u = sum (z-m) e^{z-m} in the log2 domain (m2 = m log2 e),
// the sums as two partial sums per 64-bit register (packed fp32 arithmetic).
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
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct EntropyState {
    float m, m2;
    uint64_t s2, u2;
    __device__ __forceinline__ void reset()
    {
        m = -INFINITY; m2 = -INFINITY;
        s2 = pack_f32x2(0.f, 0.f);
        u2 = s2;
    }
    // Sums after a rise of their reference by -shift (log2 domain), f = 2^shift. A rise that leaves nothing of them leaves nothing of
    // infinite ones either: below -1.5e9, where masks lie, the rounding of m2 is itself an exponent that can overflow.
    // (A NaN stays one.)
    static __device__ __forceinline__ void rescale(float& s, float& u, float shift, float f)
    {
        const bool gone = f == 0.f;
        u = gone && u == u ? 0.f : (u + shift * s) * f;
        s = gone && s == s ? 0.f : s * f;
    }
    // 32 more logits of the row (fp32 accumulators plus bias)
    __device__ __forceinline__ void add_chunk(const uint32_t (&acc)[32], const __nv_bfloat16* bias)
    {
        constexpr float kLog2e = 1.4426950408889634f;
        float z[32];
        if (bias) {
            const uint4* bias4 = (const uint4*)bias;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4 b = bias4[i];
                const uint32_t bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    z[i * 8 + j * 2] = __uint_as_float(acc[i * 8 + j * 2]) + __uint_as_float(bw[j] << 16);
                    z[i * 8 + j * 2 + 1] = __uint_as_float(acc[i * 8 + j * 2 + 1]) + __uint_as_float(bw[j] & 0xffff0000u);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) z[i] = __uint_as_float(acc[i]);
        }
        float cm = z[0];
#pragma unroll
        for (int i = 1; i < 32; ++i) cm = fmaxf(cm, z[i]);
        if (cm > m) {
            // raise the reference: both sums scale by f = e^{m - m'}, u also shifts by (m - m') s
            const float shift = (m - cm) * kLog2e;          // -inf the first time: f = 0
            const float f = ex2_approx(shift);
            float s_lo, s_hi, u_lo, u_hi;
            unpack_f32x2(s2, s_lo, s_hi);
            unpack_f32x2(u2, u_lo, u_hi);
            rescale(s_lo, u_lo, shift, f);
            rescale(s_hi, u_hi, shift, f);
            s2 = pack_f32x2(s_lo, s_hi);
            u2 = pack_f32x2(u_lo, u_hi);
            m = cm;
            m2 = cm * kLog2e;
        }
        const uint64_t log2e2 = pack_f32x2(kLog2e, kLog2e), neg_m2 = pack_f32x2(-m2, -m2);
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
            const uint64_t d2 = fma_f32x2(pack_f32x2(z[i], z[i + 1]), log2e2, neg_m2);
            float d0, d1;
            unpack_f32x2(d2, d0, d1);
            const uint64_t e2 = pack_f32x2(ex2_approx(d0), ex2_approx(d1));
            s2 = add_f32x2(s2, e2);
            u2 = fma_f32x2(d2, e2, u2);
        }
    }
    // A part of a row, for the pair that merges: slot of [m, s, u][256 rows] at the row.
    __device__ __forceinline__ void publish(float* slot) const
    {
        float s_lo, s_hi, u_lo, u_hi;
        unpack_f32x2(s2, s_lo, s_hi);
        unpack_f32x2(u2, u_lo, u_hi);
        __stcg(slot, m);
        __stcg(slot + 256, s_lo + s_hi);
        __stcg(slot + 512, u_lo + u_hi);
    }
    // One more part. (A part without a finite maximum is not finite itself, and stays so in the result.)
    __device__ __forceinline__ void merge(const float* slot, bool first)
    {
        constexpr float kLog2e = 1.4426950408889634f;
        const float m_p = __ldcg(slot);
        float s_p = __ldcg(slot + 256), u_p = __ldcg(slot + 512);
        if (first) {
            m = m_p;
            s2 = pack_f32x2(s_p, 0.f);
            u2 = pack_f32x2(u_p, 0.f);
            return;
        }
        float s, u, zero;
        unpack_f32x2(s2, s, zero);
        unpack_f32x2(u2, u, zero);
        const float top = fmaxf(m, m_p), d = (m - top) * kLog2e, d_p = (m_p - top) * kLog2e;
        rescale(s, u, d, ex2_approx(d));
        rescale(s_p, u_p, d_p, ex2_approx(d_p));
        s += s_p;
        u += u_p;
        m = top;
        s2 = pack_f32x2(s, 0.f);
        u2 = pack_f32x2(u, 0.f);
    }
    // H = ln s - u/s (u in log2 units); non-finite inputs give NaN and flag the status word
    __device__ __forceinline__ float finish(unsigned int* status) const
    {
        float s_lo, s_hi, u_lo, u_hi;
        unpack_f32x2(s2, s_lo, s_hi);
        unpack_f32x2(u2, u_lo, u_hi);
        const float s = s_lo + s_hi, u = u_lo + u_hi;
        float h = logf(s) - (u / s) * 0.6931471805599453f;
        if (!(fabsf(m) < INFINITY) || !(fabsf(h) < INFINITY)) {
            h = __int_as_float(0x7fc00000);
            atomicOr(status, NOVA_DEV_NONFINITE);
        } else if (h <= 0.f) {
            h = 0.f;
        }
        return h;
    }
};

// Barriers (all in each CTA's shared memory at equal offsets):
//   full[s]       leader's copy is used: one arrival (its own expect_tx) + the bytes of both CTAs
//   empty[s]      each CTA's copy, signalled in both CTAs by the leader's tcgen05.commit
//   acc_full[a]   each CTA's copy, same; a = accumulator buffer of tile parity
//   acc_empty[a]  leader's copy: one arrival per epilogue warp of both CTAs (16)
// DIFF: the residual epilogue with a second output. Without one there are registers to fetch two chunks ahead.
template <int BN, int STAGES, int EPI, bool DIFF>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
gemm_bf16_tn_pair(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                  const __grid_constant__ CUtensorMap tmap_w_half, const GemmParams p, const int span_host,
                  const int tiles_full_host, const int num_tiles_host, const int group, const SplitCaps caps)
{
    using L = PairSmem<BN, STAGES>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full_bar = (uint64_t*)(smem + L::kBarOff);
    uint64_t* empty_bar = full_bar + STAGES;
    uint64_t* acc_full = empty_bar + STAGES;     // 2
    uint64_t* acc_empty = acc_full + 2;          // 2
    uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();     // 0 = leader
    const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
    if (!count_known(p)) pdl_wait();
    if (EPI != NOVA_EPI_ENTROPY && p.m_dev && split_plan(true_rows(p), p.N, p.K / BK, caps).takes) return leave_to_other(p);     // the split kernel's problem
    const int num_kb = p.K / BK;
    // The work list is the host's, or, when only the device knows the row count, the same plan
    // rebuilt here from that count (every thread computes the same values).
    int M = p.M, span = span_host, tiles_full = tiles_full_host, num_tiles = num_tiles_host;
    if (p.m_dev) {
        M = true_rows(p);
        const int tiles_m = (M + kPairBM - 1) / kPairBM, tiles_n = (p.N + BN - 1) / BN;
        const int tiles = tiles_m * tiles_n;
        const int rem = tiles % num_pairs;
        tiles_full = (group == 0 && rem > 0 && 2 * rem <= num_pairs) ? tiles - rem : tiles;
        num_tiles = tiles_full + 2 * (tiles - tiles_full);
        span = (group != 0 || M >= p.N) ? -tiles_n : tiles_m;
    }
    constexpr uint32_t kTmemCols = 2 * BN;       // two accumulator buffers

    if (threadIdx.x == 0) {
        abort_flag_s = 0;
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&acc_full[a], 1);
            mbar_init(&acc_empty[a], 16);
        }
        fence_barrier_init();
        prefetch_tmap(&tmap_a);
        prefetch_tmap(&tmap_w);
        prefetch_tmap(&tmap_w_half);
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, kTmemCols);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                          // both CTAs' barriers exist before either signals the other
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if (count_known(p)) pdl_wait();
    if (p.early_trigger) pdl_launch_dependents();
    if (blockIdx.x == 0) advance_kv_len(p);

    if (warp == 0) {
        if (elect_one()) {
            long it = 0;                         // k-blocks issued so far over all tiles of this pair
            bool ok = true;
            for (int local = 0; ok; ++local) {
                const int tile = pair_entry(local, pair, num_pairs, num_tiles, group);
                if (tile < 0) break;
                const PairTile t = decode_tile<BN>(tile, span, tiles_full);
                const int m0 = t.m0 + (int)rank * 128;
                const int n0 = t.n0 + (int)rank * (t.bn / 2);
                const CUtensorMap* wmap = (t.bn == BN) ? &tmap_w : &tmap_w_half;
                const uint32_t stage_tx = 2u * (uint32_t)(L::kABytes + (t.bn / 2) * BK * 2);
                for (int kb = 0; kb < num_kb; ++kb, ++it) {
                    const int s = (int)(it % STAGES);
                    if (it >= STAGES && !mbar_wait(&empty_bar[s], (uint32_t)((it / STAGES) - 1) & 1, abort_flag, p.status)) {
                        ok = false;
                        break;
                    }
                    uint8_t* a_dst = smem + s * L::kStageBytes;
                    uint8_t* b_dst = a_dst + L::kABytes;
                    if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], stage_tx);
                    const uint32_t bar = map_to_cta(smem_u32(&full_bar[s]), 0);
                    tma_load_2d_pair(a_dst, &tmap_a, bar, kb * BK, m0);
                    tma_load_2d_pair(b_dst, wmap, bar, kb * BK, n0);
                }
            }
            if (*abort_flag && rank == 0) {
                // let the copies already issued land before shared memory is released
                for (long k2 = (it > STAGES ? it - STAGES : 0); k2 < it; ++k2)
                    mbar_drain(&full_bar[k2 % STAGES], (uint32_t)(k2 / STAGES) & 1);
            }
        }
    } else if (warp == 1) {
        if (rank == 0 && elect_one()) {
            // One elected thread of the leader CTA does nothing but wait and issue. Per 64-wide k-block
            // the tensor core works 512 clocks (four M=256, N=256, K=16 instructions); the thread spends
            // about 80 clocks per instruction, 50 on the commit and 65 on a wait that is already
            // satisfied, which leaves a margin. The earlier form, the whole warp in lockstep with every
            // lane polling the barrier and a vote after it, paid about 300 clocks per wait and made the
            // issuing warp, not the tensor core, the limit of the main loop (tensor pipe 75 % active).
            constexpr uint32_t idesc_whole = idesc_bf16_f32(kPairBM, BN, 0);
            constexpr uint32_t idesc_half = idesc_bf16_f32(kPairBM, BN / 2, 0);
            const uint64_t a_desc = smem_desc_sw128(smem_u32(smem), 16, 1024);
            int s = 0;                 // ring position and phase parity of the next k-block
            uint32_t par = 0;
            int local = 0;
            bool ok = true;
            for (; ok; ++local) {
                const int tile = pair_entry(local, pair, num_pairs, num_tiles, group);
                if (tile < 0) break;
                const int a = local & 1;
                if (local >= 2) {
                    ok = mbar_wait(&acc_empty[a], (uint32_t)((local >> 1) - 1) & 1, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                }
                const uint32_t d_tmem = tmem_base + (uint32_t)(a * BN);
                const uint32_t idesc = (tile < tiles_full) ? idesc_whole : idesc_half;
                for (int kb = 0; kb < num_kb; ++kb) {
                    ok = mbar_wait(&full_bar[s], par, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t ad = a_desc + (uint32_t)s * (uint32_t)(L::kStageBytes >> 4);
                    const uint64_t bd = ad + (uint32_t)(L::kABytes >> 4);
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        mma_bf16_ss_pair(d_tmem, ad + (uint32_t)(kk * 2), bd + (uint32_t)(kk * 2), idesc, (kb | kk) ? 1u : 0u);
                    mma_commit_pair(&empty_bar[s], 3);      // frees the stage in both CTAs
                    if (++s == STAGES) { s = 0; par ^= 1u; }
                }
                if (ok) mma_commit_pair(&acc_full[a], 3);    // accumulator complete in both CTAs
            }
        }
    } else {
        // epilogue: warp w may touch TMEM lanes 32*(w%4) .. +31 of this CTA's half of the tile. Two
        // warps share each lane quarter and take alternate 32-column chunks: the epilogue of a tile
        // is a long chain of dependent instructions per thread, and with one warp per quarter the
        // GELU epilogue took longer than the tile's main loop. (The entropy epilogue carries a row's
        // state from chunk to chunk in one thread, so there the second warp of a quarter only
        // signals.)
        const int q = warp & 3;
        const int c_first = (warp - 2) >> 2;
        const bool idle_warp = (EPI == NOVA_EPI_ENTROPY) && warp >= 6;
        const uint32_t acc_empty_leader = map_to_cta(smem_u32(&acc_empty[0]), 0);
        int local = 0;
        bool ok = true;
        EntropyState est;
        est.reset();
        for (; ok; ++local) {
            const int tile = pair_entry(local, pair, num_pairs, num_tiles, group);
            if (tile < 0) break;
            const int a = local & 1;
            const PairTile t = decode_tile<BN>(tile, span, tiles_full);
            const int row0 = t.m0 + (int)rank * 128 + q * 32, row = row0 + lane;
            const int n0 = t.n0, n_chunks = t.bn / 32;
            const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * BN);
            if constexpr (EPI == NOVA_EPI_ENTROPY) {
                ok = mbar_wait_warp(&acc_full[a], (uint32_t)(local >> 1) & 1, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
#pragma unroll 1
                for (int c = 0; c < n_chunks && !idle_warp; ++c) {
                    const int col0 = n0 + c * 32;
                    uint32_t acc[32];
                    tmem_ld32(t_addr + (uint32_t)(c * 32), acc);
                    tmem_ld_wait();
                    if (row < M && col0 < p.N) est.add_chunk(acc, p.bias ? p.bias + col0 : nullptr);
                }
            } else {
                // After the turn-round this lane holds features 4 * (lane % 8) .. + 3 of a chunk's 32, of rows
                // row0 + lane / 8 + 4 i. What the epilogue reads of the first chunk is fetched before the accumulator is
                // ready, of the next one while this one is worked on, with a residual alone of the one after that
                // (K = 2048 leaves little time for it: by itself, 8192 rows x 2048 features 71.4 -> 68.2 us, 3277 rows 37.7 -> 34.6; whole calls,
                // at the power limit, the same); in a pair's last tile all of it is brought to L2 before. With a residual the
                // loop is not unrolled: a launch whose pairs have one tile each runs this code once. After the last MMA of
                // 2252 rows x 1920 features, gated, it takes 6.4 us (7 before, unrolled and with the gate's row looked up and loaded
                // in turn), 8.7 with a second output (13, its other operand loaded where it was used): latency of what is
                // in flight per SM, 32 KB. GELU unrolled takes 2.5 us, in a loop 4.1.
                const int rows0 = row0 + (lane >> 3);
                const int chunks = row0 < M ? min(n_chunks, (p.N - n0) / 32) : 0;
                int col = n0 + c_first * 32 + (lane & 7) * 4;
                EpiRows<EPI> er;
                constexpr bool kTwoAhead = EPI == NOVA_EPI_BIAS_RES && !DIFF;
                EpiData<EPI, DIFF> ed, ed_next;
                uint2 bias = make_uint2(0, 0);
                const bool last_tile = pair_entry(local + 1, pair, num_pairs, num_tiles, group) < 0;
                if (EPI == NOVA_EPI_BIAS_RES && last_tile && chunks > 0) {
                    // the tile's part of this lane's row, of the residual (first warp of the quarter) or of diff_in
                    const int at = min(row, M - 1), in = p.res_row ? p.res_row[at] : at, out = p.out_row ? p.out_row[at] : at;
                    const __nv_bfloat16* src = c_first == 0 ? p.res + (long)in * p.N : p.diff_out ? p.diff_in + (long)out * p.N : nullptr;
                    if (src)
                        for (int c = 0; c < chunks; c += 2) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + n0 + c * 32));
                }
                if (c_first < chunks) {
                    er.template load<4>(p, rows0, M);
                    bias = *(const uint2*)(p.bias + col);
                    ed.fetch(p, er, col);
                    if (kTwoAhead && c_first + 2 < chunks) ed_next.fetch(p, er, col + 64);
                }
                ok = mbar_wait_warp(&acc_full[a], (uint32_t)(local >> 1) & 1, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                // the next kernel is let in at the last tile (measured at the split kernel's trigger)
                if (last_tile) pdl_launch_dependents();
                float* turn = (float*)(smem + L::kTurnOff + (warp - 2) * 4096);
#pragma unroll (EPI == NOVA_EPI_BIAS_RES ? 1 : BN / 64)
                for (int c = 0; c < BN / 64; ++c, col += 64) {
                    const int ch = 2 * c + c_first;
                    if (ch >= chunks) break;
                    EpiData<EPI, DIFF> ed_after;
                    uint2 bias_next = make_uint2(0, 0);
                    if (ch + 2 < chunks) {
                        bias_next = *(const uint2*)(p.bias + col + 64);
                        if (!kTwoAhead) ed_next.fetch(p, er, col + 64);
                    }
                    if (kTwoAhead && ch + 4 < chunks) ed_after.fetch(p, er, col + 128);
                    uint32_t acc[32];
                    tmem_ld32(t_addr + (uint32_t)(ch * 32), acc);
                    tmem_ld_wait();
                    // 32 rows x 32 fp32, 16-byte pieces XOR-swizzled by the row: no bank conflicts either way
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        *(uint4*)(turn + lane * 32 + ((i ^ (lane & 7)) << 2)) =
                            make_uint4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
                    __syncwarp();
                    float v[4][4];
                    auto take = [&](int from) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int rr = (lane >> 3) + 4 * (from + i);
                            *(float4*)v[i] = *(const float4*)(turn + rr * 32 + (((lane & 7) ^ (rr & 7)) << 2));
                        }
                    };
                    take(0);
                    epi_store<EPI, 4, 0, DIFF>(p, rows0, M, er, col, bias, ed, v);
                    take(4);
                    epi_store<EPI, 4, 4, DIFF>(p, rows0, M, er, col, bias, ed, v);
                    ed = ed_next;
                    if (kTwoAhead) ed_next = ed_after;
                    bias = bias_next;
                }
            }
            if (EPI == NOVA_EPI_ENTROPY && !idle_warp && (t.n0 + BN >= p.N || pair_entry(local + 1, pair, num_pairs, num_tiles, group) < 0)) {
                // this pair's last column tile of the row block
                bool mine = true;
                const int block0 = group < 0 ? tile - tile % -group : 0, first = range_owner(block0, num_pairs, num_tiles);
                const int last = range_owner(block0 - group - 1, num_pairs, num_tiles);
                if (group < 0 && first != last) {
                    // a pair's parts: of its first row block, and of another that is its last
                    auto slot = [&](int of) {
                        const int which = range_start(of, num_pairs, num_tiles) < block0 ? 1 : 0;
                        return p.head_part + (size_t)(of * 2 + which) * NOVA_HEAD_SLOT_FLOATS + rank * 128 + q * 32 + lane;
                    };
                    est.publish(slot(pair));
                    // A ticket for each warp's 32 rows, not one for the block behind a barrier: a warp that gives up a wait leaves
                    // the loop alone, and the others would stay at a barrier for good.
                    __threadfence();
                    __syncwarp();
                    unsigned int drawn = 0;
                    if (lane == 0) {
                        unsigned int* ticket = p.head_tickets + (first * 2 + rank) * 4 + q;
                        drawn = atomicAdd(ticket, 1u);
                        if ((int)drawn == last - first) *ticket = 0;       // ready for the next launch
                        __threadfence();
                    }
                    mine = (int)__shfl_sync(0xffffffffu, drawn, 0) == last - first;      // everybody else has published
                    if (mine) {
                        for (int of = first; of <= last; ++of) est.merge(slot(of), of == first);      // in this order, whoever does it
                    }
                }
                if (mine && row < M) p.ent[row] = est.finish(p.status);
                est.reset();
            }
            // this warp has read its part of the buffer: tell the leader's MMA thread
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acc_empty_leader + (uint32_t)(a * 8));
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();     // the peer may still read this CTA's shared memory or signal its barriers
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

template <int BN, int STAGES, int EPI, bool DIFF = false>
nova_status launch_pair(nova_ctx* ctx, const nova_gemm_args& a, cudaStream_t st)
{
    using L = PairSmem<BN, STAGES>;
    CUtensorMap ta, tw;
    const uint64_t da[2] = {(uint64_t)a.K, (uint64_t)a.M}, sa[1] = {(uint64_t)a.K * 2};
    const uint64_t dw[2] = {(uint64_t)a.K, (uint64_t)a.N}, sw[1] = {(uint64_t)a.K * 2};
    CUtensorMap tw_half;
    if (!make_tmap_bf16(ctx, &ta, a.A, 2, da, sa, 128) || !make_tmap_bf16(ctx, &tw, a.W, 2, dw, sw, BN / 2) ||
        !make_tmap_bf16(ctx, &tw_half, a.W, 2, dw, sw, BN / 4))
        return nova_fail(ctx, NOVA_ERR_CUDA, "gemm: cuTensorMapEncodeTiled failed");
    auto kern = gemm_bf16_tn_pair<BN, STAGES, EPI, DIFF>;
    static bool attr_done[64];
    if (ctx->device < 64 && !attr_done[ctx->device]) {
        NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::kTotal));
        attr_done[ctx->device] = true;
    }
    GemmParams p = make_params(ctx, a);
    const int tiles_m = (a.M + kPairBM - 1) / kPairBM, tiles_n = (a.N + BN - 1) / BN;
    const int tiles = tiles_m * tiles_n;
    constexpr bool entropy = (EPI == NOVA_EPI_ENTROPY);
    const int all_pairs = min(ctx->num_sms / 2, NOVA_TICKETS / 8), block_pairs = min(tiles_m, all_pairs);
    const bool ranges = entropy && 6 * ((tiles + all_pairs - 1) / all_pairs) <= 5 * ((tiles_m + block_pairs - 1) / block_pairs) * tiles_n;
    const int pairs = entropy && !ranges ? block_pairs : min(tiles, all_pairs);
    // a last partial wave that would occupy at most half of the pairs runs as half-width tiles
    const int rem = tiles % pairs;
    const int tiles_full = (!entropy && rem > 0 && 2 * rem <= pairs) ? tiles - rem : tiles;
    const int entries = tiles_full + 2 * (tiles - tiles_full);
    {
        nova_launch_scope scope(ctx, a.cat, st);
        // sweep the smaller operand; the entropy epilogue needs the N-fastest order
        const int span = (entropy || (long)a.M >= (long)a.N) ? -tiles_n : tiles_m;
        NOVA_CUDA_CHECK(ctx, nova_launch_pdl(kern, dim3(2 * pairs), dim3(kPairThreads), L::kTotal, st, 0, ta, tw, tw_half, p, span,
                                             tiles_full, entries, !entropy ? 0 : ranges ? -tiles_n : tiles_n, split_caps(ctx->num_sms)));
    }
    return NOVA_OK;
}

// ---- split-K kernel for problems that leave SM pairs idle ------------------------------------------
// With few 256 x 256 tiles a GEMM is bound by latency and by how many SMs pull weights, not by the
// tensor cores. Here the weights are the M operand: a pair of CTAs computes out^T[256 features, nt tokens], nt
// a multiple of 32 up to 256, so that few tokens cost little padding, and K is split over s = 1 or 2
// pairs of one cluster. Each pair sends every other one its share of the tokens of the fp32 partial tile
// straight into that pair's shared memory (in the ring, which is idle by then) as [part][token][feature];
// after a cluster barrier each CTA adds up the parts of its tokens, always in the order 0, 1, and
// runs the epilogue on four consecutive features per lane, with the residual rows fetched before the
// accumulator was ready. No global scratch, no atomics, nothing that depends on timing.
// Measured in a graph over cold weights, against the kernel this replaced (one 128 x 128 tile per CTA, three
// stages, no split): tokens x features x K = 256 x 1024 x 4096 11 us (26), 300 x 2048 x 8192 19 us (61),
// 300 x 6144 x 2048 14 us (19). Launch, first load, exchange and epilogue are 5 to 7 us of each.
constexpr int kSplitThreads = 320;     // producer warp, MMA warp, eight epilogue warps
constexpr int kSplitRing = 192 * 1024;
constexpr int kSplitSmem = kSplitRing + 1024 /*alignment slack*/ + 256 /*barriers*/;
constexpr int kSplitMaxStages = 10;

__device__ __forceinline__ void st_shared(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t cluster_addr, uint32_t v)
{
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
// Barriers as in gemm_bf16_tn_pair (full: the pair leader's copy counts both CTAs' bytes; empty and
// acc_full: signalled in both CTAs by the leader's commit). A unit of work is one output tile, run by s
// consecutive pairs of a cluster of pc pairs. Every CTA passes the same cluster barriers whether or not
// its pair has a unit, also after a failed wait.
template <int EPI>
__global__ void __launch_bounds__(kSplitThreads, 1)
gemm_bf16_split(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
                const GemmParams p, const int pc, const int box, const SplitPlan plan_host, const SplitCaps caps)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (!count_known(p)) pdl_wait();
    const int M = true_rows(p);
    const int num_kb = p.K / BK;
    const SplitPlan plan = p.m_dev ? split_plan(M, p.N, num_kb, caps) : plan_host;
    if (!plan.takes) return leave_to_other(p);      // (only with a device-side count)
    if (M <= 0) {
        pdl_wait();
        if (blockIdx.x == 0) advance_kv_len(p);
        return;
    }
    const int nt = plan.nt, s = 1 << plan.ls;
    const int tiles_t = (M + nt - 1) / nt;
    const int units = ((p.N + 255) / 256) * tiles_t;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full_bar = (uint64_t*)(smem + kSplitRing);
    uint64_t* empty_bar = full_bar + kSplitMaxStages;
    uint64_t* acc_full = empty_bar + kSplitMaxStages;
    uint32_t* tmem_slot = (uint32_t*)(acc_full + 1);
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;

    const uint32_t crank = cluster_ctarank();
    const int r = (int)(crank & 1u), pi = (int)(crank >> 1);          // CTA of the pair, pair of the cluster
    const uint32_t leader = crank & ~1u;
    const int groups = pc >> plan.ls, group = pi >> plan.ls, part = pi & (s - 1);   // units of the cluster, mine, my share of K
    const int num_clusters = gridDim.x / (2 * pc), cluster = blockIdx.x / (2 * pc);
    const int kb0 = part * num_kb / s, kb1 = (part + 1) * num_kb / s;
    const int stage_bytes = 16384 + nt * 64;
    const int stages = min(kSplitMaxStages, kSplitRing / stage_bytes);
    const int share = nt >> plan.ls;                                  // tokens whose sums this pair completes

    if (threadIdx.x == 0) {
        abort_flag_s = 0;
        for (int i = 0; i < stages; ++i) {
            mbar_init(&full_bar[i], 1);
            mbar_init(&empty_bar[i], 1);
        }
        mbar_init(acc_full, 1);
        fence_barrier_init();
        prefetch_tmap(&tmap_w);
        prefetch_tmap(&tmap_x);
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, 256);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if (count_known(p)) pdl_wait();
    if (p.early_trigger) pdl_launch_dependents();
    if (blockIdx.x == 0) advance_kv_len(p);

    int it0 = 0;                 // k-blocks of the earlier units: position in the ring
    uint32_t acc_parity = 0;
    for (int c = cluster; c * groups < units; c += num_clusters, acc_parity ^= 1u, it0 += kb1 - kb0) {
        const int unit = c * groups + group;
        const bool active = unit < units;
        const int f0 = (unit / tiles_t) * 256 + r * 128;              // this CTA's first feature
        const int t0 = (unit % tiles_t) * nt;                         // the unit's first token
        // epilogue of this thread: features col .. col + 3 of the tokens first, first + 8, ... < t_end
        const int col = f0 + lane * 4;
        const int first = t0 + part * share + warp - 2, t_end = min(t0 + (part + 1) * share, M);
        EpiRows<EPI> er;
        EpiData<EPI, true> ed;
        uint2 bias = make_uint2(0, 0);
        if (warp == 0) {
            if (active && elect_one()) {
                const uint32_t stage_tx = 2u * (uint32_t)stage_bytes;
                int issued = it0, stage = it0 % stages;
                uint32_t phase = (uint32_t)(it0 / stages) & 1u;
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (issued >= stages && !mbar_wait(&empty_bar[stage], phase ^ 1u, abort_flag, p.status)) break;
                    uint8_t* w_dst = smem + stage * stage_bytes;
                    uint8_t* x_dst = w_dst + 16384;
                    if (r == 0) mbar_arrive_expect_tx(&full_bar[stage], stage_tx);
                    const uint32_t bar = map_to_cta(smem_u32(&full_bar[stage]), leader);
                    tma_load_2d_pair(w_dst, &tmap_w, bar, kb * BK, f0);
                    for (int i = 0; i < nt / 2; i += box)
                        tma_load_2d_pair(x_dst + i * 128, &tmap_x, bar, kb * BK, t0 + r * (nt / 2) + i);
                    ++issued;
                    if (++stage == stages) { stage = 0; phase ^= 1u; }
                }
                if (*abort_flag && r == 0)      // let the copies already issued land before anything reuses the ring
                    for (int i = max(0, issued - stages); i < issued; ++i)
                        mbar_drain(&full_bar[i % stages], (uint32_t)(i / stages) & 1u);
            }
        } else if (warp == 1) {
            if (active && r == 0 && elect_one()) {
                const uint32_t idesc = idesc_bf16_f32(256, nt, 0);
                const uint64_t w_desc = smem_desc_sw128(smem_u32(smem), 16, 1024);
                int stage = it0 % stages;
                uint32_t phase = (uint32_t)(it0 / stages) & 1u;
                bool ok = true;
                for (int kb = kb0; kb < kb1; ++kb) {
                    ok = mbar_wait(&full_bar[stage], phase, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t wd = w_desc + (uint32_t)stage * (uint32_t)(stage_bytes >> 4);
                    const uint64_t xd = wd + (16384u >> 4);
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        mma_bf16_ss_pair(tmem_base, wd + (uint32_t)(kk * 2), xd + (uint32_t)(kk * 2), idesc,
                                         (kb != kb0 || kk) ? 1u : 0u);
                    mma_commit_pair(&empty_bar[stage], (uint16_t)(3u << leader));
                    if (++stage == stages) { stage = 0; phase ^= 1u; }
                }
                if (ok) mma_commit_pair(acc_full, (uint16_t)(3u << leader));
            }
        } else if (active) {
            if (EPI == NOVA_EPI_BIAS_RES) {
                // the rows of the later tokens, residual and diff_in, to L2: one token per lane, two lines of each
                for (int t = t0 + part * share + threadIdx.x - 64; t < t_end; t += 256) {
                    const long in = p.res_row ? p.res_row[t] : t, out = p.out_row ? p.out_row[t] : t;
                    for (int c = f0; c < min(f0 + 128, p.N); c += 64) {
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(p.res + in * p.N + c));
                        if (p.diff_out) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.diff_in + out * p.N + c));
                    }
                }
            }
            if (col < p.N && first < t_end) {
                bias = *(const uint2*)(p.bias + col);
                er.template load<8>(p, first, t_end);
                ed.fetch(p, er, col);
            }
            if (mbar_wait_warp(acc_full, acc_parity, abort_flag, p.status)) tc_fence_after();
        }
        __syncwarp();
        // Every pair's main loop is over: the rings may be written. (Unsplit, a CTA writes only its own, which acc_full gave free.)
        if (s > 1) cluster_sync_all();
        // The next kernel is let in when the last main loop is over: with the trigger at the start its first CTAs sat
        // on the SMs this grid leaves free, and it ended later. With the same in the kernel for many tiles, us: a
        // 16-layer 256x256 generation 9489 -> 9292, 20x20 scale of one image 3140 -> 3097, last 64x64 scale in a
        // graph 6905 -> 6858. (Right after the wait the generation gains as much and the others less.)
        if (warp >= 2 && (c + num_clusters) * groups >= units) pdl_launch_dependents();
        if (warp >= 2 && active) {
            // token t of this CTA's 128 features (one per lane and tensor-memory lane quarter) to the pair that
            // completes it; the store of a warp is 128 contiguous bytes
            const int q = warp & 3;
            const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16);
            const uint32_t slot = smem_u32(smem) + (uint32_t)(part * share * 512 + (q * 32 + lane) * 4);
#pragma unroll 1
            for (int ch = (warp - 2) >> 2; ch < nt / 32; ch += 2) {
                uint32_t acc[32];
                tmem_ld32(t_addr + (uint32_t)(ch * 32), acc);
                tmem_ld_wait();
#pragma unroll
                for (int g = 0; g < 4; ++g) {        // eight tokens always belong to one pair (share % 8 == 0)
                    const int t = ch * 32 + g * 8, owner = t >= share;          // (two parts at most)
                    const uint32_t off = (uint32_t)((t - owner * share) * 512);
                    if (owner == part) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) st_shared(slot + off + (uint32_t)(i * 512), acc[g * 8 + i]);
                    } else {
                        const uint32_t dst = map_to_cta(slot, (uint32_t)(2 * ((group << plan.ls) + owner) + r)) + off;
#pragma unroll
                        for (int i = 0; i < 8; ++i) st_cluster(dst + (uint32_t)(i * 512), acc[g * 8 + i]);
                    }
                }
            }
            tc_fence_before();
        }
        __syncwarp();
        if (s > 1) cluster_sync_all();          // every part of this CTA's tokens has arrived
        else if (warp >= 2) asm volatile("bar.sync 1, 256;" ::: "memory");
        if (warp >= 2 && active && col < p.N) {
            const float* parts = (const float*)smem + lane * 4 - (t0 + part * share) * 128;
            for (int t = first; t < t_end; t += 64) {
                EpiRows<EPI> er_next;
                if (t + 64 < t_end) er_next.template load<8>(p, t + 64, t_end);      // (there are no registers for what they point to)
                float v[4][4];
                auto take = [&](int from) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) *(float4*)v[i] = *(const float4*)(parts + (t + 8 * (from + i)) * 128);
                    for (int j = 1; j < s; ++j) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float4 w = *(const float4*)(parts + (j * share + t + 8 * (from + i)) * 128);
                            v[i][0] += w.x; v[i][1] += w.y; v[i][2] += w.z; v[i][3] += w.w;
                        }
                    }
                };
                take(0);
                epi_store<EPI, 8, 0, true>(p, t, t_end, er, col, bias, ed, v);
                if (t + 32 < t_end) {
                    take(4);
                    epi_store<EPI, 8, 4, true>(p, t, t_end, er, col, bias, ed, v);
                }
                if (t + 64 < t_end) {
                    er = er_next;
                    ed.fetch(p, er, col);
                }
            }
        }
        fence_proxy_async_smem();    // the next unit's copies overwrite what was written and read here
        __syncthreads();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();     // a peer's commit may still signal this CTA's barriers
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 256);
    }
}

// Once per context: shared memory opt-in of the split kernel; its clusters have to fit the device at all.
nova_status split_setup(nova_ctx* ctx)
{
    if (ctx->attr_split) return NOVA_OK;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(kSplitThreads); cfg.dynamicSmemBytes = kSplitSmem; cfg.attrs = attr; cfg.numAttrs = 1;
    NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(gemm_bf16_split<NOVA_EPI_QKV>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem));
    NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(gemm_bf16_split<NOVA_EPI_BIAS_RES>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem));
    NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(gemm_bf16_split<NOVA_EPI_BIAS_GELU>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem));
    for (int ls = 0; ls < 2; ++ls) {
        attr[0].val.clusterDim.x = 2u << ls;
        cfg.gridDim = dim3(2u << ls);
        int n = 0;
        NOVA_CUDA_CHECK(ctx, cudaOccupancyMaxActiveClusters(&n, gemm_bf16_split<NOVA_EPI_BIAS_RES>, &cfg));
        if (n < 1) return nova_fail(ctx, NOVA_ERR_CUDA, "gemm: no cluster of the split kernel fits the device");
    }
    ctx->attr_split = true;
    return NOVA_OK;
}

template <int EPI>
nova_status launch_split(nova_ctx* ctx, const nova_gemm_args& a, const SplitPlan& plan, cudaStream_t st)
{
    const SplitCaps caps = split_caps(ctx->num_sms);
    const int tiles_n = (a.N + 255) / 256;
    int pc, box, clusters;
    if (a.m_dev) {
        // only the device knows the row count: clusters for the wider split; unsplit tiles run two to a cluster
        pc = a.K / BK >= 2 ? 2 : 1; box = 16; clusters = caps.c[pc - 1];
    } else {
        pc = 1 << plan.ls; box = plan.nt / 2; clusters = tiles_n * ((a.M + plan.nt - 1) / plan.nt);
    }
    CUtensorMap tw, tx;
    const uint64_t dx[2] = {(uint64_t)a.K, (uint64_t)a.M}, sx[1] = {(uint64_t)a.K * 2};
    const uint64_t dw[2] = {(uint64_t)a.K, (uint64_t)a.N}, sw[1] = {(uint64_t)a.K * 2};
    if (!make_tmap_bf16(ctx, &tw, a.W, 2, dw, sw, 128) || !make_tmap_bf16(ctx, &tx, a.A, 2, dx, sx, (uint32_t)box))
        return nova_fail(ctx, NOVA_ERR_CUDA, "gemm: cuTensorMapEncodeTiled failed");
    const GemmParams p = make_params(ctx, a);
    {
        nova_launch_scope scope(ctx, a.cat, st);
        NOVA_CUDA_CHECK(ctx, nova_launch_pdl(gemm_bf16_split<EPI>, dim3(clusters * 2 * pc), dim3(kSplitThreads), kSplitSmem, st, 2 * pc,
                                             tw, tx, p, pc, box, plan, caps));
    }
    return NOVA_OK;
}

template <int EPI>
nova_status launch_gemm(nova_ctx* ctx, const nova_gemm_args& a, cudaStream_t st)
{
    // When only the device knows the row count and the bound is past the split kernel's range, both kernels
    // are launched and the one whose range the true count is not in returns at once.
    const nova_status rc = split_setup(ctx);
    if (rc != NOVA_OK) return rc;
    const SplitPlan plan = split_plan(a.M, a.N, a.K / BK, split_caps(ctx->num_sms));
    if (plan.takes || a.m_dev) {
        const nova_status rs = launch_split<EPI>(ctx, a, plan, st);
        if (rs != NOVA_OK || plan.takes) return rs;
    }
    if (EPI == NOVA_EPI_BIAS_RES && a.diff_out) return launch_pair<256, 6, EPI, EPI == NOVA_EPI_BIAS_RES>(ctx, a, st);
    return launch_pair<256, 6, EPI>(ctx, a, st);
}

}  // namespace

extern "C" int nova_debug_gemm_plan(int num_sms, int M, int N, int K, int* k_parts, int* token_tile)
{
    const SplitPlan plan = split_plan(M, N, K / BK, split_caps(num_sms));
    *k_parts = 1 << plan.ls;
    *token_tile = plan.nt;
    return plan.takes ? 1 : 0;
}

nova_status nova_launch_gemm(nova_ctx* ctx, const nova_gemm_args& a, cudaStream_t st)
{
    if (a.M <= 0) return NOVA_OK;
    if (a.K % BK || a.N % 32 || a.K < BK) return nova_fail(ctx, NOVA_ERR_SHAPE, "gemm: K must be a multiple of 64 and N of 32");
    if (ctx->num_sms < 2) return nova_fail(ctx, NOVA_ERR_SHAPE, "gemm: needs at least two SMs");
    if (a.epilogue == NOVA_EPI_ENTROPY) return launch_pair<256, 6, NOVA_EPI_ENTROPY>(ctx, a, st);
    if (a.epilogue == NOVA_EPI_QKV) return launch_gemm<NOVA_EPI_QKV>(ctx, a, st);
    if (a.epilogue == NOVA_EPI_BIAS_GELU) return launch_gemm<NOVA_EPI_BIAS_GELU>(ctx, a, st);
    return launch_gemm<NOVA_EPI_BIAS_RES>(ctx, a, st);
}
