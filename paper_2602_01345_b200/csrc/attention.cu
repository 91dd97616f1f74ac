// Attention of the kept queries over [prior-scale K/V cache ++ kept tokens' own K/V]
// (no mask), on the sm_100a tensor cores.
//
// A persistent CTA takes 128 query rows of one image and one head at a time and streams over 128-key tiles
// of K and V; at head size 128 two CTAs form a pair (cta_group::2) on 256 rows and each brings in half of
// every tile, because a CTA alone would need 1280 clocks of shared-memory bandwidth per 128 x 128 tile where
// the tensor core needs 1024. Sixteen warps:
//   warp 0        TMA producer: Q (two buffers) and a ring of stages {K of a tile, V of the tile three before it}
//   warp 1        tcgen05.mma issuer (the pair's leader issues for both): O += P_u V_u, then S_{u+3}
//   warps 4-7     epilogue: O / l to bf16, or a partial result, while the next rows are under way
//   warps 8-15    softmax, two warpgroups that take the key tiles in turn, one query row per thread: the row of
//                 S from tensor memory to registers, P = 2^((s - m) * scale - 48) packed to bf16 and stored over the
//                 S columns, from where O += P V takes it as its A operand
// Tensor memory holds O and three S buffers, so S runs up to three tiles ahead of O += P V, across the
// boundary between two work items: neither the latency of a softmax nor its hand-overs are on the tensor
// core's path as long as a tile's softmax takes less than two tiles of tensor work. (With both 128-row tiles
// of 256 rows in one CTA there was room for one S buffer each, and S, softmax and P V of a tile followed one
// another: 3285 clocks per key tile for 2048 clocks of tensor work.)
// Probabilities are taken against a reference maximum m, the row's maximum over its first key tile: bf16 and fp32
// share their exponent range, so a reference that is not the running maximum costs no precision, and it cancels
// in the final division by l. (The whole tile's, not that of some of its keys: a key that holds most of a row's
// weight then has probability 1 where it lies in that tile, which bf16 holds exactly. Over the last 32 keys alone the
// attention's error against 64 bits was 2.76e-3 instead of 2.47e-3 for peaked rows over 217 keys.) They are scaled
// by 2^-kHeadroom, exactly, because what follows can be far above the first tile and never far below what matters.
// Only a score about 2^128 (88 nats) above the reference, seen as a huge row sum, could get near the end of the
// range; work items in which one appears are run once more at the end, with a first pass over the keys that finds the
// rows' true maxima. A launch in which that happens to all items takes 2.6 times as long (4 x 2048 rows x 8473 keys, 16
// heads x 128: 428 -> 1110 us).
// K tiles are K-major operands; V tiles are the MN-major B operand, i.e. V is consumed exactly as it lies in
// the cache ([keys, dh]). The last key tile ends at the last key and overlaps the one before it (its repeated
// columns are masked; rows before the first key read as zeros), so no row past the end is ever loaded.
// MMAs issued by one thread execute in issue order, which orders "P_u read by O += P_u V" before "its
// buffer overwritten by S_{u+3}".
// When the last round of work items would fill at most half of the CTAs (pairs), each of its items is shared
// by two that take half of the key tiles each and merge their partial results (see below).
// Every mbarrier wait is bounded.
// What bounds it: at many keys power (head size 128 runs at 1.6 to 1.7 GHz) and the exponentials: 1340 clocks per
// key tile of 256 rows for 1024 of tensor work, 1050 without exponentials. In the smallest calls the chain of
// table, loads, S, softmax, O. Measured against the kernel before it (two tiles of one item in a CTA), us:
// 3277 rows x 29414 keys, 16 heads x 128: 684 -> 572; 4 x 2048 x 8473: 510 -> 416; 1024 x 7449: 86 -> 52;
// 300 x 821: 22.8 -> 12.5; 4 x 563 x 1779, 30 heads x 64: 80 -> 55; 2 x 128 x 552, 16 x 64: 11.8 -> 9.2.
#include "tc_common.cuh"

namespace {

using namespace tc;

constexpr int BQ = 128;        // query rows per CTA
constexpr int BKV = 128;       // keys per tile
constexpr int kBufs = 3;       // S buffers in tensor memory
constexpr int kThreads = 512;  // warpgroups: producer + issuer (+2 idle warps), epilogue, softmax 0, softmax 1
constexpr int kSlabBytes = 128 * 128;   // [128 rows][64 bf16]
// The probability of a score equal to the reference is 2^-kHeadroom. A row's sum of probabilities over one key tile at
// or above kHugeSum (or NaN) means a score about 2^(80 + kHeadroom) above the reference. That is far below
// anything that could overflow fp32 in l or O (sums over 2^16 keys, values up to 2^20), and at the other end
// probabilities down to 2^-78 of the reference's, and O of values down to 2^-54, keep all their bits.
constexpr float kHeadroom = 48.f;
constexpr float kHugeSum = 1.2089258e24f;   // 2^80
// Passes whose row sums and references are kept. A warpgroup that reaches pass i has done its last tile before
// that, tile t >= i - 2 if passes are single tiles; S of it was issued after O += P V of tile t - kBufs, which
// waited for the epilogue of the pass before that tile's: passes up to i - kBufs - 3 are done with their slots.
constexpr int kSlots = kBufs + 3;

template <int DH>
struct AttnCfg {
    static constexpr bool kPair = (DH == 128);
    static constexpr int kCtas = kPair ? 2 : 1;
    static constexpr int kRows = kCtas * BQ;                    // query rows of one work item
    static constexpr int kKRows = BKV / kCtas;                  // rows of K per CTA (all of dh)
    static constexpr int kVCols = DH / kCtas;                   // columns of V per CTA (all keys)
    static constexpr int kQBytes = BQ * DH * 2;
    static constexpr int kTileBytes = kKRows * DH * 2;          // K and V alike (BKV * kVCols * 2)
    static constexpr int kStages = kPair ? 4 : 5;               // stage: K of a tile and V of the tile kBufs before it
    static constexpr int kStageOff = 2 * kQBytes;
    static constexpr int kLOff = kStageOff + kStages * 2 * kTileBytes;  // [kSlots][2][128] row sums of the two warpgroups
    static constexpr int kMOff = kLOff + kSlots * 2 * BQ * 4;           // [kSlots][128] reference maxima
    static constexpr int kAOff = kMOff + kSlots * BQ * 4;               // [2][128] maxima of a maximum pass
    static constexpr int kTabOff = kAOff + 2 * BQ * 4;                  // [kTable] passes
    static constexpr int kBarOff = kTabOff + 64 * 44;
    static constexpr int kTotal = kBarOff + 512 + 1024;
    static_assert(kVCols == 64, "a V stage is one 128-byte-wide slab");
};

struct AttnParams {
    const int32_t* cu_keep;
    const int32_t* kv_len;
    __nv_bfloat16* o;
    int B, C, Lmax, n_heads, slots;      // slots: CTAs (pairs) that run at the same time
    int own_keys;          // 1: keys = cache rows followed by this call's k_b rows; 0: cache rows only (cross-attention)
    float scale_log2e;     // (1 / sqrt(dh)) * log2(e)
    // key-split of a last partial round: per split item two partial results [2][kRows][DH + 4] fp32
    // (unnormalised O row, reference maximum, sum) and a ticket counter per CTA; part == NULL: no split
    float* part;
    unsigned int* tickets;
    int part_slots;
    unsigned int* status;
};

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&t);
}

// ---- two fp32 values per 64-bit register: one instruction does both lanes' arithmetic ----------
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
__device__ __forceinline__ uint64_t add_rm_f32x2(uint64_t a, uint64_t b)   // rounds toward -inf
{
    uint64_t r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t sub_f32x2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// 2^x for two values without the special-function unit, which the softmax would otherwise
// saturate (it evaluates 16 exponentials per clock per SM against 128 multiply-adds). With
// t = x + 1.5 * 2^23 rounded toward -inf, the low bits of t hold j = floor(x) and f = x - j lies in
// [0, 1); 2^f comes from a cubic fitted to 9.2e-5 relative error (far below the bf16 rounding the
// probabilities get next) and j is added to the exponent field as an integer. x is clamped to
// [-126, 126] so that the exponent cannot wrap; a masked (-inf) score therefore yields 2^-126, not 0,
// and one far above the reference a value that the overflow check sees.
__device__ __forceinline__ void exp2_poly_x2(uint64_t x2, float& p0, float& p1)
{
    float x0, x1;
    unpack_f32x2(x2, x0, x1);
    const uint64_t xc = pack_f32x2(fminf(fmaxf(x0, -126.f), 126.f), fminf(fmaxf(x1, -126.f), 126.f));
    const uint64_t magic = pack_f32x2(12582912.f, 12582912.f);
    const uint64_t t = add_rm_f32x2(xc, magic);
    const uint64_t f = sub_f32x2(xc, sub_f32x2(t, magic));
    uint64_t q = fma_f32x2(f, pack_f32x2(0.07711965590715408f, 0.07711965590715408f),
                           pack_f32x2(0.2276432067155838f, 0.2276432067155838f));
    q = fma_f32x2(q, f, pack_f32x2(0.6950892806053162f, 0.6950892806053162f));
    q = fma_f32x2(q, f, pack_f32x2(1.f, 1.f));
    float q0, q1, t0, t1;
    unpack_f32x2(q, q0, q1);
    unpack_f32x2(t, t0, t1);
    p0 = __uint_as_float(__float_as_uint(q0) + (__float_as_uint(t0) << 23));
    p1 = __uint_as_float(__float_as_uint(q1) + (__float_as_uint(t1) << 23));
}

// One pass over the keys of a work item. Work items are (head, query block), blocks fastest so that CTAs
// running together share K/V in L2. All items of an image cost the same, so when the last round of them would
// occupy at most half of the slots, each of its items becomes two passes, one per half of the keys. Both leave
// their unnormalised result (O row, reference maximum, sum) in scratch memory and draw a ticket; the one that
// draws the second ticket finds the other's result complete, merges the two and writes the output. Nobody
// waits for anybody.
// The passes of a CTA (pair) are laid out in shared memory, kTable at a time: the roles read what they need of
// them instead of each carrying the whole state in its few registers.
constexpr int kTable = 64;
// Publishing and merging a partial result takes as long as about five key tiles, which halving fewer than twelve
// would not win back.
constexpr int kSplitTiles = 12;
struct Pass {
    int x;               // first column of the head
    int b, q_begin, rows_valid;
    int n;               // key tiles of this pass; 0: nothing to do (but zeros to write if `empty`)
    int first;           // first key of the first tile
    int last;            // first key of the last tile (it ends at the image's last key if the pass does)
    int masked;          // columns of the last tile that repeat keys of the tile before, or precede key 0
    int half;            // -1, or which half of a split item, + 2 * its slot
    int empty;
    int over;            // past the last pass of the launch
};

// cu, len: cu_keep and kv_len, or copies of them in shared memory.
template <int DH>
__device__ __forceinline__ Pass make_pass(const AttnParams& p, const int32_t* cu, const int32_t* len, int entry)
{
    constexpr int kRows = AttnCfg<DH>::kRows;
    Pass r;
    r.n = 0;
    r.empty = 0;
    r.over = 0;
    int units = 0;
    for (int i = 0; i < p.B; ++i) units += (cu[i + 1] - cu[i] + kRows - 1) / kRows;
    const int items = units * p.n_heads, rem = items % p.slots;
    const bool split = p.part && rem > 0 && 2 * rem <= p.slots && rem <= p.part_slots;
    const int whole = split ? items - rem : items;
    if (entry >= whole + 2 * (items - whole)) {
        r.over = 1;
        return r;
    }
    int item = entry, khalf = -1, slot = 0;
    if (item >= whole) {
        slot = (item - whole) >> 1;
        khalf = (item - whole) & 1;
        item = whole + slot;
    }
    const int head = item / units;
    int block = item - head * units, k_b = 0;
    r.x = head * DH;
    for (r.b = 0; r.b < p.B; ++r.b) {
        const int c0 = cu[r.b];
        k_b = cu[r.b + 1] - c0;
        const int blocks = (k_b + kRows - 1) / kRows;
        if (block < blocks) { r.q_begin = c0 + block * kRows; break; }
        block -= blocks;
    }
    r.rows_valid = min(kRows, k_b - block * kRows);
    const int n_keys = min(max(len[r.b], 0) + (p.own_keys ? k_b : 0), p.Lmax);
    const int tiles = (n_keys + BKV - 1) / BKV;
    if (khalf >= 0 && tiles < kSplitTiles) {      // too few key tiles to share: the first half takes them all
        if (khalf == 1) return r;
        khalf = -1;
    }
    const int t0 = khalf == 1 ? (tiles + 1) / 2 : 0, t1 = khalf == 0 ? (tiles + 1) / 2 : tiles;
    r.n = t1 - t0;
    r.empty = r.n == 0;
    r.first = t0 * BKV;
    r.last = t1 == tiles ? n_keys - BKV : (t1 - 1) * BKV;
    r.masked = t1 == tiles ? tiles * BKV - n_keys : 0;
    r.half = khalf < 0 ? -1 : khalf + 2 * slot;
    return r;
}

template <int DH>
__global__ void __launch_bounds__(kThreads, 1)
attention_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                 const __grid_constant__ CUtensorMap tmap_v, const AttnParams p)
{
    using L = AttnCfg<DH>;
    constexpr bool kPair = L::kPair;
    constexpr int kStages = L::kStages;
    // Tensor memory: O (fp32, DH columns) at column 0, S buffer i (fp32) at 128 + 128 i; P (bf16 pairs) over the
    // first 64 columns of its S buffer.
    constexpr uint32_t kTmemCols = 512;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    // Barriers; at head size 128 those marked * are used in the leader's shared memory and count both CTAs, and
    // commits signal the others in both.
    uint64_t* bars = (uint64_t*)(smem + L::kBarOff);
    uint64_t* q_full = bars;                          // 2 *
    uint64_t* q_empty = q_full + 2;                   // 2
    uint64_t* kv_full = q_empty + 2;                  // kStages *
    uint64_t* kv_empty = kv_full + kStages;           // kStages: everything that reads a stage is done
    uint64_t* s_full = kv_empty + kStages;            // kBufs: S of a tile is there
    uint64_t* p_full = s_full + kBufs;                // kBufs *, one arrival per warp of the tile's warpgroup
    uint64_t* o_full = p_full + kBufs;                // 1
    uint64_t* o_empty = o_full + 1;                   // 1 *, one arrival per epilogue warp
    uint64_t* m_full = o_empty + 1;                   // kSlots, one arrival per warp of the first tile's warpgroup
    uint64_t* l_full = m_full + kSlots;               // kSlots, one arrival per softmax warp
    uint32_t* tmem_slot = (uint32_t*)(l_full + kSlots);
    __shared__ int abort_flag_s;
    __shared__ int ticket_s;
    __shared__ unsigned long long redo_s;             // passes of the round in which a row sum was huge in this CTA
    __shared__ unsigned long long redo_peer_s;        // the same of the pair's other CTA, written by it
    constexpr int kCuCopy = 64;
    __shared__ int32_t cu_s[kCuCopy], len_s[kCuCopy];
    volatile int* abort_flag = &abort_flag_s;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = kPair ? cluster_ctarank() : 0u;
    const int me = kPair ? blockIdx.x >> 1 : blockIdx.x, stride = kPair ? gridDim.x >> 1 : gridDim.x;

    if (threadIdx.x == 0) {
        abort_flag_s = 0;
        redo_s = 0;
        for (int i = 0; i < 2; ++i) { mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1); }
        for (int i = 0; i < kStages; ++i) { mbar_init(&kv_full[i], 1); mbar_init(&kv_empty[i], 1); }
        for (int i = 0; i < kBufs; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 4 * L::kCtas); }
        mbar_init(o_full, 1);
        mbar_init(o_empty, 4 * L::kCtas);
        for (int i = 0; i < kSlots; ++i) { mbar_init(&m_full[i], 4); mbar_init(&l_full[i], 8); }
        fence_barrier_init();
        prefetch_tmap(&tmap_q);
        prefetch_tmap(&tmap_k);
        prefetch_tmap(&tmap_v);
    }
    if (warp == 1) {
        if constexpr (kPair) tmem_alloc_pair(tmem_slot, kTmemCols);
        else tmem_alloc(tmem_slot, kTmemCols);
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (kPair) cluster_sync_all();         // both CTAs' barriers exist before either signals the other
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    // The passes of a CTA are laid out in shared memory, kTable at a time.
    Pass* table = (Pass*)(smem + L::kTabOff);
    static_assert(kTable * sizeof(Pass) <= 64 * 44, "pass table");
    const bool copy = p.B < kCuCopy;
    auto lay_out = [&](int base) {
        if (base == 0 && copy) {
            if (threadIdx.x <= p.B) cu_s[threadIdx.x] = p.cu_keep[threadIdx.x];
            else if (threadIdx.x >= 128 && threadIdx.x < 128 + p.B) len_s[threadIdx.x - 128] = p.kv_len[threadIdx.x - 128];
        }
        __syncthreads();
        if (threadIdx.x < kTable) table[threadIdx.x] = make_pass<DH>(p, copy ? cu_s : p.cu_keep, copy ? len_s : p.kv_len, me + (base + threadIdx.x) * stride);
        if (threadIdx.x == 0) redo_s = 0;
        __syncthreads();
    };
    // The first of them before the wait. What it reads, kept counts and cache lengths, was complete before the GEMM ahead of
    // this launch (or ahead of the query/key transform) passed its own wait, and that GEMM has let this launch in only after
    // it. Laid out behind the wait it was 1.5 us of each launch: 20x20 scale of one image, 32 layers, 2622 -> 2590 us, 16-layer
    // 256x256 generation 8713 -> 8645, 512x512 scale 8796 -> 8744.
    lay_out(0);
    pdl_wait();

    auto commit = [&](uint64_t* bar) {
        if constexpr (kPair) mma_commit_pair(bar, 3);
        else mma_commit(bar);
    };
    // arrival of one warp at a barrier of the leader
    auto arrive_leader = [&](uint64_t* bar) {
        if (kPair && rank != 0) mbar_arrive_cluster(map_to_cta(smem_u32(bar), 0));
        else mbar_arrive(bar);
    };
    // Rounds: up to kTable passes, then, if a row sum in any of them was huge (in either CTA of the pair), those
    // passes once more with a maximum pass before each; then the next kTable. begin_round lays out the table if
    // there are passes left; end_of_round gives the passes to run again.
    auto begin_round = [&](int base) -> bool {
        if (base == 0) return true;
        if (table[kTable - 1].over) return false;
        lay_out(base);
        return true;
    };
    auto end_of_round = [&]() -> unsigned long long {
        __syncwarp();
        __syncthreads();
        unsigned long long mask = *(volatile unsigned long long*)&redo_s;
        if constexpr (kPair) {
            if (threadIdx.x == 0)
                asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(map_to_cta(smem_u32(&redo_peer_s), rank ^ 1u)), "l"(mask) : "memory");
            __syncwarp();
            cluster_sync_all();
            mask |= *(volatile unsigned long long*)&redo_peer_s;
        }
        return mask;
    };
    // next pass to run from index i on (of those in `only`, if that is not 0), kTable if none is left
    auto next_pass = [&](int i, unsigned long long only) -> int {
        for (; i < kTable; ++i) {
            if (table[i].over) return kTable;
            if (table[i].n > 0 && (!only || ((only >> i) & 1ull))) break;
        }
        return i;
    };

    if (warp < 4) {
        int st = 0, qb = 0;                            // ring positions
        uint32_t spar = 0, qpar = 0;                   // and their phase parities
        int units = 0, qcount = 0;                     // loaded so far (producer)
        int sbuf = 0, pbuf = 0;                        // S buffer of the next S, of the next P (issuer)
        uint32_t ppar = 0, opar = 1;
        bool o_used = false;
        for (int base = 0; begin_round(base); base += kTable) {
            unsigned long long only = 0;
            do {
                // S runs kBufs tiles ahead of O += P V, across the passes: two cursors over the table
                int si = next_pass(0, only), s_n = si < kTable ? table[si].n : 0, s_left = s_n, s_passes = only ? 2 : 1;
                auto s_step = [&]() -> bool {          // past one S tile; true at the end of a pass
                    if (--s_left) return false;
                    if (--s_passes == 0) {
                        si = next_pass(si + 1, only);
                        s_passes = only ? 2 : 1;
                    }
                    s_n = s_left = si < kTable ? table[si].n : 0;
                    return true;
                };
                if (warp == 0) {
                    if (elect_one()) {
                        bool ok = true;
                        // one stage: V of tile vj of pass vi (vi < 0: none) and K of the next S tile, if there is one
                        auto load_stage = [&](int vi, int vj) {
                            if (s_left == 0 && vi < 0) return;
                            // (the stage's last use is waited for by its own barrier, which cannot complete twice
                            // before the next fill; S's barriers go on without the producer and could)
                            if (units >= kStages && !mbar_wait(&kv_empty[st], spar ^ 1u, abort_flag, p.status)) { ok = false; return; }
                            const bool has_k = s_left > 0;
                            if (has_k && s_left == s_n) {
                                if (qcount >= 2 && !mbar_wait(&q_empty[qb], qpar ^ 1u, abort_flag, p.status)) { ok = false; return; }
                                if (rank == 0) mbar_arrive_expect_tx(&q_full[qb], L::kCtas * L::kQBytes);
#pragma unroll
                                for (int sl = 0; sl < DH / 64; ++sl) {
                                    uint8_t* dst = smem + qb * L::kQBytes + sl * kSlabBytes;
                                    const int row = table[si].q_begin + (int)rank * BQ;
                                    if constexpr (kPair) tma_load_2d_pair(dst, &tmap_q, map_to_cta(smem_u32(&q_full[qb]), 0), table[si].x + sl * 64, row);
                                    else tma_load_2d(dst, &tmap_q, &q_full[qb], table[si].x + sl * 64, row);
                                }
                                ++qcount;
                                if (++qb == 2) { qb = 0; qpar ^= 1u; }
                            }
                            uint8_t* dst = smem + L::kStageOff + st * 2 * L::kTileBytes;
                            if (rank == 0)
                                mbar_arrive_expect_tx(&kv_full[st], (uint32_t)((has_k ? L::kCtas * L::kTileBytes : 0) + (vi >= 0 ? L::kCtas * L::kTileBytes : 0)));
                            const uint32_t bar = kPair ? map_to_cta(smem_u32(&kv_full[st]), 0) : 0u;
                            if (vi >= 0) {
                                const int y = vj == table[vi].n - 1 ? table[vi].last : table[vi].first + vj * BKV;
                                if constexpr (kPair) tma_load_3d_pair(dst + L::kTileBytes, &tmap_v, bar, table[vi].x + (int)rank * L::kVCols, y, table[vi].b);
                                else tma_load_3d(dst + L::kTileBytes, &tmap_v, &kv_full[st], table[vi].x, y, table[vi].b);
                            }
                            if (has_k) {
                                const int j = s_n - s_left;
                                const int y = (s_left == 1 ? table[si].last : table[si].first + j * BKV) + (int)rank * L::kKRows;
#pragma unroll
                                for (int sl = 0; sl < DH / 64; ++sl) {
                                    if constexpr (kPair) tma_load_3d_pair(dst + sl * L::kKRows * 128, &tmap_k, bar, table[si].x + sl * 64, y, table[si].b);
                                    else tma_load_3d(dst + sl * L::kKRows * 128, &tmap_k, &kv_full[st], table[si].x + sl * 64, y, table[si].b);
                                }
                                s_step();
                            }
                            ++units;
                            if (++st == kStages) { st = 0; spar ^= 1u; }
                        };
                        for (int i = 0; i < kBufs && ok; ++i) load_stage(-1, 0);
                        for (int i = next_pass(0, only); i < kTable && ok; i = next_pass(i + 1, only)) {
                            const int n = table[i].n;
                            for (int pass = only ? 0 : 1; pass < 2; ++pass)        // 0: maximum pass (K only)
                                for (int j = 0; j < n && ok; ++j) load_stage(pass ? i : -1, j);
                        }
                        // A round ends with every copy landed and every use of a stage or of Q done.
                        for (int i = max(0, units - kStages); i < units && ok; ++i)
                            ok = mbar_wait(&kv_empty[i % kStages], (uint32_t)(i / kStages) & 1u, abort_flag, p.status);
                        for (int i = max(0, qcount - 2); i < qcount && ok; ++i)
                            ok = mbar_wait(&q_empty[i & 1], (uint32_t)(i >> 1) & 1u, abort_flag, p.status);
                        if (!ok || *abort_flag) {       // what is in flight gets some time to finish before memory is released
                            if (rank == 0) {
                                for (int i = max(0, qcount - 2); i < qcount; ++i) mbar_drain(&q_full[i & 1], (uint32_t)(i >> 1) & 1u);
                                for (int i = max(0, units - kStages); i < units; ++i) mbar_drain(&kv_full[i % kStages], (uint32_t)(i / kStages) & 1u);
                            }
                            for (int i = max(0, units - kStages); i < units; ++i) mbar_drain(&kv_empty[i % kStages], (uint32_t)(i / kStages) & 1u);
                        }
                    }
                } else if (warp == 1) {
                    if (rank == 0 && elect_one()) {
                        constexpr uint32_t idesc_s = idesc_bf16_f32(L::kRows, BKV, 0);
                        constexpr uint32_t idesc_o = idesc_bf16_f32(L::kRows, DH, 1);
                        // Shared-memory descriptors: (address >> 4) sits in the low 14 bits, so stepping through
                        // a tile or to another stage is an integer add.
                        const uint64_t q_desc = smem_desc_sw128(smem_u32(smem), 16, 1024);
                        const uint64_t k_desc = smem_desc_sw128(smem_u32(smem + L::kStageOff), 16, 1024);
                        const uint64_t v_desc = smem_desc_sw128(smem_u32(smem + L::kStageOff + L::kTileBytes), kSlabBytes, 1024);
                        bool ok = true, new_q = true;
                        // S of the next tile, whichever pass it belongs to, with K in stage `from`.
                        auto issue_s = [&](int from) {
                            if (new_q) {
                                ok = mbar_wait(&q_full[qb], qpar, abort_flag, p.status);
                                if (!ok) return;
                                tc_fence_after();
                            }
                            const uint64_t qd = q_desc + (uint32_t)(qb * (L::kQBytes >> 4));
                            const uint64_t kd = k_desc + (uint32_t)(from * (2 * L::kTileBytes >> 4));
                            const uint32_t s_tmem = tmem_base + 128u + BKV * (uint32_t)sbuf;
#pragma unroll
                            for (int kk = 0; kk < DH / 16; ++kk) {
                                const uint32_t qo = (kk >> 2) * (kSlabBytes >> 4) + (kk & 3) * 2;         // 32 bytes per 16 k
                                const uint32_t ko = (kk >> 2) * (L::kKRows * 128 >> 4) + (kk & 3) * 2;
                                if constexpr (kPair) mma_bf16_ss_pair(s_tmem, qd + qo, kd + ko, idesc_s, kk ? 1u : 0u);
                                else mma_bf16_ss(s_tmem, qd + qo, kd + ko, idesc_s, kk ? 1u : 0u);
                            }
                            commit(&s_full[sbuf]);
                            if (++sbuf == kBufs) sbuf = 0;
                            new_q = s_step();
                            if (new_q) {
                                commit(&q_empty[qb]);
                                if (++qb == 2) { qb = 0; qpar ^= 1u; }
                            }
                        };
                        auto take_stage = [&]() -> int {
                            ok = mbar_wait(&kv_full[st], spar, abort_flag, p.status);
                            tc_fence_after();
                            const int at = st;
                            if (++st == kStages) { st = 0; spar ^= 1u; }
                            return at;
                        };
                        for (int i = 0; i < kBufs && ok && s_left; ++i) {
                            const int at = take_stage();
                            if (!ok) break;
                            issue_s(at);
                            commit(&kv_empty[at]);
                        }
                        for (int i = next_pass(0, only); i < kTable && ok; i = next_pass(i + 1, only)) {
                            const int n = table[i].n;
                            for (int pass = only ? 0 : 1; pass < 2 && ok; ++pass) {
                                for (int j = 0; j < n && ok; ++j) {
                                    int at = -1;
                                    if (pass || s_left) at = take_stage();
                                    if (ok && pass && j == 0) {
                                        if (o_used) ok = mbar_wait(o_empty, opar, abort_flag, p.status);
                                        o_used = true;
                                        opar ^= 1u;
                                    }
                                    if (ok) ok = mbar_wait(&p_full[pbuf], ppar, abort_flag, p.status);
                                    if (!ok) break;
                                    tc_fence_after();
                                    if (pass) {
                                        const uint64_t vd = v_desc + (uint32_t)(at * (2 * L::kTileBytes >> 4));
                                        const uint32_t p_tmem = tmem_base + 128u + BKV * (uint32_t)pbuf;
#pragma unroll
                                        for (int kk = 0; kk < BKV / 16; ++kk) {
                                            const uint32_t acc = kk ? 1u : (j ? 1u : 0u);
                                            if constexpr (kPair) mma_bf16_ts_pair(tmem_base, p_tmem + kk * 8, vd + (uint32_t)(kk * 128), idesc_o, acc);
                                            else mma_bf16_ts(tmem_base, p_tmem + kk * 8, vd + (uint32_t)(kk * 128), idesc_o, acc);
                                        }
                                        if (j == n - 1) commit(o_full);
                                    }
                                    if (++pbuf == kBufs) { pbuf = 0; ppar ^= 1u; }
                                    if (s_left) issue_s(at);
                                    if (at >= 0) commit(&kv_empty[at]);
                                }
                            }
                        }
                    }
                }
                const unsigned long long again = end_of_round();
                if (only || !again) break;
                only = again;
            } while (true);
        }
    } else if (warp < 8) {
        // ---- epilogue -------------------------------------------------------------------------------
        const int q = warp & 3, row = q * 32 + lane;              // row within the CTA's 128 = tensor-memory lane
        const int grow = (int)rank * BQ + row;                    // row within the work item
        const uint32_t o_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        const float* l_s = (const float*)(smem + L::kLOff);
        const float* m_s = (const float*)(smem + L::kMOff);
        int np = 0;                                               // passes with an O so far
        for (int base = 0; begin_round(base); base += kTable) {
            unsigned long long only = 0;
            for (int i = 0; i < kTable && !table[i].over; ++i)
                if (table[i].empty && grow < table[i].rows_valid) {
                    // nothing to attend to: the output rows are zero
                    __nv_bfloat16* dst_row = p.o + (long)(table[i].q_begin + grow) * p.C + table[i].x;
                    for (int v = 0; v < DH / 8; ++v) *(uint4*)(dst_row + v * 8) = make_uint4(0, 0, 0, 0);
                }
            do {
                for (int i = next_pass(0, only); i < kTable; i = next_pass(i + 1, only), ++np) {
                    const int half = table[i].half, rows_valid = table[i].rows_valid;
                    __nv_bfloat16* dst_row = p.o + (long)(table[i].q_begin + grow) * p.C + table[i].x;
                    const int slot = np % kSlots;
                    // (after a failed wait everybody goes on with garbage to the end: the status word says so)
                    bool ok = mbar_wait_warp(&l_full[slot], (uint32_t)(np / kSlots) & 1u, abort_flag, p.status);
                    const float l_run = l_s[(slot * 2 + 0) * BQ + row] + l_s[(slot * 2 + 1) * BQ + row];
                    const float m_ref = m_s[slot * BQ + row];
                    // The first time, a pass that will be run again is left alone; the second time, one that
                    // only the other CTA of the pair asked for.
                    const bool huge = (*(volatile unsigned long long*)&redo_s >> i) & 1ull;
                    const bool act = only ? huge : !huge;
                    ok = mbar_wait_warp(o_full, (uint32_t)np & 1u, abort_flag, p.status) && ok;
                    tc_fence_after();
                    // The next kernel is let in at the last pass. A trigger at the start puts its first CTAs on the SMs
                    // this grid leaves free, long before the others find room, and it ends later for it: a 16-layer
                    // 256x256 generation took 9750 us with the trigger at the start, 9600 after the table, 9667 at
                    // the end, 9518 to 9534 here or at the first pass.
                    if (next_pass(i + 1, only) == kTable) pdl_launch_dependents();
                    if (act && half < 0) {
                        const float inv = 1.f / l_run;
#pragma unroll 1
                        for (int cch = 0; cch < DH / 32; ++cch) {
                            uint32_t ov[32];
                            tmem_ld32(o_addr + cch * 32, ov);
                            tmem_ld_wait();
                            if (ok && grow < rows_valid) {
                                uint4* dst = (uint4*)(dst_row + cch * 32);
#pragma unroll
                                for (int g = 0; g < 4; ++g)
                                    dst[g] = make_uint4(
                                        pack_bf16(__uint_as_float(ov[g * 8]) * inv, __uint_as_float(ov[g * 8 + 1]) * inv),
                                        pack_bf16(__uint_as_float(ov[g * 8 + 2]) * inv, __uint_as_float(ov[g * 8 + 3]) * inv),
                                        pack_bf16(__uint_as_float(ov[g * 8 + 4]) * inv, __uint_as_float(ov[g * 8 + 5]) * inv),
                                        pack_bf16(__uint_as_float(ov[g * 8 + 6]) * inv, __uint_as_float(ov[g * 8 + 7]) * inv));
                            }
                        }
                    } else if (act) {
                        const int khalf = half & 1, tail_slot = half >> 1;
                        const float c = p.scale_log2e;
                        // ---- half of the keys: publish the partial result, then merge if the other is there. The two
                        // CTAs of a pair do so independently, each for its rows.
                        // [DH columns, then reference and sum][rows]: a warp's accesses are 128 contiguous bytes
                        float* mine = p.part + (size_t)(tail_slot * 2 + khalf) * (DH + 4) * L::kRows + grow;
                        const float* other = p.part + (size_t)(tail_slot * 2 + (khalf ^ 1)) * (DH + 4) * L::kRows + grow;
                        unsigned int* ticket = p.tickets + tail_slot * L::kCtas + rank;
#pragma unroll 1
                        for (int cch = 0; cch < DH / 32; ++cch) {
                            uint32_t ov[32];
                            tmem_ld32(o_addr + cch * 32, ov);
                            tmem_ld_wait();
#pragma unroll
                            for (int g = 0; g < 32; ++g) mine[(cch * 32 + g) * L::kRows] = __uint_as_float(ov[g]);
                        }
                        mine[DH * L::kRows] = m_ref;
                        mine[(DH + 1) * L::kRows] = l_run;
                        __threadfence();
                        asm volatile("bar.sync 1, 128;" ::: "memory");
                        if (threadIdx.x == 128) {
                            const unsigned int t = atomicAdd(ticket, 1u);
                            if (t == 1u) *ticket = 0;          // ready for the next launch
                            ticket_s = (int)t;
                        }
                        asm volatile("bar.sync 1, 128;" ::: "memory");
                        if (ok && ticket_s == 1) {
                            // the other fenced its partial result before it drew ticket 0
                            // The merge is written in terms of (half 0, half 1), not (mine, other), with every
                            // rounding spelled out: either may be the one that merges, and the output must
                            // not depend on which.
                            const float m_o = __ldcg(other + DH * L::kRows), l_o = __ldcg(other + (DH + 1) * L::kRows);
                            const float m_new = fmaxf(m_ref, m_o);
                            const float a_me = ex2((m_ref - m_new) * c), a_o = ex2((m_o - m_new) * c);
                            const bool first = (khalf == 0);
                            const float a0 = first ? a_me : a_o, a1 = first ? a_o : a_me;
                            const float l0 = first ? l_run : l_o, l1 = first ? l_o : l_run;
                            const float inv = 1.f / __fmaf_rn(l0, a0, __fmul_rn(l1, a1));
                            const float w0 = a0 * inv, w1 = a1 * inv;
                            const float w_me = first ? w0 : w1, w_o = first ? w1 : w0;
                            auto mix = [&](uint32_t mine_bits, float theirs) {
                                const float v = __uint_as_float(mine_bits);
                                // half 0's term is the multiply-add operand, half 1's the rounded product
                                return first ? __fmaf_rn(v, w_me, __fmul_rn(theirs, w_o))
                                             : __fmaf_rn(theirs, w_o, __fmul_rn(v, w_me));
                            };
#pragma unroll 1
                            for (int cch = 0; cch < DH / 32; ++cch) {
                                uint32_t ov[32];
                                tmem_ld32(o_addr + cch * 32, ov);
                                tmem_ld_wait();
                                float th[32];
#pragma unroll
                                for (int g = 0; g < 32; ++g) th[g] = __ldcg(other + (cch * 32 + g) * L::kRows);
                                if (grow < rows_valid) {
                                    uint4* dst = (uint4*)(dst_row + cch * 32);
#pragma unroll
                                    for (int g = 0; g < 4; ++g)
                                        dst[g] = make_uint4(
                                            pack_bf16(mix(ov[g * 8], th[g * 8]), mix(ov[g * 8 + 1], th[g * 8 + 1])),
                                            pack_bf16(mix(ov[g * 8 + 2], th[g * 8 + 2]), mix(ov[g * 8 + 3], th[g * 8 + 3])),
                                            pack_bf16(mix(ov[g * 8 + 4], th[g * 8 + 4]), mix(ov[g * 8 + 5], th[g * 8 + 5])),
                                            pack_bf16(mix(ov[g * 8 + 6], th[g * 8 + 6]), mix(ov[g * 8 + 7], th[g * 8 + 7])));
                                }
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_leader(o_empty);
                }
                const unsigned long long again = end_of_round();
                if (only || !again) break;
                only = again;
            } while (true);
        }
    } else {
        // ---- softmax ------------------------------------------------------------------------------------
        const int wg = (warp - 8) >> 2, q = warp & 3, row = q * 32 + lane;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        const float c = p.scale_log2e;
        float* l_s = (float*)(smem + L::kLOff) + wg * BQ + row;
        float* m_s = (float*)(smem + L::kMOff) + row;
        float* a_s = (float*)(smem + L::kAOff) + row;
        // Polynomial share of the exponentials (pairs out of every four pairs of scores). The
        // special-function unit delivers one exponential per 8 clocks and scheduler; the polynomial
        // costs a scheduler about as much in issue slots, so it does not replace that unit, it only
        // works beside it: a quarter of the scores on the polynomial measured best at both head sizes
        // (6.9 clocks per score and scheduler against 7.5 at a half and 8.2 with none).
        constexpr int kPolyPairs = 1;
        int np = 0;                            // ordinary passes so far
        int mine = wg;                         // tiles until this warpgroup's next one
        int buf = wg;                          // S buffer of that tile: every other one, of three
        uint32_t par = 0;                      // and its phase parity
        for (int base = 0; begin_round(base); base += kTable) {
            unsigned long long only = 0;
            do {
            for (int i = next_pass(0, only); i < kTable; i = next_pass(i + 1, only)) {
            const int n = table[i].n, masked = table[i].masked;
            float m_true = -1e30f;             // the row's maximum over all keys, from a maximum pass
            for (int pass = only ? 0 : 1; pass < 2; ++pass) {
                const int slot = np % kSlots;
                // The reference maximum starts at a finite floor, not -inf: (-inf) - (-inf) must not appear.
                float m_ref = -1e30f, l_run = 0.f, m_run = -1e30f;
                bool huge = false;
                // tiles alternate between the warpgroups, also across passes
                int j = mine;
                for (; j < n; j += 2) {
                    const uint32_t s_addr = tmem_base + lane_off + 128u + BKV * (uint32_t)buf;
                    mbar_wait_warp(&s_full[buf], par, abort_flag, p.status);
                    tc_fence_after();
                    uint64_t* done = &p_full[buf];
                    if (buf == 0) buf = 2;                       // two tiles on
                    else { --buf; par ^= 1u; }
                    // The row is taken 32 scores at a time, in loops that are not unrolled: the code of a whole
                    // row is 16 KB, and fetching it costs a launch's first tile 6 us. The latency of the
                    // tensor-memory reads hides behind the other warpgroup.
                    const int skip = j == n - 1 ? masked : 0;       // columns that do not count
                    auto load = [&](int ch, uint32_t (&sv)[32]) {
                        tmem_ld32(s_addr + ch * 32, sv);
                        tmem_ld_wait();
                        if (skip > ch * 32) {
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                if (ch * 32 + e < skip) sv[e] = 0xff800000u;   // -inf: a key of the tile before, or none
                        }
                    };
                    if (pass == 0 || (j == 0 && !only)) {
                        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
                        for (int ch = skip >> 5; ch < 4; ++ch) {
                            uint32_t sv[32];
                            load(ch, sv);
#pragma unroll
                            for (int e = 0; e < 32; e += 2) mx[(e >> 1) & 3] = fmax3(mx[(e >> 1) & 3], __uint_as_float(sv[e]), __uint_as_float(sv[e + 1]));
                        }
                        m_run = fmaxf(m_run, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])));
                    }
                    if (pass == 0) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) arrive_leader(done);
                        continue;
                    }
                    if (j == 0) {
                        // the row's reference, for both warpgroups and the epilogue
                        m_ref = only ? m_true : m_run;
                        m_s[slot * BQ] = m_ref;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&m_full[slot]);
                    } else if (j == 1) {
                        mbar_wait_warp(&m_full[slot], (uint32_t)(np / kSlots) & 1u, abort_flag, p.status);
                        m_ref = m_s[slot * BQ];
                    }
                    // p = 2^(s*c - m*c - kHeadroom): 16 registers of bf16 pairs per chunk, written over columns of S that have
                    // been read
                    const uint64_t c2 = pack_f32x2(c, c);
                    const uint64_t nm2 = pack_f32x2(fmaf(-m_ref, c, -kHeadroom), fmaf(-m_ref, c, -kHeadroom));
                    uint64_t lsum_a = pack_f32x2(0.f, 0.f), lsum_b = lsum_a;
                    // (chunks of which no column counts take zeros and no arithmetic: three of four in the smallest calls,
                    // 7.1 -> 6.3 us for eight images with one kept token each)
                    int ch = 0;
#pragma unroll 1
                    for (; (ch + 1) * 32 <= skip; ++ch) {
                        uint32_t zero[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) zero[e] = 0u;
                        tmem_st16(s_addr + ch * 16, zero);
                    }
#pragma unroll 1
                    for (; ch < 4; ++ch) {
                        uint32_t sv[32], pk[16];
                        load(ch, sv);
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int i = 8 * g + 2 * e;
                                const uint64_t y = fma_f32x2(pack_f32x2(__uint_as_float(sv[i]), __uint_as_float(sv[i + 1])), c2, nm2);
                                float p0, p1;
                                if (e < kPolyPairs) {
                                    exp2_poly_x2(y, p0, p1);
                                } else {
                                    float y0, y1;
                                    unpack_f32x2(y, y0, y1);
                                    p0 = ex2(y0);
                                    p1 = ex2(y1);
                                }
                                if (e & 1) lsum_b = add_f32x2(lsum_b, pack_f32x2(p0, p1));
                                else lsum_a = add_f32x2(lsum_a, pack_f32x2(p0, p1));
                                pk[4 * g + e] = pack_bf16(p0, p1);
                            }
                        }
                        tmem_st16(s_addr + ch * 16, pk);
                    }
                    float s0, s1, s2, s3;
                    unpack_f32x2(lsum_a, s0, s1);
                    unpack_f32x2(lsum_b, s2, s3);
                    const float lsum = (s0 + s2) + (s1 + s3);
                    huge |= !(lsum < kHugeSum);
                    l_run += lsum;
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_leader(done);
                }
                mine = j - n;
                if (pass == 0) {
                    a_s[wg * BQ] = m_run;
                    asm volatile("bar.sync 2, 256;" ::: "memory");
                    m_true = fmaxf(a_s[0], a_s[BQ]);
                    asm volatile("bar.sync 2, 256;" ::: "memory");
                    continue;
                }
                l_s[slot * 2 * BQ] = l_run;
                // (only rows of this item may ask: those past its last one are the next image's, or whatever the
                // buffer held, and must not decide how the others are rounded)
                huge = huge && (int)rank * BQ + row < table[i].rows_valid;
                if (!only && __any_sync(0xffffffffu, huge) && lane == 0) atomicOr(&redo_s, 1ull << i);
                __syncwarp();
                if (lane == 0) mbar_arrive(&l_full[slot]);
                ++np;
            }
            }
            const unsigned long long again = end_of_round();
            if (only || !again) break;
            only = again;
            } while (true);
        }
    }
    // (the last end_of_round saw everybody's work done: nobody signals this CTA any more)
    tc_fence_before();
    __syncwarp();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        if constexpr (kPair) tmem_dealloc_pair(tmem_base, kTmemCols);
        else tmem_dealloc(tmem_base, kTmemCols);
    }
}

template <int DH>
nova_status launch(nova_ctx* ctx, const nova_attn_args& a, cudaStream_t st)
{
    using L = AttnCfg<DH>;
    CUtensorMap tq, tk, tv;
    const uint64_t dq[2] = {(uint64_t)a.C, (uint64_t)a.M}, sq[1] = {(uint64_t)a.C * 2};
    const uint64_t dk[3] = {(uint64_t)a.C, (uint64_t)a.Lmax, (uint64_t)a.B};
    const uint64_t sk[2] = {(uint64_t)a.C * 2, (uint64_t)a.Lmax * a.C * 2};
    if (!make_tmap_bf16(ctx, &tq, a.q, 2, dq, sq, BQ) || !make_tmap_bf16(ctx, &tk, a.k_cache, 3, dk, sk, L::kKRows) ||
        !make_tmap_bf16(ctx, &tv, a.v_cache, 3, dk, sk, BKV))
        return nova_fail(ctx, NOVA_ERR_CUDA, "attention: cuTensorMapEncodeTiled failed");
    if (!ctx->attr_attn) {   // both head sizes once per context
        NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(attention_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<64>::kTotal));
        NOVA_CUDA_CHECK(ctx, cudaFuncSetAttribute(attention_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<128>::kTotal));
        ctx->attr_attn = true;
    }
    AttnParams p;
    p.cu_keep = a.cu_keep; p.kv_len = a.kv_len; p.o = a.o; p.B = a.B; p.C = a.C; p.Lmax = a.Lmax;
    p.scale_log2e = (float)((1.0 / sqrt((double)DH)) * 1.4426950408889634);
    p.status = ctx->dev_status;
    p.n_heads = a.n_heads; p.slots = ctx->num_sms / L::kCtas;
    p.own_keys = a.cache_only ? 0 : 1;
    // scratch for a key-split last round: [slots][2][kRows][DH + 4] fp32; tickets live in the context's
    // status allocation (zero at creation, reset by the CTA that draws the second ticket)
    const size_t slot_bytes = (size_t)2 * L::kRows * (DH + 4) * sizeof(float);
    const bool can_split = a.scratch && (a.Lmax + BKV - 1) / BKV >= kSplitTiles;
    p.part = can_split ? (float*)a.scratch : nullptr;
    p.part_slots = can_split ? (int)min((size_t)(NOVA_ATTN_TICKETS / L::kCtas), a.scratch_bytes / slot_bytes) : 0;
    p.tickets = ctx->dev_status + NOVA_ATTN_TICKET_WORD0;
    // One CTA (pair) per SM (two), or fewer if there cannot be as much work: upper bound of the work items (the
    // kept counts per image live on the device), each split in two at most.
    const long items = (((long)a.M + (long)a.B * (L::kRows - 1)) / L::kRows) * a.n_heads;
    const int ctas = (int)min((long)p.slots, (can_split ? 2 : 1) * items) * L::kCtas;
    {
        nova_launch_scope scope(ctx, NOVA_K_ATTENTION, st);
        NOVA_CUDA_CHECK(ctx, nova_launch_pdl(attention_kernel<DH>, dim3(ctas), dim3(kThreads), L::kTotal, st, L::kPair ? 2 : 0, tq, tk, tv, p));
    }
    return NOVA_OK;
}

}  // namespace

nova_status nova_launch_attention(nova_ctx* ctx, const nova_attn_args& a, cudaStream_t st)
{
    if (a.M <= 0) return NOVA_OK;
    const int dh = a.C / a.n_heads;
    if (dh == 64) return launch<64>(ctx, a, st);
    if (dh == 128) return launch<128>(ctx, a, st);
    return nova_fail(ctx, NOVA_ERR_SHAPE, "attention: head dimension must be 64 or 128");
}
