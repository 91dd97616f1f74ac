// Eq. 15-16: scatter the layer output back to the full token map, fill the pruned rows from
// the previous scale's residual cache (bilinear resize, half-pixel centres) and write the new
// residual cache.
//
// A row is shared by one or two warps, two 128-bit pieces of each operand per thread and turn, all of them
// loaded before the first store. Work item r < M is kept row r of the compacted output; work item r >= M is entry
// r - M of the pruned index list. Every byte of x_in, y_kept, x_out and cache_out is touched exactly once; cache_prev
// is small and re-read through L2.
// What bounds it: HBM at many rows, the latency of list -> rows -> store at few. With one warp per row and one piece at
// a time each piece waited for the one before it to be stored. Pruned rows alone, back to back over buffers larger than
// L2, us before -> with two warps / with one: 100 rows of 2048 6.8 -> 3.6 / 3.9; 1640 x 1024 6.8 -> 4.8 / 5.0; 1844 x 1920
// 10.5 -> 9.2 / 9.6; 3072 x 2048 12.7 -> 11.2 / 11.3; 4800 x 2048 16.4 -> 16.9 / 17.2; 6144 x 2048 22.5 -> 20.3 / 19.8; 8192 x 2048
// 27.6 -> 27.7 / 27.1; 8192 x 1024 15.3 -> 16.5 / 15.4; 13108 x 2048 38.6 -> 37.4 with one (5.3 TB/s). (Over buffers that fit L2 one piece at a time
// was the faster for 4800 to 8192 rows, 12.4 and 22.5 us against 13.5 and 23.9, with every row in flight at once.)
#include "common.cuh"

namespace {

constexpr int kThreads = 128;
// Up to this many rows two warps share a row, above it one warp has it to itself (fewer index computations).
constexpr long kWideRows = 5000;
constexpr long kRowsBeside = 8;       // rows of a group of threads at most, in a launch that works beside another

__device__ __forceinline__ uint4 ld_stream(const uint4* p)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ void st_cs(uint4* p, uint4 v)
{
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" :: "l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void unpack2(uint32_t w, float& lo, float& hi)
{
    lo = __uint_as_float(w << 16);
    hi = __uint_as_float(w & 0xffff0000u);
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&t);
}

// wait_last: launched behind a kernel whose results it neither reads nor overwrites (see the launch in
// block.cu); it then works beside that one and waits only to end after it.
// PRUNED_ONLY: the kept rows are written by the block's last epilogue; work items start at the first pruned entry.
template <bool PRUNED_ONLY>
__global__ void __launch_bounds__(kThreads, 6)
restore_kernel(const uint4* x_in, const uint4* y_kept, const int32_t* keep_idx, const int32_t* prune_idx,
               const int32_t* cu_keep, const uint4* cache_prev,
               int hp, int wp, int h, int w, int vec_per_row, int row_threads, int B, int M, bool m_on_device, bool wait_last,
               uint4* __restrict__ x_out, uint4* __restrict__ cache_out)
{
    if (!wait_last) {
        pdl_launch_dependents();
        pdl_wait();
    }
    if (m_on_device) M = cu_keep[B];    // the kept count lives on the device
    const int rows_per_block = kThreads / row_threads, sub = threadIdx.x / row_threads, lane = threadIdx.x - sub * row_threads;
    const int N = h * w;
    const long total = (long)B * N;
    const long stride = (long)gridDim.x * rows_per_block;
    long r = (long)blockIdx.x * rows_per_block + sub + (PRUNED_ONLY ? M : 0);
    int i_next = r >= M && r < total ? prune_idx[r - M] : 0;
    for (; r < total; r += stride) {
        const int i = i_next;
        if (PRUNED_ONLY && r + stride < total) i_next = prune_idx[r + stride - M];
        if (!PRUNED_ONLY && r < M) {
            // kept row: find its image (largest b with cu_keep[b] <= r)
            int lo = 0, hi = B;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (cu_keep[mid] <= r) lo = mid; else hi = mid;
            }
            const long row = (long)lo * N + keep_idx[r];
            const uint4* ysrc = y_kept + r * vec_per_row;
            const uint4* xsrc = x_in + row * vec_per_row;
            for (int v0 = lane; v0 < vec_per_row; v0 += 2 * row_threads) {
                uint4 yv[2], xv[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int v = v0 + i * row_threads;
                    if (v < vec_per_row) {
                        yv[i] = ld_stream(ysrc + v);
                        if (cache_out) xv[i] = ld_stream(xsrc + v);
                    }
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int v = v0 + i * row_threads;
                    if (v >= vec_per_row) break;
                    st_cs(x_out + row * vec_per_row + v, yv[i]);
                    if (cache_out) {
                        const uint32_t yw[4] = {yv[i].x, yv[i].y, yv[i].z, yv[i].w}, xw[4] = {xv[i].x, xv[i].y, xv[i].z, xv[i].w};
                        uint32_t o[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            float y0, y1, x0, x1;
                            unpack2(yw[q], y0, y1);
                            unpack2(xw[q], x0, x1);
                            o[q] = pack2(y0 - x0, y1 - x1);
                        }
                        st_cs(cache_out + row * vec_per_row + v, make_uint4(o[0], o[1], o[2], o[3]));
                    }
                }
            }
        } else {
            // pruned row: entry p of the pruned list; image b has its entries at [b*N - cu_keep[b], ...)
            const long p = r - M;
            int lo = 0, hi = B;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if ((long)mid * N - cu_keep[mid] <= p) lo = mid; else hi = mid;
            }
            const int b = lo;
            const int oy = i / w, ox = i - oy * w;
            float sy = ((float)oy + 0.5f) * ((float)hp / (float)h) - 0.5f;
            float sx = ((float)ox + 0.5f) * ((float)wp / (float)w) - 0.5f;
            sy = fmaxf(sy, 0.f);
            sx = fmaxf(sx, 0.f);
            int y0 = min((int)sy, hp - 1), x0 = min((int)sx, wp - 1);
            const int y1 = min(y0 + 1, hp - 1), x1 = min(x0 + 1, wp - 1);
            const float fy = sy - (float)y0, fx = sx - (float)x0;
            const float w00 = (1.f - fy) * (1.f - fx), w01 = (1.f - fy) * fx, w10 = fy * (1.f - fx), w11 = fy * fx;
            const uint4* c_y0 = cache_prev + (((long)b * hp + y0) * wp + x0) * vec_per_row;      // (64-bit: a cache may be large)
            const uint4* c_y1 = cache_prev + (((long)b * hp + y1) * wp + x0) * vec_per_row;
            const int right = (x1 - x0) * vec_per_row;
            const long row = ((long)b * N + i) * vec_per_row;
            for (int v0 = lane; v0 < vec_per_row; v0 += 2 * row_threads) {
                uint4 xv[2], c[2][4];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int v = v0 + k * row_threads;
                    if (v < vec_per_row) {
                        xv[k] = ld_stream(x_in + row + v);
                        c[k][0] = c_y0[v]; c[k][1] = c_y0[v + right]; c[k][2] = c_y1[v]; c[k][3] = c_y1[v + right];
                    }
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int v = v0 + k * row_threads;
                    if (v >= vec_per_row) break;
                    const uint32_t xw[4] = {xv[k].x, xv[k].y, xv[k].z, xv[k].w};
                    const uint32_t aw[4] = {c[k][0].x, c[k][0].y, c[k][0].z, c[k][0].w}, bw[4] = {c[k][1].x, c[k][1].y, c[k][1].z, c[k][1].w};
                    const uint32_t cw[4] = {c[k][2].x, c[k][2].y, c[k][2].z, c[k][2].w}, dw[4] = {c[k][3].x, c[k][3].y, c[k][3].z, c[k][3].w};
                    uint32_t o[4], u[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float xl, xh, al, ah, bl, bh, cl, ch, dl, dh;
                        unpack2(xw[q], xl, xh);
                        unpack2(aw[q], al, ah);
                        unpack2(bw[q], bl, bh);
                        unpack2(cw[q], cl, ch);
                        unpack2(dw[q], dl, dh);
                        const float ul = w00 * al + w01 * bl + w10 * cl + w11 * dl;
                        const float uh = w00 * ah + w01 * bh + w10 * ch + w11 * dh;
                        u[q] = pack2(ul, uh);
                        o[q] = pack2(xl + ul, xh + uh);
                    }
                    st_cs(x_out + row + v, make_uint4(o[0], o[1], o[2], o[3]));
                    if (cache_out) st_cs(cache_out + row + v, make_uint4(u[0], u[1], u[2], u[3]));
                }
            }
        }
        if (!PRUNED_ONLY) break;        // (launched with a group of threads for every row)
    }
    if (wait_last) {
        pdl_launch_dependents();
        pdl_wait();
    }
}

}  // namespace

static nova_status restore(nova_ctx* ctx, const void* x_in, const void* y_kept,
                           const int32_t* keep_idx, const int32_t* prune_idx,
                           const int32_t* cu_keep, const void* cache_prev,
                           int hp, int wp, int h, int w, int C, int B, int M, bool m_on_device,
                           void* x_out, void* cache_out, void* stream, bool pruned_only = false, bool wait_last = false)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (B < 0 || h < 0 || w < 0 || C < 1 || M < 0 || (long)M > (long)B * h * w)
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_restore_from_cache: bad sizes");
    const long total = (long)B * h * w;
    if (total == 0) return NOVA_OK;
    if (C % 8) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_restore_from_cache: C must be a multiple of 8");
    if (!x_in || !x_out || !cu_keep || (M > 0 && !pruned_only && (!y_kept || !keep_idx)))
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_restore_from_cache: null pointer");
    if ((M < total || m_on_device) && (!prune_idx || !cache_prev || hp < 1 || wp < 1))
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_restore_from_cache: pruned rows need prune_idx and cache_prev");
    if (x_out == x_in) return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_restore_from_cache: x_out aliases x_in");
    if (!nova_aligned16(x_in) || !nova_aligned16(x_out) || !nova_aligned16(y_kept) ||
        !nova_aligned16(cache_prev) || !nova_aligned16(cache_out))
        return nova_fail(ctx, NOVA_ERR_ALIGNMENT, "nova_restore_from_cache: tensors must be 16-byte aligned");
    NOVA_DEVICE_GUARD(ctx, "nova_restore_from_cache");
    {
        // pruned_only: the kept list is not read (and may be null)
        const nova_status chk = nova_debug_check_lists(ctx, "nova_restore_from_cache", pruned_only ? nullptr : keep_idx,
                                                       prune_idx, cu_keep, B, h * w, M, !m_on_device, (cudaStream_t)stream);
        if (chk != NOVA_OK) return chk;
    }
    // rows this launch may have to visit: all of them, or only the pruned ones (when the host knows M)
    const long items = (pruned_only && !m_on_device) ? total - M : total;
    if (items == 0) return NOVA_OK;
    const int row_threads = items > kWideRows ? 32 : 64;
    const int rows_per_block = kThreads / row_threads;
    long blocks = (items + rows_per_block - 1) / rows_per_block;
    // Beside another kernel one block per SM finds room: as many rows per block as that takes, up to kRowsBeside.
    // (Not as many blocks as run at once: by themselves 8192 rows take 31 us that way instead of 33, but the next layer's first kernel
    // starts as blocks end, and a scale of 32 layers with 13107 pruned rows each took 33.2 ms instead of 33.0.)
    if (pruned_only && wait_last) blocks = max((blocks + kRowsBeside - 1) / kRowsBeside, min(blocks, (long)ctx->num_sms));
    nova_launch_scope scope(ctx, NOVA_K_RESTORE, (cudaStream_t)stream);
    NOVA_CUDA_CHECK(ctx, nova_launch_pdl(
        pruned_only ? restore_kernel<true> : restore_kernel<false>, dim3((unsigned)blocks), dim3(kThreads), 0, (cudaStream_t)stream, 0, (const uint4*)x_in, (const uint4*)y_kept, keep_idx, prune_idx, cu_keep, (const uint4*)cache_prev,
        hp, wp, h, w, C / 8, row_threads, B, M, m_on_device, wait_last, (uint4*)x_out, (uint4*)cache_out));
    return NOVA_OK;
}

extern "C" nova_status nova_restore_from_cache(nova_ctx* ctx, const void* x_in, const void* y_kept,
                                               const int32_t* keep_idx, const int32_t* prune_idx,
                                               const int32_t* cu_keep, const void* cache_prev,
                                               int hp, int wp, int h, int w, int C, int B, int M,
                                               void* x_out, void* cache_out, void* stream)
{
    return restore(ctx, x_in, y_kept, keep_idx, prune_idx, cu_keep, cache_prev, hp, wp, h, w, C, B, M, false,
                   x_out, cache_out, stream);
}

extern "C" nova_status nova_restore_from_cache_device(nova_ctx* ctx, const void* x_in, const void* y_kept,
                                                      const int32_t* keep_idx, const int32_t* prune_idx,
                                                      const int32_t* cu_keep, const void* cache_prev,
                                                      int hp, int wp, int h, int w, int C, int B,
                                                      void* x_out, void* cache_out, void* stream)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    const long total = (long)B * h * w;
    if (total > 0x7fffffffL) return nova_fail(ctx, NOVA_ERR_SHAPE, "nova_restore_from_cache_device: too many rows");
    return restore(ctx, x_in, y_kept, keep_idx, prune_idx, cu_keep, cache_prev, hp, wp, h, w, C, B, (int)total, true,
                   x_out, cache_out, stream);
}


// Eq. 16 for the pruned rows only: used by nova_pruned_layer_forward, whose last GEMM epilogue writes the
// kept rows of x_out and cache_out. With wait_last the kernel starts before the launch before it has ended.
nova_status nova_restore_pruned_rows(nova_ctx* ctx, const void* x_in, const int32_t* prune_idx,
                                     const int32_t* cu_keep, const void* cache_prev,
                                     int hp, int wp, int h, int w, int C, int B, int M, bool m_on_device,
                                     void* x_out, void* cache_out, void* stream, bool wait_last)
{
    return restore(ctx, x_in, nullptr, nullptr, prune_idx, cu_keep, cache_prev, hp, wp, h, w, C, B, M, m_on_device,
                   x_out, cache_out, stream, true, wait_last);
}
