// One pruned scale through a range of layers in one call (host code only): the launches of the other
// entry points in the order a decoder needs them, without a return to the caller between two of them.
// A small scale is bound by the host (eight launches of about 2.5 us per layer), so what a binding adds per
// layer - argument marshalling, slices, shapes - is time on the critical path.
#include <climits>
#include <new>

#include "common.cuh"

// Eq. 8-13 for layers 1 .. L on mean_host [L, B]; the counts of layers first + 1 .. L go to keep. Nothing is thrown past
// the C entry point: without host memory for the tables the call fails with a status.
static nova_status scale_keep_counts(nova_ctx* ctx, const nova_sched_params* p, int B, int t, int first, int L, int N,
                                     const float* hbar_scale, const float* mean_host, int32_t* keep)
{
    try {
        std::vector<float> hbar_layer((size_t)B * L);
        for (int j = 0; j < L; ++j)
            for (int b = 0; b < B; ++b) hbar_layer[(size_t)b * L + j] = mean_host[(size_t)j * B + b];
        std::vector<int32_t> t_star(B), act(B), keep_all((size_t)L * B);
        std::vector<double> ratio_scale(B), ratio_layer((size_t)L * B);
        const nova_status rc = nova_keep_ratios_layers(p, B, t, L, N, hbar_scale, hbar_layer.data(), t_star.data(), act.data(),
                                                       ratio_scale.data(), ratio_layer.data(), keep_all.data());
        if (rc != NOVA_OK) return nova_fail(ctx, rc, "nova_pruned_scale_forward: bad schedule parameters");
        memcpy(keep, keep_all.data() + (size_t)first * B, sizeof(int32_t) * B * (size_t)(L - first));
        return NOVA_OK;
    } catch (const std::bad_alloc&) {
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_scale_forward: no host memory for this many layers and images");
    }
}

extern "C" nova_status nova_pruned_scale_forward(nova_ctx* ctx, const nova_scale_layers* sl, const nova_scale_io* io,
                                                 const nova_block_shape* s, const nova_sched_params* p, int t,
                                                 int first, int count, int append_kv, void* stream)
{
    if (!ctx) return NOVA_ERR_INVALID_ARG;
    if (!sl || !io || !s || !p || first < 0 || count < 0 || count > INT_MAX - first || t < 1)
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_scale_forward: null argument or bad range");
    if (!sl->weights || !sl->logits || !sl->k_cache || !sl->v_cache || !sl->kv_len || !sl->cache_prev || !io->ent || !io->mean ||
        !io->mean_host || !io->hbar_scale || !io->keep_idx || !io->prune_idx || !io->cu_keep || !io->x_in || !io->x_buf[0] ||
        !io->x_buf[1] || !io->keep)
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_scale_forward: null tensor");
    if (io->scale_logits && (!io->scale_ent || !io->scale_mean || !io->scale_mean_host))
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_scale_forward: scale_logits without their outputs");
    const int B = s->B, N = s->N, L = first + count;
    const long BN = (long)B * N;
    if (B < 1 || N < 1 || (long)io->h * io->w != N)
        return nova_fail(ctx, NOVA_ERR_INVALID_ARG, "nova_pruned_scale_forward: h * w must equal N");
    if (count == 0) return NOVA_OK;
    NOVA_DEVICE_GUARD(ctx, "nova_pruned_scale_forward");
    cudaStream_t st = (cudaStream_t)stream;
    nova_status rc;
    // entropy maps; their means cross to the host in one go
    float *ent = io->ent + first * BN, *mean = io->mean + (long)first * B;
    if (io->scale_logits) {
        rc = nova_scale_entropy(ctx, io->scale_logits, io->logits_dtype, B, N, io->V, io->row_stride, io->scale_ent, io->scale_mean, stream);
        if (rc != NOVA_OK) return rc;
    }
    rc = nova_scale_entropy_layers(ctx, sl->logits + first, count, io->logits_dtype, B, N, io->V, io->row_stride, ent, mean, stream);
    if (rc != NOVA_OK) return rc;
    if (io->scale_logits)
        NOVA_CUDA_CHECK(ctx, cudaMemcpyAsync(io->scale_mean_host, io->scale_mean, sizeof(float) * B, cudaMemcpyDeviceToHost, st));
    NOVA_CUDA_CHECK(ctx, cudaMemcpyAsync(io->mean_host + (long)first * B, mean, sizeof(float) * B * count, cudaMemcpyDeviceToHost, st));
    NOVA_CUDA_CHECK(ctx, cudaStreamSynchronize(st));
    if (io->scale_logits)
        for (int b = 0; b < B; ++b) io->hbar_scale[(long)b * t + t - 1] = io->scale_mean_host[b];
    int32_t* keep = io->keep + (long)first * B;
    rc = scale_keep_counts(ctx, p, B, t, first, L, N, io->hbar_scale, io->mean_host, keep);
    if (rc != NOVA_OK) return rc;
    rc = nova_select_topk_grouped(ctx, ent, count, B, N, keep, io->keep_idx + first * BN, io->prune_idx + first * BN,
                                  io->cu_keep + (long)first * (B + 1), nullptr, stream);
    if (rc != NOVA_OK) return rc;
    const void* x = io->x_in;
    for (int j = first; j < L; ++j) {
        int32_t *keep_idx = io->keep_idx + j * BN, *prune_idx = io->prune_idx + j * BN, *cu = io->cu_keep + (long)j * (B + 1);
        nova_block_shape sj = *s;
        sj.M = 0;
        for (int b = 0; b < B; ++b) sj.M += io->keep[(long)j * B + b];
        void* out = io->x_buf[(j & 1) ^ (x == io->x_buf[j & 1])];
        rc = nova_pruned_layer_forward(ctx, sl->weights[j], sl->modulation ? sl->modulation[j] : nullptr, &sj, x, keep_idx, prune_idx,
                                       cu, sl->k_cache[j], sl->v_cache[j], sl->kv_len[j], append_kv, sl->cache_prev[j],
                                       sl->cache_prev[j] ? sl->hp : 0, sl->cache_prev[j] ? sl->wp : 0, io->h, io->w, out,
                                       sl->cache_out ? sl->cache_out[j] : nullptr, 0, stream);
        if (rc != NOVA_OK) return rc;
        x = out;
    }
    return NOVA_OK;
}
