"""CPU-only checks of the C-ABI library: it loads without a GPU, exports every symbol the
header declares, and its host-side schedule arithmetic (Eq. 8-13) is bit-identical to the
oracle's on random histories."""
import ctypes
import os
import re

import numpy as np
import pytest
import torch

import oracle
import paper_2602_01345_b200 as nova

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "nova.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(nova_[a-z0-9_]+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    names = _declared_functions()
    assert {"nova_scale_entropy", "nova_keep_ratios", "nova_select_topk",
            "nova_pruned_block_forward", "nova_restore_from_cache"} <= set(names)
    lib = ctypes.CDLL(nova.lib_path())
    for n in names:
        assert hasattr(lib, n), f"{n} declared in include/nova.h but not exported"


def test_status_strings_and_default_params():
    lib = ctypes.CDLL(nova.lib_path())
    lib.nova_status_string.restype = ctypes.c_char_p
    assert lib.nova_status_string(0) == b"ok"
    assert lib.nova_status_string(6) == b"device-side wait expired"
    from paper_2602_01345_b200.binding import _SchedParams
    p = _SchedParams()
    lib.nova_sched_params_default(ctypes.byref(p))
    assert (p.t_est, p.alpha, p.tau, p.lam, p.k_min, p.ratio_max, p.force_act_scale) == (5, 0.5, 0.8, 0.1, 1, 1.0, 0)
    assert p.force_keep_ratio < 0


def test_workspace_bytes_host_side():
    ok = nova.BlockShape(B=2, N=256, C=1024, n_heads=16, F=4096, Lmax=680, M=256)
    need = nova.nova_block_workspace_bytes(ok)
    assert need >= 256 * (4 * 1024 + 4096) * 2
    bad = nova.BlockShape(B=2, N=256, C=1000, n_heads=16, F=4096, Lmax=680, M=256)
    assert nova.nova_block_workspace_bytes(bad) == 0
    bad_dh = nova.BlockShape(B=2, N=256, C=1024, n_heads=32, F=4096, Lmax=680, M=256)   # dh = 32
    assert nova.nova_block_workspace_bytes(bad_dh) == 0


def test_gemm_warps_that_give_up_alone_share_no_barrier():
    """In the GEMM for many tiles (and the head's entropy) each warp leaves its loop on its own when a bounded wait fails, so
    the loops may not hold a barrier at which the others would stay: read from the source, as a wait that fails beside
    one that does not cannot be arranged on a GPU without leaving it in an unknown state."""
    text = open(os.path.join(ROOT, "paper_2602_01345_b200", "csrc", "gemm.cu")).read()
    kernel = text[text.index("gemm_bf16_tn_pair(const"):text.index("nova_status launch_pair(")]
    roles = re.sub(r"//[^\n]*", "", kernel[kernel.index("if (warp == 0) {"):kernel.rindex("__syncthreads();")])
    assert "if (!ok) break;" in roles
    assert not re.search(r"bar\.sync|barrier\.sync|__syncthreads|__barrier_sync|cluster_sync", roles)


def _compare(p_or, p_lib, t, j, N, hs, hl):
    want = oracle.keep_ratios(p_or, t, j, N, hs, hl)
    got = nova.nova_keep_ratios(p_lib, t, j, N, torch.from_numpy(hs), torch.from_numpy(hl) if hl is not None else None)
    for key in ("t_star", "act_scale", "keep"):
        assert np.array_equal(got[key].numpy(), want[key]), key
    for key in ("ratio_scale", "ratio_layer"):
        assert np.array_equal(got[key].numpy(), want[key]), key     # bit-identical doubles


def test_keep_ratios_bit_exact_against_oracle_random_histories():
    rng = np.random.default_rng(0)
    for trial in range(300):
        B = int(rng.integers(1, 9))
        T = int(rng.integers(1, 17))
        L = int(rng.integers(1, 33))
        N = int(rng.choice([1, 7, 256, 1024, 4096, 16384]))
        # rising-then-flattening curves with noise so every branch of the trigger is visited
        t_axis = np.arange(1, T + 1)
        t0 = rng.uniform(1, 8, (B, 1))
        hs = (2 + 6 / (1 + np.exp(-(t_axis[None] - t0) / rng.uniform(0.4, 2, (B, 1)))) +
              0.05 * rng.standard_normal((B, T))).astype(np.float32)
        j = int(rng.integers(1, L + 1))
        hl = (hs[:, -1:] * rng.uniform(0.7, 1.3, (B, j))).astype(np.float32)
        kw = dict(t_est=int(rng.integers(2, 7)), alpha=float(rng.uniform(0.1, 0.9)),
                  tau=float(rng.uniform(0.3, 2.0)), lam=float(rng.uniform(0, 0.3)),
                  k_min=int(rng.integers(0, 4)), ratio_max=float(rng.uniform(0.5, 1.0)))
        if trial % 5 == 0:
            kw["force_act_scale"] = int(rng.integers(1, T + 2))
        if trial % 7 == 0:
            kw["force_keep_ratio"] = float(rng.choice([0.2, 0.25, 0.5, 0.75, 1.0]))
        _compare(oracle.SchedParams(**kw), nova.SchedParams(**kw), T, j, N, hs, hl)


def test_keep_ratios_all_layers_equals_layer_by_layer_and_oracle():
    """The all-layers call gives, for every layer j, what the per-layer call and the oracle give on
    the means of layers 1..j (Eq. 12-13), bit for bit."""
    rng = np.random.default_rng(3)
    for trial in range(40):
        B, T, L = int(rng.integers(1, 9)), int(rng.integers(6, 14)), int(rng.integers(1, 33))
        N = int(rng.choice([256, 1024, 4096]))
        t_axis = np.arange(1, T + 1)
        hs = (2 + 6 / (1 + np.exp(-(t_axis[None] - rng.uniform(1, 6, (B, 1))) / rng.uniform(0.4, 2, (B, 1)))) +
              0.05 * rng.standard_normal((B, T))).astype(np.float32)
        hl = (hs[:, -1:] * rng.uniform(0.7, 1.3, (B, L))).astype(np.float32)
        kw = dict(lam=float(rng.uniform(0, 0.3)), tau=float(rng.uniform(0.3, 2.0)))
        if trial % 4 == 0:
            kw["force_act_scale"] = T - 1
        got = nova.nova_keep_ratios_layers(nova.SchedParams(**kw), T, N, torch.from_numpy(hs), torch.from_numpy(hl))
        pruned = 0
        for j in range(1, L + 1):
            want = oracle.keep_ratios(oracle.SchedParams(**kw), T, j, N, hs, hl[:, :j].copy())
            assert np.array_equal(got["keep"][j - 1].numpy(), want["keep"]), (trial, j)
            assert np.array_equal(got["ratio_layer"][j - 1].numpy(), want["ratio_layer"]), (trial, j)
            pruned += int((want["keep"] < N).sum())
        assert np.array_equal(got["t_star"].numpy(), want["t_star"])
        assert np.array_equal(got["act_scale"].numpy(), want["act_scale"])
        assert np.array_equal(got["ratio_scale"].numpy(), want["ratio_scale"])
        if trial % 4 == 0:
            assert pruned > 0


def test_keep_ratios_worked_example_and_errors():
    hs = np.array([[1, 2, 3, 4, 5, 6, 6, 6, 6, 6]], np.float32)
    got = nova.nova_keep_ratios(nova.SchedParams(), 8, 1, 256, torch.from_numpy(hs[:, :8]))
    assert got["t_star"].item() == 7 and got["act_scale"].item() == 8 and got["keep"].item() == 128
    import pytest
    with pytest.raises(nova.NovaError):
        nova.nova_keep_ratios(nova.SchedParams(tau=0.0), 8, 1, 256, torch.from_numpy(hs[:, :8]))
    with pytest.raises(nova.NovaError):
        nova.nova_keep_ratios(nova.SchedParams(t_est=1), 8, 1, 256, torch.from_numpy(hs[:, :8]))


def test_overlapping_kernels_use_no_non_coherent_loads():
    """Kernels launched with programmatic stream serialisation live while the launch before them still writes.
    ld.global.nc (which a `const T* __restrict__` parameter or __ldg lets the compiler use) is only for memory that nobody writes
    during the kernel's life, and griddepcontrol.wait does not order it."""
    csrc = os.path.join(ROOT, "paper_2602_01345_b200", "csrc")
    seen = set()
    for name in sorted(os.listdir(csrc)):
        text = re.sub(r"//[^\n]*|__(launch_bounds|cluster_dims)__\([^()]*\)", "", open(os.path.join(csrc, name)).read())
        if "nova_launch_pdl(" not in text or name == "common.cuh":
            continue
        assert "ld.global.nc" not in text and "__ldg" not in text, name
        for m in re.finditer(r"__global__[^;{]*?(\w+)\(([^{;]*)\)\s*\{", text):
            if "pdl_wait();" in text[m.end():]:
                assert not re.search(r"const\s+[\w ]+\*\s*__restrict__", m.group(2)), (name, m.group(1))
                seen.add(m.group(1))
    assert {"layernorm_rows", "qk_transform_kernel", "restore_kernel", "gemm_bf16_tn_pair", "gemm_bf16_split", "attention_kernel"} <= seen


def _scale_call(B=2, N=6, C=64, L=3):
    """A ScaleCall on host memory without a context: its tables can be looked at, and every native call is refused."""
    from paper_2602_01345_b200 import binding as nv

    class NoContext:
        handle = None

        def check(self, status):
            if status:
                raise nova.NovaError(status, "refused")

    z = lambda *s, dtype=torch.float32: torch.zeros(s, dtype=dtype)  # noqa: E731
    i32, bf16 = torch.int32, torch.bfloat16
    call = nv.ScaleCall(NoContext(), nova.BlockShape(B, N, C, 1, 64, 32, B * N), 2, 3, L, z(L, B, N), z(L, B), z(L, B), z(L, B * N, dtype=i32),
                        z(L, B * N, dtype=i32), z(L, B + 1, dtype=i32), [z(B, N, C, dtype=bf16) for _ in range(2)])
    weights = [type("W", (), {"c": nv._BlockWeights()}) for _ in range(L)]
    caches = [z(B, 32, C, dtype=bf16) for _ in range(L)]
    layers = dict(weights=weights, modulation=None, k_caches=caches, v_caches=caches, kv_len=z(L, B, dtype=i32),
                  cache_prev=[z(B, 2, 2, C, dtype=bf16) for _ in range(L)], cache_out=None)
    return call, layers


def test_scale_call_forgets_the_scale_logits_of_a_pass_that_failed():
    call, layers = _scale_call()
    call.set_layers(**layers)
    logits = torch.zeros((2, 6, 32), dtype=torch.bfloat16)
    call.set_logits([logits] * 3)
    call.set_scale_logits(logits, torch.zeros(2, 6), torch.zeros(2), torch.zeros(2))
    with pytest.raises(nova.NovaError):
        call.run(nova.SchedParams(), 1, torch.zeros(2, 1), torch.zeros((2, 6, 64), dtype=torch.bfloat16), 0, 3, True, stream=0)
    assert call.io.scale_logits is None


def test_scale_call_takes_only_lengths_that_lie_together():
    """kv_len: a whole [L, B] tensor, rows of a wider one, or a tensor per layer; never strided views, whose
    neighbours would be read and advanced instead, and never 64-bit lengths."""
    call, layers = _scale_call()
    L, B, i32 = 3, 2, torch.int32
    table = call._tables[5]
    for good in (torch.zeros((L, B), dtype=i32), torch.zeros((L + 1, B), dtype=i32), torch.zeros((L, B + 2), dtype=i32)[:, :B],
                 list(torch.zeros((L, B), dtype=i32).unbind(0)), torch.zeros((2 * L, B), dtype=i32)[::2]):
        call.set_layers(**{**layers, "kv_len": good})
        assert [table[j] for j in range(L)] == [good[j].data_ptr() for j in range(L)]
    for bad in (torch.zeros((B, L), dtype=i32).t(), list(torch.zeros((B, L), dtype=i32).unbind(1)),
                torch.zeros((L, B), dtype=torch.int64), torch.zeros((L, 1), dtype=i32)):
        with pytest.raises(AssertionError):
            call.set_layers(**{**layers, "kv_len": bad})


def test_scale_call_takes_only_contiguous_caches():
    call, layers = _scale_call()
    for name in ("k_caches", "v_caches", "cache_prev", "cache_out"):
        wide = torch.zeros((3, 2, 2, 2, 128), dtype=torch.bfloat16)
        views = [t[..., :64] if name.startswith("cache") else t.flatten(1, 2)[..., :64] for t in wide]
        with pytest.raises(AssertionError):
            call.set_layers(**{**layers, name: views})


def test_scale_call_takes_layers_without_modulation_among_others():
    call, layers = _scale_call()
    shift = {"shift1": torch.zeros((2, 64), dtype=torch.bfloat16)}
    call.set_layers(**{**layers, "modulation": [shift, None, {}]})
    assert [bool(p) for p in call._tables[1]] == [True, False, False]
    call.set_layers(**{**layers, "modulation": [None, shift, shift]})
    assert [bool(p) for p in call._tables[1]] == [False, True, True]


def test_scale_call_ignores_logits_past_its_last_layer():
    call, _ = _scale_call()
    logits = torch.zeros((5, 2, 6, 32), dtype=torch.bfloat16)
    for given in (logits, list(logits), [*logits[:3], None]):
        call.set_logits(given)
        assert [call._tables[2][j] for j in range(3)] == [logits[j].data_ptr() for j in range(3)]
    with pytest.raises(AssertionError):
        call.set_logits(logits[:2])


def _gemm_plan(num_sms, M, N, K):
    lib = ctypes.CDLL(nova.lib_path())
    parts, tile = ctypes.c_int(), ctypes.c_int()
    takes = lib.nova_debug_gemm_plan(num_sms, M, N, K, ctypes.byref(parts), ctypes.byref(tile))
    return bool(takes), parts.value, tile.value


def test_gemm_plan_follows_from_the_sizes_and_the_sm_count():
    """The plan needs no device and is the one measured on 148 SMs; its token tiles all run at once on the
    clusters it counts on (two SMs lost per GPC and cluster of four), and past the first row count that the split
    kernel leaves to the other one it takes none."""
    assert _gemm_plan(148, 256, 1024, 4096) == (True, 2, 32)
    assert _gemm_plan(148, 300, 2048, 8192) == (True, 2, 96)
    assert _gemm_plan(148, 300, 6144, 2048) == (True, 1, 128)
    assert _gemm_plan(148, 1600, 2048, 8192)[0] and not _gemm_plan(148, 2250, 1920, 7680)[0]
    assert not _gemm_plan(148, 8192, 2048, 2048)[0]
    for num_sms in (2, 18, 64, 132, 148, 160):
        for N, K in ((1024, 1024), (1920, 7680), (6144, 2048), (64, 64), (320, 320)):
            taken = True
            for M in (*range(1, 400, 7), *range(400, 3000, 61)):
                takes, parts, tile = _gemm_plan(num_sms, M, N, K)
                assert taken or not takes
                taken = takes
                if takes:
                    assert parts in (1, 2) and parts <= K // 64 and tile % 32 == 0 and 32 <= tile <= 256
                    clusters = num_sms // 2 if parts == 1 else max(1, (num_sms - 16) // 4)
                    assert -(-N // 256) * -(-M // tile) <= clusters
