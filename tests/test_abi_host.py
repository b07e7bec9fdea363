"""CPU-only checks of the boundary: the library builds, loads, exports every symbol that
include/sbn.h declares, and rejects bad arguments on the host before touching the GPU."""
import ctypes
import os
import re

import pytest

from paper_2603_05168_b200 import build as sbn_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    sbn_build.build()
    from paper_2603_05168_b200 import binding
    return binding.lib()


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "sbn.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(sbn_[a-z0-9_]+)\s*\(", text)))


def test_header_symbols_are_exported(L):
    names = _declared_functions()
    assert {"sbn_quantize_mask_pack", "sbn_quant_act", "sbn_sparse_bitlinear", "sbn_bitlinear"} <= set(names)
    for n in names:
        assert hasattr(L, n), f"{n} declared in sbn.h but not exported"
    from paper_2603_05168_b200 import binding
    assert sorted(binding.EXPORTS) == names


def test_every_included_source_triggers_a_rebuild():
    """Whatever libsbn.cu includes from csrc is among the files whose change makes build() compile again."""
    known, todo, seen = set(sbn_build.sources()), ["libsbn.cu"], set()
    while todo:
        name = todo.pop()
        if name in seen or not os.path.exists(os.path.join(sbn_build.CSRC, name)):
            continue
        seen.add(name)
        todo += re.findall(r'#include "([^"]+)"', open(os.path.join(sbn_build.CSRC, name)).read())
    assert len(seen) > 15
    assert {os.path.join(sbn_build.CSRC, n) for n in seen} <= known


def test_status_strings(L):
    from paper_2603_05168_b200 import binding
    seen = {binding.status_string(i) for i in range(8)}
    assert len(seen) == 8
    assert binding.status_string(99) == "unknown status"


def test_workspace_query(L):
    from paper_2603_05168_b200 import binding as b
    assert b.sbn_workspace_bytes(b.OP_QUANTIZE_MASK_PACK, 0, 256, 256) >= 8 * 148
    assert b.sbn_workspace_bytes(b.OP_QUANT_ACT, 64, 0, 256) == 0
    # large T: no split-K; few tokens: split-K inside clusters, reduced on chip -- no scratch either
    assert b.sbn_workspace_bytes(b.OP_SPARSE_BITLINEAR, 4096, 2560, 2560) == 0
    assert b.sbn_workspace_bytes(b.OP_SPARSE_BITLINEAR, 4, 2560, 2560) == 0
    # split-K through global memory (here forced): int32 [T][N] sums + one counter per output tile
    b.sbn_set_gemm_tuning(64, 5)
    try:
        assert b.sbn_workspace_bytes(b.OP_SPARSE_BITLINEAR, 4, 2560, 2560) == 4 * 2560 * 4 + 20 * 4
    finally:
        b.sbn_set_gemm_tuning(0, 0)
    assert b.sbn_workspace_bytes(b.OP_BITLINEAR, 4, 2560, 100) == 0      # illegal shape -> 0
    assert b.sbn_workspace_bytes(77, 4, 2560, 2560) == 0


def test_argument_validation_on_host(L):
    # fake, never dereferenced, 16-byte aligned "device pointers": every call below must return
    # an error code from the host-side checks before any CUDA call is made
    p = ctypes.c_void_p(0x1000)
    odd = ctypes.c_void_p(0x1004)
    NULL, SHAPE, ALIGN, UNSUP, WS = 1, 2, 3, 4, 5
    assert L.sbn_quant_act(None, 4, 256, p, p, None) == NULL
    assert L.sbn_quant_act(p, 0, 256, p, p, None) == SHAPE
    assert L.sbn_quant_act(p, 4, 100, p, p, None) == SHAPE
    assert L.sbn_quant_act(odd, 4, 256, p, p, None) == ALIGN
    nq = lambda **k: L.sbn_norm_quant_act(k.get("x", p), k.get("T", 4), k.get("K", 256), k.get("g", p),
                                          ctypes.c_float(k.get("eps", 1e-6)), p, p, None)
    assert nq(x=None) == NULL
    assert nq(T=0) == SHAPE
    assert nq(K=100) == SHAPE
    assert nq(K=16384 + 128) == UNSUP           # row no longer fits in registers
    assert nq(eps=-1.0) == SHAPE
    assert nq(g=odd) == ALIGN
    assert nq(x=odd) == ALIGN
    qmp16 = lambda **k: L.sbn_quantize_mask_pack_bf16(k.get("W", p), k.get("N", 256), k.get("K", 256), k.get("n", 2),
                                                      k.get("m", 4), p, p, p, None, None, None, p, k.get("wsb", 1 << 20), None)
    assert qmp16(W=None) == NULL
    assert qmp16(n=5, m=8) == UNSUP
    assert qmp16(n=6, m=8, K=384) == SHAPE      # 6:8 needs K % 256 == 0
    assert qmp16(K=64) == SHAPE
    assert qmp16(wsb=8) == WS
    assert qmp16(W=odd) == ALIGN
    qmp = lambda **k: L.sbn_quantize_mask_pack(k.get("W", p), k.get("N", 256), k.get("K", 256), k.get("n", 2),
                                               k.get("m", 4), p, p, p, None, k.get("prev"), k.get("flip"),
                                               k.get("ws", p), k.get("wsb", 1 << 20), None)
    assert qmp(W=None) == NULL
    assert qmp(n=4, m=8) == UNSUP
    assert qmp(n=6, m=8, K=128) == SHAPE        # 6:8 needs K % 256 == 0
    assert L.sbn_quantize_mask_pack(p, 256, 256, 6, 8, p, p, p, p, None, None, p, 1 << 20, None) == UNSUP   # 6:8 with dense_q
    assert L.sbn_quant_act_expand68(None, 4, 256, p, p, None) == NULL
    assert L.sbn_quant_act_expand68(p, 4, 384, p, p, None) == SHAPE
    assert L.sbn_quant_act_expand68(p, 4, 256, odd, p, None) == ALIGN
    assert L.sbn_norm_quant_act_expand68(p, 4, 384, p, ctypes.c_float(1e-6), p, p, None) == SHAPE
    assert L.sbn_norm_quant_act_expand68(p, 4, 16384 + 256, p, ctypes.c_float(1e-6), p, p, None) == UNSUP
    assert L.sbn_norm_quant_act_expand68(p, 4, 256, odd, ctypes.c_float(1e-6), p, p, None) == ALIGN
    assert L.sbn_expanded_k(2560, 6, 8) == 3840 and L.sbn_expanded_k(2560, 2, 4) == 2560
    assert L.sbn_expanded_k(2560 + 128, 6, 8) == 0 and L.sbn_expanded_k(2560, 3, 4) == 0
    assert qmp(N=100) == SHAPE
    assert qmp(K=64) == SHAPE
    assert qmp(wsb=8) == WS
    assert qmp(ws=None) == WS
    assert qmp(prev=p) == NULL           # prev_meta without flip_bits
    assert qmp(W=odd) == ALIGN
    gemm = lambda **k: L.sbn_sparse_bitlinear(k.get("xq", p), p, k.get("T", 64), p, k.get("meta", p), p,
                                              k.get("N", 256), k.get("K", 256), None, p, k.get("dt", 0), None,
                                              k.get("ws"), k.get("wsb", 0), None)
    assert gemm(xq=None) == NULL
    assert gemm(meta=None) == NULL
    assert gemm(T=0) == SHAPE
    assert gemm(N=130) == SHAPE
    assert gemm(K=192) == SHAPE
    assert gemm(dt=5) == UNSUP
    assert gemm(xq=odd) == ALIGN
    L.sbn_set_gemm_tuning(64, 5)                    # split-K through global memory needs its scratch
    try:
        assert gemm(T=4, N=2560, K=2560) == WS
    finally:
        L.sbn_set_gemm_tuning(0, 0)
    assert L.sbn_bitlinear(p, p, 64, None, p, 256, 256, None, p, 0, None, None, 0, None) == NULL
    # packed weights: conversion and the few-token GEMM on them
    assert L.sbn_pack_vals2(None, 256, 256, p, None) == NULL
    assert L.sbn_pack_vals2(p, 100, 256, p, None) == SHAPE
    assert L.sbn_pack_vals2(p, 256, 256, odd, None) == ALIGN
    pk = lambda **k: L.sbn_sparse_bitlinear_packed(k.get("xq", p), p, k.get("T", 16), k.get("v2", p), k.get("meta", p), p,
                                                   k.get("N", 256), k.get("K", 512), None, p, k.get("dt", 0), None, None)
    assert pk(v2=None) == NULL
    assert pk(meta=None) == NULL
    assert pk(T=0) == SHAPE
    assert pk(K=192) == SHAPE
    assert pk(T=2000) == UNSUP              # few tokens only
    assert pk(K=128) == UNSUP               # at least two k-blocks to split
    assert pk(dt=7) == UNSUP
    assert pk(xq=odd) == ALIGN
    from paper_2603_05168_b200 import binding as b
    assert L.sbn_quantize_mask_pack_batched(0, p, p, 1 << 20, None) == SHAPE
    assert L.sbn_quantize_mask_pack_batched(2, None, p, 1 << 20, None) == NULL
    jobs = (b.PackJob * 2)()
    for j in jobs:
        j.W, j.N, j.K, j.vals, j.meta, j.w_scale = 0x1000, 256, 256, 0x1000, 0x1000, 0x1000
    assert L.sbn_quantize_mask_pack_batched(2, ctypes.cast(jobs, ctypes.c_void_p), p, 16, None) == WS
    jobs[1].K = 100
    assert L.sbn_quantize_mask_pack_batched(2, ctypes.cast(jobs, ctypes.c_void_p), p, 1 << 20, None) == SHAPE
    assert b.sbn_batch_workspace_bytes(3) >= 3 * 148 * 16


def test_binding_fails_loudly_without_library(tmp_path, monkeypatch):
    from paper_2603_05168_b200 import binding
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "LIB_PATH", str(tmp_path / "missing.so"))
    with pytest.raises(RuntimeError):
        binding.lib()


def test_dispatch_plan_is_sane(L):
    # host-only: the dispatcher's choices for the shapes the benchmarks use (kernel, tile, split, cluster)
    from paper_2603_05168_b200 import binding as b
    assert b.sbn_plan_gemm(True, 4096, 3840, 2560)[0] == 3            # large T, short K: CTA pairs, 256-feature tiles
    assert b.sbn_plan_gemm(True, 8192, 4096, 11008)[0] == 2           # large T, long K: CTA pairs, 512-feature tiles
    k, bn, split, cluster = b.sbn_plan_gemm(True, 16, 3840, 2560)     # few tokens: cluster split-K, 32-token tile
    assert (k, bn, split) == (1, 32, 1) and cluster in (2, 3, 4)
    for T in (1, 16, 32):
        for (N, K) in ((3840, 2560), (2560, 6912), (11008, 4096), (4096, 11008)):
            k, bn, split, cluster = b.sbn_plan_gemm(True, T, N, K)
            assert k == 1 and split == 1 and cluster in (2, 3, 4), (T, N, K)
            tiles = (N // 128) * ((T + bn - 1) // bn)
            assert tiles * cluster <= (296 if bn <= 64 else 148)       # every CTA resident at once
    assert b.sbn_plan_gemm(True, 16, 100, 2560) == (0, 0, 0, 0)        # illegal shape


def test_fused_entry_validation_on_host(L):
    p = ctypes.c_void_p(0x1000)
    odd = ctypes.c_void_p(0x1004)
    NULL, SHAPE, ALIGN, UNSUP = 1, 2, 3, 4
    fs = lambda **k: L.sbn_quant_act_sparse_bitlinear(k.get("x", p), k.get("T", 8), p, k.get("meta", p), p, k.get("N", 256),
                                                      k.get("K", 512), None, p, k.get("dt", 0), None, None, None)
    assert fs(x=None) == NULL
    assert fs(meta=None) == NULL
    assert fs(T=0) == SHAPE
    assert fs(N=100) == SHAPE
    assert fs(T=300) == UNSUP
    assert fs(K=128) == UNSUP
    assert fs(dt=9) == UNSUP
    assert fs(x=odd) == ALIGN
    assert L.sbn_quant_act_bitlinear(p, 8, None, p, 256, 512, None, p, 0, None, None, None) == NULL


def test_canonical_layout_calls_validate_on_host(L):
    p, q = ctypes.c_void_p(0x1000), ctypes.c_void_p(0x2000)
    odd = ctypes.c_void_p(0x1008)
    NULL, SHAPE, ALIGN, UNSUP = 1, 2, 3, 4
    for fn in (L.sbn_unpack_canonical, L.sbn_tile_canonical):
        assert fn(None, None, 256, 256, None, None, None) == NULL          # nothing to convert
        assert fn(p, None, 256, 256, None, None, None) == NULL             # a source without its destination
        assert fn(p, p, 256, 100, q, q, None) == SHAPE
        assert fn(p, p, 0, 256, q, q, None) == SHAPE
        assert fn(odd, p, 256, 256, q, q, None) == ALIGN
        assert fn(p, p, 256, 256, p, q, None) == UNSUP                     # in place


def test_native_calls_marshal_like_the_abi(L, monkeypatch):
    """The extension hands every argument of a tensor call to the C ABI where sbn.h has it (fake functions, CPU tensors)."""
    import torch
    from paper_2603_05168_b200 import binding as b
    seen = {}

    def fake(name):
        argtypes = getattr(L, name).argtypes
        def f(*args):
            seen[name] = args
            return 3
        return ctypes.CFUNCTYPE(ctypes.c_int, *argtypes)(f)

    fakes = {name: fake(name) for name in b._NATIVE_CALLS}
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 1, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda dev: 0x70 + dev, raising=False)
    monkeypatch.setattr(b, "lib", lambda: type("Fake", (), fakes))
    monkeypatch.setattr(b, "_native", None)                          # restored afterwards: the next real use binds again
    monkeypatch.setattr(b, "status_string", lambda code: "")
    T, N, K = 3, 128, 256
    t = lambda *shape, dt=torch.int8: torch.zeros(shape, dtype=dt)
    x, xq, sc, vals, meta, w = t(T, K, dt=torch.bfloat16), t(16 * K), t(T, dt=torch.float32), t(N, K // 2), t(N, K // 8), t(1)
    y, yf, bias, acc, ws, q = t(T, N, dt=torch.bfloat16), t(T, N, dt=torch.float32), t(N), t(T), t(5, dt=torch.int32), t(N, K)
    p = lambda v: v.data_ptr()
    calls = [
        (lambda: b.sbn_quant_act(x, xq, sc), "sbn_quant_act", (p(x), T, K, p(xq), p(sc))),
        (lambda: b.sbn_quant_act_expand68(x, xq, sc), "sbn_quant_act_expand68", (p(x), T, K, p(xq), p(sc))),
        (lambda: b.sbn_norm_quant_act(x, xq, sc, gain=bias, eps=0.5), "sbn_norm_quant_act", (p(x), T, K, p(bias), 0.5, p(xq), p(sc))),
        (lambda: b.sbn_norm_quant_act(x, xq, sc, expand68=True), "sbn_norm_quant_act_expand68", (p(x), T, K, None, ctypes.c_float(1e-6).value, p(xq), p(sc))),
        (lambda: b.sbn_sparse_bitlinear(xq, sc, vals, meta, w, y, bias=bias, ws=ws), "sbn_sparse_bitlinear",
         (p(xq), p(sc), T, p(vals), p(meta), p(w), N, K, p(bias), p(y), b.OUT_BF16, None, p(ws), 20)),
        (lambda: b.sbn_bitlinear(xq, sc, q, w, yf, acc_out=acc), "sbn_bitlinear",
         (p(xq), p(sc), T, p(q), p(w), N, K, None, p(yf), b.OUT_F32, p(acc), None, 0)),
        (lambda: b.sbn_sparse_bitlinear_packed(xq, sc, meta, vals, w, y, acc_out=acc), "sbn_sparse_bitlinear_packed",
         (p(xq), p(sc), T, p(meta), p(vals), p(w), N, K, None, p(y), b.OUT_BF16, p(acc))),
        (lambda: b.sbn_quant_act_sparse_bitlinear(x, vals, meta, w, yf, bias=bias, a_scale_out=sc), "sbn_quant_act_sparse_bitlinear",
         (p(x), T, p(vals), p(meta), p(w), N, K, p(bias), p(yf), b.OUT_F32, None, p(sc))),
        (lambda: b.sbn_quant_act_bitlinear(x, q, w, y), "sbn_quant_act_bitlinear",
         (p(x), T, p(q), p(w), N, K, None, p(y), b.OUT_BF16, None, None)),
    ]
    for call, name, want in calls:
        with pytest.raises(b.SbnError) as err:
            call()
        assert err.value.code == 3
        assert seen.pop(name) == want + (0x71,), name
    with pytest.raises(ValueError):
        b.sbn_quant_act(xq, xq, sc)                                  # not two-dimensional
    assert not seen


def test_plans_never_ask_for_more_clusters_than_fit(L):
    """The split-K clusters of a plan are resident all at once: 148 / 88 / 70 of 2 / 3 / 4 CTAs at two per SM (narrow tiles),
    74 / 44 / 33 at one (wide tiles)."""
    import random
    from paper_2603_05168_b200 import binding as b
    rng = random.Random(3)
    seen = set()
    for _ in range(20000):
        T, N, K = round(2 ** rng.uniform(0, 12)), 128 * round(2 ** rng.uniform(0, 7)), 128 * round(2 ** rng.uniform(1, 7.5))
        kernel, bn, split, cluster = b.sbn_plan_gemm(rng.random() < 0.5, T, N, K)
        assert bn % 16 == 0 and 32 <= bn <= 256
        if kernel == 1:
            tiles = N // 128 * -(-T // bn)
            assert tiles <= ({2: 148, 3: 88, 4: 70} if bn <= 64 else {2: 74, 3: 44, 4: 33})[cluster], (T, N, K)
            assert cluster <= K // 128
        seen.add((kernel, cluster, bn > 64))
    assert len(seen) >= 9                                             # tiles, both pairs, every cluster size in both widths


def test_unsplit_wide_tiles_are_reported_and_at_most_one_per_sm(L):
    import random
    from paper_2603_05168_b200 import binding as b
    rng = random.Random(4)
    assert b.sbn_plan_gemm(False, 600, 4096, 11008)[0] == 4
    n = 0
    for _ in range(5000):
        T, N, K = round(2 ** rng.uniform(6, 11.5)), 128 * round(2 ** rng.uniform(0, 7)), 128 * round(2 ** rng.uniform(1, 7.5))
        assert b.sbn_plan_gemm(True, T, N, K)[0] != 4                 # dense weights only
        kernel, bn, split, cluster = b.sbn_plan_gemm(False, T, N, K)
        if kernel == 0:
            assert bn in (64, 128, 256), (T, N, K)                    # the widths that the single-CTA kernel has
        if kernel == 4:
            n += 1
            assert 80 <= bn <= 256 and bn % 16 == 0 and (split, cluster) == (1, 0)
            assert 64 < T <= 2048 and N // 128 * -(-T // bn) <= 148, (T, N, K)
    assert n > 100


def test_forced_cluster_plans_are_ones_that_a_kernel_has(L):
    """Whatever sbn_set_gemm_tuning is given: narrow tiles have code for clusters of 2, 3, 4 and 8 CTAs only (5 to 7, or 1, would
    address CTAs that do not exist), wide tiles are at least 80 tokens wide."""
    from paper_2603_05168_b200 import binding as b
    try:
        for tile in [*range(32, 100), 128, 255, 256, 300]:
            for split in range(-9, 0):
                for sparse, T, N, K in [(True, 72, 256, 2560), (False, 300, 384, 1024), (True, 9, 128, 256), (False, 100, 128, 128)]:
                    b.sbn_set_gemm_tuning(tile, split)
                    kernel, bn, _, cluster = plan = b.sbn_plan_gemm(sparse, T, N, K)
                    assert bn % 16 == 0 and cluster <= max(1, K // 128), (tile, split, plan)
                    if kernel == 1:
                        assert cluster in (2, 3, 4, 8) if bn <= 64 else 2 <= cluster <= 8, (tile, split, plan)
                        assert bn in (32, 64) or bn >= 80, (tile, split, plan)
                    if 64 < tile < 80 and K >= 256:                   # rounds down to 64, a narrow tile
                        b.sbn_set_gemm_tuning(64, split)
                        assert plan == b.sbn_plan_gemm(sparse, T, N, K), (tile, split)
    finally:
        b.sbn_set_gemm_tuning(0, 0)


def test_wide_matrices_run_on_pairs_and_long_dense_rows_may_split(L):
    from paper_2603_05168_b200 import binding as b
    assert b.sbn_plan_gemm(True, 16, 20480, 4096)[0] in (2, 3)        # 160 row tiles: more than the clusters have places
    assert b.sbn_plan_gemm(False, 9, 2304, 24576)[2] > 1              # K through global memory, with a workspace
    assert b.sbn_workspace_bytes(b.OP_BITLINEAR, 9, 2304, 24576) > 0
    assert b.sbn_workspace_bytes(b.OP_BITLINEAR, 8, 2304, 24576) == 0  # the register-fed kernel needs none
    for T in (9, 16, 64, 201, 777):
        assert b.sbn_workspace_bytes(b.OP_SPARSE_BITLINEAR, T, 2304, 24576) == 0
        assert b.sbn_workspace_bytes(b.OP_BITLINEAR, T, 2304, 12288) == 0
