"""GPU parity: the CUDA path (through the C ABI) against the CPU oracle on the same seeded
inputs.  Integer artefacts (ternary values, metadata, int8 activations, int32 accumulators, flip
counts) must match bit for bit; fp32 outputs within 1e-5 relative; bf16 outputs within 1 ulp."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_05168_b200 import binding as b
from paper_2603_05168_b200 import inputs

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_harness import (gpu_norm_quant_act, bf16_dev, bf16_tensor_bits, dev, expand68_columns, fold68, gpu_gemm,
                             gpu_gemm_packed, gpu_pack_vals2, gpu_quant_act, gpu_quant_act_expand68, gpu_quantize_mask_pack,
                             gpu_quantize_mask_pack68, gpu_unpack_canonical, tile_meta, tile_vals,
                             xq_to_numpy, y_to_f32_numpy)


@pytest.fixture(autouse=True)
def _reset_tuning():
    b.sbn_set_gemm_tuning(0, 0)
    yield
    b.sbn_set_gemm_tuning(0, 0)


def _oracle_pack(W):
    r = oracle.quantize_mask_pack(W)
    if r["near_tie"]:
        pytest.skip("gamma within rounding distance of an fp32 midpoint for this seed")
    return r


def _assert_y(y_gpu_f32, y_ref, rel=1e-5):
    denom = np.maximum(np.abs(y_ref), 1e-30)
    err = np.abs(y_gpu_f32 - y_ref) / denom
    err[y_ref == 0] = np.abs(y_gpu_f32[y_ref == 0])
    assert err.max() <= rel, f"max rel err {err.max()}"


# ------------------------------------------------------------------------------------------------
# part 2: activations
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("T,K", [(64, 256), (1, 2560), (5, 128), (67, 2560), (33, 6912), (19, 11008),
                                 (3, 4096), (2, 16384), (3, 17408), (300, 128)])
def test_quant_act_parity(T, K):
    x = inputs.activations_bf16(T, K, seed=100 + T + K, token_lognormal_sigma=0.5)
    xq_ref, s_ref = oracle.quant_act(x)
    xq, s = gpu_quant_act(x)
    assert np.array_equal(xq_to_numpy(xq, T, K), xq_ref)
    assert np.array_equal(s.cpu().numpy(), s_ref)


def test_quant_act_edge_rows():
    K = 256
    x = np.zeros((6, K), np.float32)
    x[0, :8] = [127, 0.5, 1.5, 2.5, -0.5, -1.5, -2.5, 3.5]       # exact halves with s_x = 1
    # row 1 stays all zero -> clamp path
    x[2, :] = 1e-7                                                # below the clamp
    x[3, 5] = -3.0e38                                             # huge magnitude
    x[4, :] = np.linspace(-1, 1, K)
    x[5, ::2] = 65280.0
    bits = inputs.f32_to_bf16_bits(x)
    xq_ref, s_ref = oracle.quant_act(bits)
    xq, s = gpu_quant_act(bits)
    assert np.array_equal(xq_to_numpy(xq, 6, K), xq_ref)
    assert np.array_equal(s.cpu().numpy(), s_ref)
    assert xq_ref[0, :8].tolist() == [127, 0, 2, 2, 0, -2, -2, 4]


# ------------------------------------------------------------------------------------------------
# part 2 with the norm fused in (Algorithm 1: x~ = Q_a(Norm(x)))
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("with_gain", [True, False])
@pytest.mark.parametrize("T,K", [(64, 256), (1, 2560), (5, 128), (67, 2560), (33, 6912), (19, 11008),
                                  (300, 4096), (9, 16384), (130, 1024)])
def test_norm_quant_act_parity(T, K, with_gain):
    x = inputs.activations_bf16(T, K, seed=T + K, token_lognormal_sigma=0.5)
    gain = (1.0 + 0.2 * np.random.default_rng(K).standard_normal(K)).astype(np.float32) if with_gain else None
    r = oracle.norm_quant_act(x, gain, 1e-6)
    xq, s = gpu_norm_quant_act(x, gain, 1e-6)
    ok = ~r["near_tie"]
    assert ok.all(), "a row's mean square sits on an fp32 rounding boundary for this seed"
    assert np.array_equal(s.cpu().numpy(), r["a_scale"])
    assert np.array_equal(xq_to_numpy(xq, T, K), r["xq"])


# around the row counts where a whole CTA per row gives way to two or more rows per CTA; columns that leave the last
# vectors of a thread empty, and the widest row the whole-CTA form takes.  Whole numbers: equality.
@pytest.mark.parametrize("T,K", [(1, 1280), (148, 1280), (149, 1280), (1, 2048), (444, 2176), (445, 2176), (444, 4096), (1, 1152)])
def test_norm_quant_act_rows_per_cta(T, K):
    test_norm_quant_act_parity(T, K, True)


# a warp per row: from the row counts where that begins, rows that leave the last round partly empty, columns that are no multiple
# of 256 (the last vectors belong to half a warp), the narrowest and widest rows
@pytest.mark.parametrize("T,K", [(1924, 1024), (1925, 1152), (2500, 2560), (1924, 5120)])
def test_quant_act_warp_per_row(T, K):
    test_quant_act_parity(T, K)


@pytest.mark.parametrize("T,K", [(1000, 1280), (1001, 1408), (5000, 2560), (1000, 3328), (7000, 3456)])
def test_norm_quant_act_warp_per_row(T, K):
    for with_gain in (True, False):
        test_norm_quant_act_parity(T, K, with_gain)
    test_norm_quant_act_rows_that_overflow(T, K)


# What a row becomes does not depend on how many rows the call has, non-finite rows included: row counts on both sides of where other
# kernels begin, every number of warps that a row of that length can have
@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("K", [1024, 1152, 2560, 3072, 4096, 5120])
def test_rows_do_not_depend_on_their_number(K, norm):
    T, parts = 7040, [16, 101, 963, 1000, 1960, 3000]
    bits = inputs.activations_bf16(T, K, seed=K).reshape(T, K)
    rng = np.random.default_rng(K)
    for t in range(0, T, 5):                                    # an infinity or a NaN or two in every fifth row, anywhere
        for v in rng.choice([0x7F80, 0xFF80, 0x7FC0, 0xFFC1, 0x7F7F], size=1 + t % 2):
            bits[t, rng.integers(K)] = v
    bits[3, :] = 0x7FC0
    quantise = gpu_norm_quant_act if norm else gpu_quant_act
    xq, s = quantise(bits)
    xq, s = xq_to_numpy(xq, T, K), s.cpu().numpy()
    begin = 0
    for n in parts:
        q, t = quantise(bits[begin:begin + n])
        assert np.array_equal(xq_to_numpy(q, n, K), xq[begin:begin + n]), n
        assert np.array_equal(t.cpu().numpy().view(np.uint32), s[begin:begin + n].view(np.uint32)), n
        begin += n
    assert begin == T


# Finite inputs whose normalised row is not finite: no scale brings such a value into range, and its code is 127 (the saturated
# end), as for every width of the kernel; with eps > 0 and finite products nothing changes.
@pytest.mark.parametrize("T,K", [(5, 256), (5, 1280), (600, 1280), (600, 2560), (5, 4096), (600, 6912), (600, 11008), (5, 16384)])
def test_norm_quant_act_rows_that_overflow(T, K):
    x = np.random.default_rng(K).standard_normal((T, K)).astype(np.float32)
    x[0] = 0.0                                        # mean square 0: r is infinite, 0 * r is not a number
    x[1] *= 1e-30                                     # squares vanish in fp32: r is infinite, x * r too
    x[2] = 0.0
    x[2, K // 2] = -1e-30
    bits = inputs.f32_to_bf16_bits(x)
    xq, s = gpu_norm_quant_act(bits, None, 0.0)
    codes = xq_to_numpy(xq, T, K)
    s = s.cpu().numpy()
    assert (codes[:3] == 127).all()
    assert s[0] == np.float32(1e-5) / np.float32(127.0) and np.isinf(s[1:3]).all()
    r = oracle.norm_quant_act(bits, None, 1e-6)
    xq, s = gpu_norm_quant_act(bits, None, 1e-6)
    ok = ~r["near_tie"]
    assert np.array_equal(xq_to_numpy(xq, T, K)[ok], r["xq"][ok])
    gain = np.full(K, 1e30, np.float32)
    gain[::7] = 3e38                                  # |xn| > 1.14 times this is out of range
    xn = np.abs(oracle.norm_quant_act(bits, None, 1e-6, want_xn=True)["xn"][3]) * gain.astype(np.float64)
    out_of_range = xn > 3.5e38
    close = np.abs(xn - 3.4e38) < 0.1e38
    assert out_of_range.any()
    xq, s = gpu_norm_quant_act(bits, gain, 1e-6)
    row = xq_to_numpy(xq, T, K)[3]
    assert np.array_equal(row[~close], np.where(out_of_range, 127, 0)[~close]) and np.isinf(s.cpu().numpy()[3])


def test_norm_quant_act_edge_rows():
    K = 512
    x = np.zeros((5, K), np.float32)
    x[1, :] = 3.0                                         # constant row: every code 127
    x[2, ::2], x[2, 1::2] = 0.0078125, -0.0078125
    x[3, 7] = 65280.0                                     # one huge outlier
    x[4, :] = np.linspace(-1, 1, K)
    bits = inputs.f32_to_bf16_bits(x)
    for eps in (0.0, 1e-6, 1e-2):
        if eps == 0.0:
            sel = [1, 2, 3, 4]                            # eps = 0 on an all-zero row is 0/0
        else:
            sel = [0, 1, 2, 3, 4]
        r = oracle.norm_quant_act(bits[sel], None, eps)
        xq, s = gpu_norm_quant_act(bits[sel], None, eps)
        assert np.array_equal(s.cpu().numpy(), r["a_scale"])
        assert np.array_equal(xq_to_numpy(xq, len(sel), K), r["xq"])


# ------------------------------------------------------------------------------------------------
# part 1: quantise, mask, pack
# ------------------------------------------------------------------------------------------------
# with_dense=False is the single-pass route (provisional ternarisation + fix-up list); asking for the
# dense W_q makes the kernel ternarise everything in a second pass -- both must give the same bits.
@pytest.mark.parametrize("with_dense", [True, False])
@pytest.mark.parametrize("N,K,seed", [(256, 256, 0), (128, 128, 1), (384, 2560, 2), (128, 6912, 3), (640, 2560, 4),
                                      (2048, 2560, 7)])
def test_quantize_mask_pack_parity(N, K, seed, with_dense):
    W = inputs.latent_weights(N, K, seed=seed)
    r = _oracle_pack(W)
    g = gpu_quantize_mask_pack(W, with_dense=with_dense)
    assert g["scale"] == r["scale"]
    assert np.array_equal(g["vals"], r["vals"])
    assert np.array_equal(g["meta"], r["meta"])
    if with_dense:
        assert np.array_equal(g["dense_q"], r["dense_q"])


@pytest.mark.parametrize("with_dense", [True, False])
def test_quantize_mask_pack_heavy_tail(with_dense):
    W = inputs.latent_weights(256, 4096, seed=5, sigma=0.015, outlier_prob=0.05, outlier_mult=10.0)
    r = _oracle_pack(W)
    g = gpu_quantize_mask_pack(W, with_dense=with_dense)
    assert g["scale"] == r["scale"]
    assert np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])
    if with_dense:
        assert np.array_equal(g["dense_q"], r["dense_q"])


def test_quantize_mask_pack_adversarial():
    N, K = 128, 256
    rng = np.random.default_rng(6)
    W = rng.standard_normal((N, K)).astype(np.float32)
    W[0, :] = 0.0                                        # all-zero groups: keep columns (0,1)
    W[1, :] = 0.75                                       # all equal
    W[2, :8] = [1, -1, 1, -1, 2, 2, -2, 2]               # sign-mirrored ties
    W[3, :] = np.tile(np.array([0.0, 0.0, 1.0, 0.0], np.float32), K // 4)
    W[4, :] = rng.choice([-1.0, 0.0, 1.0], size=K)       # ternary rows
    W[5, :16] = np.float32(1e-30)                        # denormal-scale magnitudes
    r = _oracle_pack(W)
    # put exact halves in: w = 0.5*scale and 1.5*scale round to 0 resp. +-1 under half-to-even
    s = r["scale"]
    W[6, :4] = [0.5 * s, -0.5 * s, 1.5 * s, np.nextafter(np.float32(0.5 * s), np.float32(1))]
    r = _oracle_pack(W)
    for with_dense in (True, False):
        g = gpu_quantize_mask_pack(W, with_dense=with_dense)
        assert g["scale"] == r["scale"]
        assert np.array_equal(g["vals"], r["vals"])
        assert np.array_equal(g["meta"], r["meta"])
        if with_dense:
            assert np.array_equal(g["dense_q"], r["dense_q"])


def test_quantize_mask_pack_degenerate_scales():
    Z = np.zeros((128, 128), np.float32)
    r = oracle.quantize_mask_pack(Z)
    for with_dense in (True, False):
        g = gpu_quantize_mask_pack(Z, with_dense=with_dense)
        assert g["scale"] == r["scale"] == np.float32(1e-5)
        assert np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])
    tiny = np.full((128, 128), 7e-6, np.float32)          # gamma below the clamp, 0.7 -> rounds to 1
    r = oracle.quantize_mask_pack(tiny)
    for with_dense in (True, False):
        g = gpu_quantize_mask_pack(tiny, with_dense=with_dense)
        assert g["scale"] == r["scale"] and np.array_equal(g["vals"], r["vals"])
        if with_dense:
            assert np.array_equal(g["dense_q"], r["dense_q"])


@pytest.mark.parametrize("with_dense", [True, False])
@pytest.mark.parametrize("N,K,seed", [(256, 256, 30), (384, 2560, 31), (128, 6912, 32), (2048, 2560, 33)])
def test_quantize_mask_pack_bf16_masters(N, K, seed, with_dense):
    # master weights kept in bf16 (Sec. 2.2): the kernel reads bf16, the oracle gets the same real
    # numbers as fp32 -- bf16 -> fp32 is exact, so the results must agree bit for bit.  bf16 weights
    # produce many exact magnitude ties inside a group, which exercises the tie rule as well.
    bits = inputs.f32_to_bf16_bits(inputs.latent_weights(N, K, seed=seed))
    W = (bits.astype(np.uint32) << 16).view(np.float32).reshape(N, K)
    r = _oracle_pack(W)
    g = gpu_quantize_mask_pack(W, with_dense=with_dense, w_bf16_bits=bits)
    assert g["scale"] == r["scale"]
    assert np.array_equal(g["vals"], r["vals"])
    assert np.array_equal(g["meta"], r["meta"])
    if with_dense:
        assert np.array_equal(g["dense_q"], r["dense_q"])


def test_quantize_mask_pack_batched_mixed_master_dtypes():
    shapes = [(256, 512), (384, 256), (128, 1280)]
    jobs, refs = [], []
    for i, (N, K) in enumerate(shapes):
        W = inputs.latent_weights(N, K, seed=40 + i)
        if i % 2 == 0:
            bits = inputs.f32_to_bf16_bits(W)
            W = (bits.astype(np.uint32) << 16).view(np.float32).reshape(N, K)
            Wd = bf16_dev(bits)
        else:
            Wd = dev(W)
        refs.append(_oracle_pack(W))
        p = b.alloc_packed(N, K)
        jobs.append(dict(W=Wd, vals=p["vals"], meta=p["meta"], w_scale=p["w_scale"]))
    arr = b.make_pack_jobs(jobs)
    ws = torch.empty(b.sbn_batch_workspace_bytes(len(jobs)), dtype=torch.uint8, device="cuda")
    b.sbn_quantize_mask_pack_batched(arr, ws)
    b.sbn_check_status()
    from gpu_harness import _meta_offsets, _vals_offsets, untile
    for (N, K), j, r in zip(shapes, jobs, refs):
        assert np.float32(j["w_scale"].cpu().numpy()[0]) == r["scale"]
        assert np.array_equal(untile(j["vals"].cpu().numpy(), _vals_offsets(N, K)), r["vals"])
        assert np.array_equal(untile(j["meta"].cpu().numpy(), _meta_offsets(N, K)), r["meta"])


def _sampled_units(N, K):
    """The units the kernel's gamma estimate looks at (restated from the kernel's description:
    256 units -- 64 for matrices below 2^18 units -- unit s at s * stride + (s * 2654435761 mod 2^32 >> 8)
    mod stride)."""
    num_units = N * K // 128
    n_s = min(num_units, 64 if num_units < (1 << 18) else 256)
    stride = num_units // n_s
    sidx = np.arange(n_s, dtype=np.uint64)
    return (sidx * stride + (((sidx * 2654435761) & 0xFFFFFFFF) >> 8) % stride).astype(np.int64)


def test_quantize_mask_pack_misleading_sample():
    # the sampled units are 1000x smaller than the rest: the bracket around the estimated threshold
    # misses the exact one and the kernel has to take its second pass -- same bits as the oracle
    N, K = 1024, 2560
    W = inputs.latent_weights(N, K, seed=11)
    KB = K // 128
    for u in _sampled_units(N, K):
        n, kb = divmod(int(u), KB)
        W[n, kb * 128:(kb + 1) * 128] *= np.float32(1e-3)
    r = _oracle_pack(W)
    g = gpu_quantize_mask_pack(W, with_dense=False)
    assert g["scale"] == r["scale"]
    assert np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])
    # and the other way round: sampled units 1000x larger
    W = inputs.latent_weights(N, K, seed=12)
    for u in _sampled_units(N, K):
        n, kb = divmod(int(u), KB)
        W[n, kb * 128:(kb + 1) * 128] *= np.float32(1e3)
    r = _oracle_pack(W)
    g = gpu_quantize_mask_pack(W, with_dense=False)
    assert g["scale"] == r["scale"]
    assert np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])


@pytest.mark.parametrize("N,K", [(256, 512), (1024, 2560)])
def test_quantize_mask_pack_everything_near_the_threshold(N, K):
    # 15 of 16 groups keep two values within 1 % of half the scale (the rounding threshold), the
    # 16th carries the mass that puts gamma there: nearly every kept value is undecided until the
    # exact gamma is known.  The small case exercises a long fix-up list, the large one (139
    # units = 8340 listed values per CTA) overflows the list and falls back to the second pass.
    rng = np.random.default_rng(13)
    a = np.float32(0.01)
    G = N * K // 4
    groups = np.zeros((G, 4), np.float32)
    heavy = (np.arange(G) % 16) == 0
    f = heavy.mean()
    H = np.float32((3.0 + f) / f) * a
    jitter = (1.0 + 0.01 * rng.uniform(-1, 1, size=(G, 2))).astype(np.float32)
    sign = rng.choice(np.array([-1.0, 1.0], np.float32), size=(G, 2))
    groups[:, 1:3] = a * jitter * sign
    groups[heavy, 1:3] = H * sign[heavy]
    groups[:, 0] = a * np.float32(1e-3)
    W = groups.reshape(N, K)
    r = _oracle_pack(W)
    kept = r["vals"]
    assert 0.2 < np.count_nonzero(kept) / kept.size < 0.8, "the construction should split the kept values"
    g = gpu_quantize_mask_pack(W, with_dense=False)
    assert g["scale"] == r["scale"]
    assert np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])


# ---- the 6:8 pattern (Sec. 2.2): three overlapping windows turn it into 2:4 over K' = 3K/2 -------
def _decode68(g):
    """GPU 6:8 result -> (mask [N][K], W_eff [N][K]) after checking that it is a valid 2:4 form in
    which no original column is carried by two windows."""
    nib = np.stack([g["meta"] & 15, g["meta"] >> 4], axis=-1)
    assert ((nib & 3) < (nib >> 2)).all(), "metadata indices must be ascending within a group of four"
    w_eff_p, mask_p = oracle.unpack24(g["vals"], g["meta"])
    assert (mask_p.reshape(mask_p.shape[0], -1, 4).sum(-1) == 2).all()
    assert np.isin(g["vals"], (-1, 0, 1)).all()
    mask = fold68(mask_p)
    assert mask.max() <= 1, "a column is kept in two windows"
    return mask.astype(np.uint8), fold68(w_eff_p).astype(np.int8)


def _assert_pack68(W, g):
    r = oracle.quantize_mask_nm(W, 6, 8)
    mask, w_eff = _decode68(g)
    assert g["scale"] == r["scale"]
    assert np.array_equal(mask, r["mask"])
    assert np.array_equal(w_eff, r["w_eff"])
    return r


def _masters(W, bf16):
    """(W, the bf16 bit patterns or None): the weights as fp32 masters, or rounded to bf16 ones of the same values."""
    if not bf16:
        return W, None
    bits = inputs.f32_to_bf16_bits(W).reshape(W.shape)
    return (bits.astype(np.uint32) << 16).view(np.float32).reshape(W.shape), bits


@pytest.mark.parametrize("N,K,seed", [(128, 256, 50), (256, 512, 51), (384, 2560, 52), (128, 6912, 53), (2048, 2560, 54),
                                      (640, 1280, 55)])
def test_pack68_parity(N, K, seed):
    W = inputs.latent_weights(N, K, seed=seed)
    _assert_pack68(W, gpu_quantize_mask_pack68(W))


def test_pack68_bf16_masters_and_ties():
    bits = inputs.f32_to_bf16_bits(inputs.latent_weights(384, 2560, seed=56))
    W = (bits.astype(np.uint32) << 16).view(np.float32).reshape(384, 2560)
    _assert_pack68(W, gpu_quantize_mask_pack68(W, w_bf16_bits=bits))


@pytest.mark.parametrize("scale", [1e-36, 1e-38, 1e-39])
def test_pack_bf16_masters_of_tiny_magnitude(scale):
    # magnitudes whose differences are subnormal: the selection subtracts, and no difference may be lost
    bits = inputs.f32_to_bf16_bits((inputs.latent_weights(256, 512, seed=61) * np.float32(scale)).astype(np.float32))
    W = (bits.astype(np.uint32) << 16).view(np.float32).reshape(256, 512)
    _assert_pack68(W, gpu_quantize_mask_pack68(W, w_bf16_bits=bits))
    r, g = _oracle_pack(W), gpu_quantize_mask_pack(W, with_dense=False, w_bf16_bits=bits)
    assert g["scale"] == r["scale"] and np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])


@pytest.mark.parametrize("N,K", [(256, 512), (4096, 4096)])      # 4096 rows: the CTAs exchange what they have seen under way
@pytest.mark.parametrize("special", [(0x7F80,), (0xFF80,), (0x7FC0,), (0x7F80, 0xFFC0, 0xFF80), (0x7F7F, 0xFF7F)])
def test_pack68_bf16_masters_show_what_is_not_finite(special, N, K):
    # bf16 masters with infinities, NaN or the largest finite magnitude give what fp32 masters of the same values do: an infinite weight
    # makes the scale infinite
    bits = inputs.f32_to_bf16_bits(inputs.latent_weights(N, K, seed=62)).reshape(N, K)
    for i, v in enumerate(special):
        bits.reshape(-1)[(104729 * (i + 1)) % bits.size] = v
        bits[5 + i, 8:16] = v                                  # a whole group
        bits[N - 1, K - 9 + i] = v
    W = (bits.astype(np.uint32) << 16).view(np.float32).reshape(N, K)
    f, g = gpu_quantize_mask_pack68(W), gpu_quantize_mask_pack68(W, w_bf16_bits=bits)
    assert f["scale"].view(np.uint32) == g["scale"].view(np.uint32)
    assert np.array_equal(f["vals"], g["vals"]) and np.array_equal(f["meta"], g["meta"])
    mean = np.abs(W.astype(np.float64)).mean()
    assert np.isnan(mean) or g["scale"] == np.float32(mean)


def _first_look(W, bf16):
    """What a single call without a hint does to its bracket around the mean |w| while it runs, on the host: (the sample's bracket,
    the bracket from the means that the CTAs have seen after their teams' first stages)."""
    units = np.abs(W.reshape(-1, 128).astype(np.float64))
    grid = min(torch.cuda.get_device_properties(0).multi_processor_count, 148)
    per = -(-len(units) // grid)
    assert per >= 700 and len(units) < 1 << 18                  # long enough for it; the sample of 64 units
    s = np.arange(64, dtype=np.uint64)
    stride = len(units) // 64
    sample = units[(s * stride + (((s * 2654435761) & 0xFFFFFFFF) >> np.uint64(8)) % stride).astype(np.int64)].mean()
    seen = min(per, 160 if bf16 else 80)                        # two teams' stages of 20 KB
    means = np.array([units[r * per:min(len(units), r * per + seen)].mean() for r in range(grid) if r * per < len(units)])
    b = 5.0 * means.std() / np.sqrt(len(means)) / means.mean() + 0.001
    assert b < 0.04
    return (sample * 0.96, sample * 1.04), (means.mean() * (1.0 - b), means.mean() * (1.0 + b))


# factor: the first 224 units of every CTA's range are smaller than the rest by this
@pytest.mark.parametrize("factor,narrows,holds", [(1.0, True, True), (0.98, True, False), (0.9, False, False)])
@pytest.mark.parametrize("bf16", [False, True])
def test_pack_long_matrix_narrows_its_bracket(bf16, factor, narrows, holds):
    # ranges long enough for the CTAs to tell each other what their first stages say about the mean: the narrowed bracket holds, or it
    # misses the mean (values decided with the wide bracket before it, the exact second pass after it), or it lies outside the sample's
    N, K = 4096, 4096
    W = inputs.latent_weights(N, K, seed=61)
    units = W.reshape(-1, 128)
    grid = min(torch.cuda.get_device_properties(0).multi_processor_count, 148)
    per = -(-len(units) // grid)
    for r in range(grid):
        units[r * per:r * per + 224] *= np.float32(factor)
    W, bits = _masters(W, bf16)
    wide, narrow = _first_look(W, bf16)
    lo, hi = max(wide[0], narrow[0]), min(wide[1], narrow[1])
    mean = np.abs(W.astype(np.float64)).mean()
    assert wide[0] < mean < wide[1]
    assert (lo < hi) == narrows and (not narrows or (lo < mean < hi) == holds)
    r, g = _oracle_pack(W), gpu_quantize_mask_pack(W, with_dense=False, w_bf16_bits=bits)
    assert g["scale"] == r["scale"] and np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])
    _assert_pack68(W, gpu_quantize_mask_pack68(W, w_bf16_bits=bits))


@pytest.mark.parametrize("bf16", [False, True])
def test_pack68_every_kept_set(bf16):
    # all 28 ways of dropping two columns of eight, each with distinct magnitudes and with ties at
    # the boundary (the dropped pair equal to a kept column: the lower column must win)
    N, K = 128, 256
    rng = np.random.default_rng(57)
    W = rng.uniform(1.0, 2.0, size=(N, K)).astype(np.float32) * rng.choice(np.array([-1, 1], np.float32), size=(N, K))
    pairs = [(i, j) for i in range(8) for j in range(i + 1, 8)]
    grp = W.reshape(N, K // 8, 8)
    for idx, (i, j) in enumerate(pairs):
        grp[idx, :, i] *= np.float32(0.01)
        grp[idx, :, j] *= np.float32(0.02)
        grp[idx + 28, :, :] = np.float32(1.0)                 # all equal but two smaller ones
        grp[idx + 28, :, i] = np.float32(0.5)
        grp[idx + 28, :, j] = np.float32(0.5)
        grp[idx + 56, :, :] = np.float32(-0.5)                # ties between dropped and kept columns
        grp[idx + 56, :, i] = np.float32(0.75)
        grp[idx + 56, :, j] = np.float32(-0.75)
    W[120, :] = 0.0                                           # all-zero groups: columns 0..5 kept
    W[121, :] = 0.3
    W, bits = _masters(W, bf16)
    _assert_pack68(W, gpu_quantize_mask_pack68(W, w_bf16_bits=bits))


@pytest.mark.parametrize("bf16", [False, True])
def test_pack68_misleading_sample_and_list_overflow(bf16):
    N, K = 1024, 2560
    W = inputs.latent_weights(N, K, seed=58)
    KB = K // 128
    for u in _sampled_units(N, K):
        n, kb = divmod(int(u), KB)
        W[n, kb * 128:(kb + 1) * 128] *= np.float32(1e-3)
    W, bits = _masters(W, bf16)
    _assert_pack68(W, gpu_quantize_mask_pack68(W, w_bf16_bits=bits))
    # nearly every kept value within 1 % of the rounding threshold: the list overflows
    rng = np.random.default_rng(59)
    a = np.float32(0.01)
    G = N * K // 8
    groups = (a * (1.0 + 0.01 * rng.uniform(-1, 1, size=(G, 8)))).astype(np.float32)
    groups *= rng.choice(np.array([-1.0, 1.0], np.float32), size=(G, 8))
    heavy = (np.arange(G) % 16) == 0
    # mean |w| must come out near 2a for thr = scale / 2 to sit at a: heavy groups carry the rest
    groups[heavy] *= np.float32(17.0)
    W, bits = _masters(groups.reshape(N, K), bf16)
    r = _assert_pack68(W, gpu_quantize_mask_pack68(W, w_bf16_bits=bits))
    frac = np.count_nonzero(r["w_eff"]) / (0.75 * r["w_eff"].size)
    assert 0.2 < frac < 0.9, "the construction should split the kept values"
    # a short list (small matrix): the fix-up route
    small = None if bits is None else bits[:256, :512].copy()
    _assert_pack68(W[:256, :512].copy(), gpu_quantize_mask_pack68(W[:256, :512].copy(), w_bf16_bits=small))


@pytest.mark.parametrize("bf16", [False, True])
def test_pack68_degenerate_scales(bf16):
    Z, bits = _masters(np.zeros((128, 256), np.float32), bf16)
    g = gpu_quantize_mask_pack68(Z, w_bf16_bits=bits)
    assert g["scale"] == np.float32(1e-5)
    _assert_pack68(Z, g)
    tiny, bits = _masters(np.full((128, 256), 7e-6, np.float32), bf16)
    _assert_pack68(tiny, gpu_quantize_mask_pack68(tiny, w_bf16_bits=bits))


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("in_place", [False, True])
def test_pack68_flip_count(in_place, bf16):
    W = inputs.latent_weights(256, 2560, seed=60)
    Wp, bits_p = _masters(inputs.perturb_weights(W, seed=61, sigma=1e-4), bf16)
    W, bits = _masters(W, bf16)
    g0 = gpu_quantize_mask_pack68(W, w_bf16_bits=bits)
    r0 = _assert_pack68(W, g0)
    g1 = gpu_quantize_mask_pack68(Wp, prev_meta=g0["meta"], in_place=in_place, w_bf16_bits=bits_p)
    r1 = _assert_pack68(Wp, g1)
    expected = oracle.flip_count(r0["mask"], r1["mask"])
    assert expected > 0
    assert g1["flips"] == expected
    assert gpu_quantize_mask_pack68(W, prev_meta=g0["meta"], w_bf16_bits=bits)["flips"] == 0


def test_pack68_rejects_what_it_cannot_do():
    p = b.alloc_packed(128, 256, n_keep=6, m_group=8)
    W = dev(np.zeros((128, 256), np.float32))
    dense = torch.empty((128, 256), dtype=torch.int8, device="cuda")
    with pytest.raises(b.SbnError):
        b.sbn_quantize_mask_pack(W, p["vals"], p["meta"], p["w_scale"], p["ws"], dense_q=dense, n_keep=6, m_group=8)
    W2 = dev(np.zeros((128, 384), np.float32))                    # K' = 576 is not a multiple of 128
    with pytest.raises(b.SbnError):
        b.sbn_quantize_mask_pack(W2, p["vals"], p["meta"], p["w_scale"], p["ws"], n_keep=6, m_group=8)
    assert b.sbn_expanded_k(256, 6, 8) == 384 and b.sbn_expanded_k(384, 6, 8) == 0
    assert b.sbn_expanded_k(384, 2, 4) == 384 and b.sbn_expanded_k(256, 5, 8) == 0


@pytest.mark.parametrize("T,K", [(64, 256), (1, 2560), (5, 512), (67, 2560), (33, 6912), (19, 11008), (300, 4096),
                                 (3, 32768)])
def test_quant_act_expand68_parity(T, K):
    bits = inputs.activations_bf16(T, K, seed=T + K, token_lognormal_sigma=1.0)
    xq_ref, s_ref = oracle.quant_act(bits)
    xq, s = gpu_quant_act_expand68(bits)
    assert np.array_equal(s.cpu().numpy(), s_ref)
    assert np.array_equal(xq_to_numpy(xq, T, 3 * K // 2), xq_ref[:, expand68_columns(K)])


@pytest.mark.parametrize("T,K", [(64, 256), (1, 2560), (67, 2560), (33, 6912), (19, 11008), (300, 4096), (3, 16384)])
def test_norm_quant_act_expand68_parity(T, K):
    bits = inputs.activations_bf16(T, K, seed=T + K + 5, token_lognormal_sigma=1.0)
    gain = (1.0 + 0.1 * np.random.default_rng(K).standard_normal(K)).astype(np.float32)
    r = oracle.norm_quant_act(bits, gain, 1e-6)
    xq, s = gpu_norm_quant_act(bits, gain, 1e-6, expand68=True)
    got = xq_to_numpy(xq, T, 3 * K // 2)
    ref = r["xq"][:, expand68_columns(K)]
    assert (~r["near_tie"]).all(), "a row's mean square sits on an fp32 rounding boundary for this seed"
    assert np.array_equal(s.cpu().numpy(), r["a_scale"])
    assert np.array_equal(got, ref)


SPARSE68_SHAPES = [(64, 256, 256), (1, 128, 512), (5, 128, 256), (130, 384, 512), (300, 256, 2560), (64, 128, 6912),
                   (700, 512, 1280), (1100, 640, 2560)]


@pytest.mark.parametrize("T,N,K", SPARSE68_SHAPES)
def test_sparse68_layer_parity(T, N, K):
    # whole 6:8 layer: pack -> expanded activations -> the unchanged sparse GEMM over K' columns;
    # the accumulators must be those of the plain integer matmul with the oracle's 6:8 W_eff
    W = inputs.latent_weights(N, K, seed=T + N + K)
    bits = inputs.activations_bf16(T, K, seed=T + N + K + 1, token_lognormal_sigma=0.5)
    r = oracle.quantize_mask_nm(W, 6, 8)
    xq_ref, s_ref = oracle.quant_act(bits)
    y_ref, acc_ref = oracle.nm_bitlinear(xq_ref, s_ref, r["w_eff"], r["scale"])
    g = gpu_quantize_mask_pack68(W)
    xq, a_scale = gpu_quant_act_expand68(bits)
    y, acc = gpu_gemm(True, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)
    yb, _ = gpu_gemm(True, xq, a_scale, g["dev"], out_dtype=torch.bfloat16, want_acc=False)
    assert np.abs(bf16_tensor_bits(yb).astype(np.int32) - oracle.f32_to_bf16_bits(y_ref).astype(np.int32)).max() <= 1


def test_worked_example_not_the_negative_control():
    # the hand-worked row of tests/golden tiled to a legal shape: quant-then-mask with the dense
    # gamma, never the mask-then-quant answer
    row = np.array([1, 1, 0.9, 0.9, 0.25, 0.25, 0, 0], np.float32)
    W = np.tile(row, (128, 16))
    g = gpu_quantize_mask_pack(W)
    assert g["scale"] == np.float32(0.5375)
    assert (g["vals"].reshape(128, -1, 4) == np.array([1, 1, 0, 0], np.int8)).all()
    assert (g["meta"] == 68).all()


@pytest.mark.parametrize("in_place", [False, True])
def test_flip_count_parity(in_place):
    W = inputs.latent_weights(256, 2560, seed=7)
    Wp = inputs.perturb_weights(W, seed=8, sigma=1e-4)
    r0 = _oracle_pack(W)
    r1 = _oracle_pack(Wp)
    g = gpu_quantize_mask_pack(Wp, with_dense=False, prev_meta=r0["meta"], in_place=in_place)
    assert np.array_equal(g["meta"], r1["meta"]) and np.array_equal(g["vals"], r1["vals"])
    assert g["flips"] == oracle.flip_count(r0["mask"], r1["mask"])
    same = gpu_quantize_mask_pack(W, with_dense=False, prev_meta=r0["meta"])
    assert same["flips"] == 0


def test_quantize_mask_pack_batched_matches_single_calls():
    # one launch for several matrices of different shapes (with and without dense W_q / flip count):
    # every job must reproduce the single call -- and the oracle -- bit for bit
    shapes = [(256, 2560), (640, 256), (128, 128), (384, 1280), (2560, 640)]
    Ws = [inputs.latent_weights(N, K, seed=40 + i, sigma=0.02 * (i + 1)) for i, (N, K) in enumerate(shapes)]
    refs = [_oracle_pack(W) for W in Ws]
    prevs = [oracle.quantize_mask_pack(inputs.perturb_weights(W, seed=60 + i, sigma=2e-3))["meta"] for i, W in enumerate(Ws)]
    jobs, singles = [], []
    for i, W in enumerate(Ws):
        N, K = W.shape
        use_prev, use_dense = (i % 2 == 0), (i % 3 != 0)
        bufs = b.alloc_packed(N, K, with_dense=use_dense)
        job = dict(W=dev(W), vals=bufs["vals"], meta=bufs["meta"], w_scale=bufs["w_scale"], dense_q=bufs.get("dense_q"))
        if use_prev:
            from gpu_harness import tile_meta
            job["prev_meta"] = dev(tile_meta(prevs[i]).reshape(N, K // 8))
            job["flip_bits"] = torch.full((1,), 777, dtype=torch.int64, device="cuda")
        jobs.append(job)
        singles.append(gpu_quantize_mask_pack(W, with_dense=use_dense, prev_meta=prevs[i] if use_prev else None))
    arr = b.make_pack_jobs(jobs)
    ws = torch.empty(b.sbn_batch_workspace_bytes(len(jobs)), dtype=torch.uint8, device="cuda")
    for _ in range(2):                                        # twice: the second run meets stale slots
        b.sbn_quantize_mask_pack_batched(arr, ws)
    b.sbn_check_status()
    from gpu_harness import _meta_offsets, _vals_offsets, untile
    for i, (job, one, r) in enumerate(zip(jobs, singles, refs)):
        N, K = Ws[i].shape
        assert np.float32(job["w_scale"].cpu().numpy()[0]) == r["scale"] == one["scale"]
        assert np.array_equal(untile(job["vals"].cpu().numpy(), _vals_offsets(N, K)), r["vals"])
        assert np.array_equal(untile(job["meta"].cpu().numpy(), _meta_offsets(N, K)), r["meta"])
        assert np.array_equal(job["vals"].cpu().numpy(), one["dev"]["vals"].cpu().numpy())
        if job.get("dense_q") is not None:
            assert np.array_equal(job["dense_q"].cpu().numpy(), one["dev"]["dense_q"].cpu().numpy())
        if "flip_bits" in job:
            want = oracle.flip_count(oracle.unpack24(r["vals"], prevs[i])[1], r["mask"])
            assert int(job["flip_bits"].item()) == want == one["flips"]


def test_quantize_mask_pack_random_batches_against_the_oracle_and_single_calls():
    # seeded random batches: 1..7 matrices of mixed shapes (fewer units than CTAs, ragged last stages, ranges
    # of several stages), fp32 and bf16 masters, Gaussian and heavy-tailed, no hints / exact hints / hints
    # inside and outside the bracket / hints on some jobs only, each batch launched twice on one workspace.
    # Every job must carry the oracle's bits (matrices the oracle flags as near-ties excepted) and the
    # single call's bits.
    import random
    rng = random.Random(20260305)
    Ns, Ks = [128, 256, 384, 640, 2560], [128, 256, 1280, 2560, 6912]
    checked = 0
    for it in range(24):
        count = rng.randint(1, 7)
        jobs, refs, singles, shapes = [], [], [], []
        mode = rng.choice(["none", "good", "off", "mixed"])
        for i in range(count):
            N, K = rng.choice(Ns), rng.choice(Ks)
            W = inputs.latent_weights(N, K, seed=7000 + 16 * it + i, sigma=rng.choice([0.02, 0.5, 1e-3]))
            if rng.random() < 0.2:
                W = inputs.latent_weights(N, K, seed=7500 + 16 * it + i, sigma=0.015, outlier_prob=0.05, outlier_mult=10.0)
            as_bf16 = rng.random() < 0.3
            if as_bf16:
                bits = inputs.f32_to_bf16_bits(W)
                W = (bits.astype(np.uint32) << 16).view(np.float32).reshape(N, K)
                Wd = bf16_dev(bits)
            else:
                Wd = dev(W)
            r = oracle.quantize_mask_pack(W)
            one = b.alloc_packed(N, K)
            b.sbn_quantize_mask_pack(Wd, one["vals"], one["meta"], one["w_scale"], one["ws"])
            bufs = b.alloc_packed(N, K)
            job = dict(W=Wd, vals=bufs["vals"], meta=bufs["meta"], w_scale=bufs["w_scale"])
            if mode in ("good", "off") or (mode == "mixed" and rng.random() < 0.5):
                f = 1.0 if mode != "off" else rng.choice([1.004, 0.99, 1.5, 0.0])
                job["gamma_hint"] = torch.tensor([float(r["scale"]) * f], dtype=torch.float32, device="cuda")
            jobs.append(job); refs.append(r); singles.append(one); shapes.append((N, K))
        arr = b.make_pack_jobs(jobs)
        ws = torch.empty(b.sbn_batch_workspace_bytes(count), dtype=torch.uint8, device="cuda")
        for _ in range(2):
            b.sbn_quantize_mask_pack_batched(arr, ws)
        b.sbn_check_status()
        for job, r, one, (N, K) in zip(jobs, refs, singles, shapes):
            for key in ("vals", "meta", "w_scale"):
                assert torch.equal(job[key], one[key]), (it, N, K, mode, key)
            if r["near_tie"]:
                continue
            vals, meta = gpu_unpack_canonical(job, N, K)
            assert np.float32(job["w_scale"].cpu().numpy()[0]) == r["scale"]
            assert np.array_equal(vals, r["vals"]) and np.array_equal(meta, r["meta"])
            checked += 1
    assert checked > 60


def test_quantize_mask_pack_full_size_in_the_bench_configuration():
    # the four BitNet-2B-shaped matrices exactly as bench.py packs them: one batched launch, no
    # dense output (the single-pass route); every byte against the oracle
    from gpu_harness import _meta_offsets, _vals_offsets, untile
    Ws = [inputs.latent_weights(N, K, seed=1 + i) for i, (_, K, N) in enumerate(inputs.SHAPES_2B)]
    jobs = []
    for W in Ws:
        N, K = W.shape
        bufs = b.alloc_packed(N, K)
        jobs.append(dict(W=dev(W), vals=bufs["vals"], meta=bufs["meta"], w_scale=bufs["w_scale"]))
    arr = b.make_pack_jobs(jobs)
    ws = torch.empty(b.sbn_batch_workspace_bytes(len(jobs)), dtype=torch.uint8, device="cuda")
    b.sbn_quantize_mask_pack_batched(arr, ws)
    b.sbn_check_status()
    for W, job in zip(Ws, jobs):
        N, K = W.shape
        r = _oracle_pack(W)
        assert np.float32(job["w_scale"].cpu().numpy()[0]) == r["scale"]
        assert np.array_equal(untile(job["vals"].cpu().numpy(), _vals_offsets(N, K)), r["vals"])
        assert np.array_equal(untile(job["meta"].cpu().numpy(), _meta_offsets(N, K)), r["meta"])


def test_quant_act_full_size():
    x = inputs.activations_bf16(4096, 6912, seed=14, token_lognormal_sigma=0.5)
    xq_ref, s_ref = oracle.quant_act(x)
    xq, s = gpu_quant_act(x)
    assert np.array_equal(s.cpu().numpy(), s_ref)
    assert np.array_equal(xq_to_numpy(xq, 4096, 6912), xq_ref)


# ------------------------------------------------------------------------------------------------
# part 3 and the dense baseline
# ------------------------------------------------------------------------------------------------
def _layer_case(T, N, K, seed, sigma=0.02):
    W = inputs.latent_weights(N, K, seed=seed, sigma=sigma)
    x = inputs.activations_bf16(T, K, seed=seed + 1000)
    r = _oracle_pack(W)
    xq_ref, s_ref = oracle.quant_act(x)
    g = gpu_quantize_mask_pack(W)
    assert np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])
    xq, a_scale = gpu_quant_act(x)
    return r, xq_ref, s_ref, g, xq, a_scale


GEMM_SHAPES = [(64, 256, 256), (1, 128, 128), (5, 128, 256), (130, 384, 512), (300, 256, 2560), (64, 128, 6912)]


@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("T,N,K", GEMM_SHAPES)
def test_gemm_parity(sparse, T, N, K):
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=T + N + K)
    if sparse:
        y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    else:
        y_ref, acc_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"])
    y, acc = gpu_gemm(sparse, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)


def _random_gemm_shapes(count, seed):
    """Seeded shapes across the dispatcher's regimes (few tokens: single-CTA tiles, split K in clusters;
    hundreds to thousands of tokens: CTA pairs with one or two M-tiles), sized for the CPU oracle."""
    import random
    rng = random.Random(seed)
    Ts = [1, 3, 8, 17, 31, 64, 100, 200, 255, 300, 511, 777, 1024, 1500, 2048]
    Ns = [128, 256, 384, 640, 1024, 2560]
    Ks = [128, 256, 384, 1280, 2560, 6912]
    out = []
    while len(out) < count:
        T, N, K = rng.choice(Ts), rng.choice(Ns), rng.choice(Ks)
        if T * N * K <= 6e8 and (T, N, K) not in out:
            out.append((T, N, K))
    return out


@pytest.mark.parametrize("T,N,K", _random_gemm_shapes(16, seed=20260306))
def test_gemm_parity_random_shapes_with_the_plan_the_library_picks(T, N, K):
    # whatever kernel and tile the dispatcher chooses for the shape: accumulators exact, outputs within tolerance
    # (fp32 out with the accumulator dump, then bf16 out alone: the register-packed epilogue of the pair kernel)
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=3 * T + 5 * N + 7 * K)
    y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    y, acc = gpu_gemm(True, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)
    yb, _ = gpu_gemm(True, xq, a_scale, g["dev"], out_dtype=torch.bfloat16, want_acc=False)
    ref_bits = oracle.f32_to_bf16_bits(y_ref).astype(np.int32)
    got_bits = bf16_tensor_bits(yb).astype(np.int32)
    # same sign assumed (values are not within one ulp of zero); 1 ulp = 1 step of the pattern
    assert np.abs(got_bits - ref_bits).max() <= 1


@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("tile", [64, 128, 256])
def test_gemm_parity_every_token_tile(sparse, tile):
    T, N, K = 333, 256, 1280
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=tile)
    b.sbn_set_gemm_tuning(tile, 1)
    if sparse:
        y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    else:
        y_ref, acc_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"])
    y, acc = gpu_gemm(sparse, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)


PAIR_CASES = [  # (T, N, K, BN): CTA-pair kernel, forced tile widths incl. ragged T and odd N/128
    (333, 128, 256, 64), (333, 256, 128, 32), (40, 384, 512, 32), (500, 640, 384, 160),
    (700, 1024, 1280, 224), (257, 1152, 2560, 96), (1000, 512, 6912, 240), (530, 256, 256, 256),
    (490, 384, 640, 240), (300, 256, 384, 48), (241, 512, 256, 240), (1000, 640, 512, 176),
]


@pytest.mark.parametrize("mt", [2, 1])          # M-tiles per CTA: 512- or 256-feature pair tiles (the latter double-buffered)
@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("T,N,K,bn", PAIR_CASES)
def test_gemm_parity_pair_kernel(sparse, T, N, K, bn, mt):
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=bn + T)
    b.sbn_set_gemm_tuning(-bn, 1 if mt == 1 else 0)
    if sparse:
        y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    else:
        y_ref, acc_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"])
    y, acc = gpu_gemm(sparse, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)
    yb, _ = gpu_gemm(sparse, xq, a_scale, g["dev"], out_dtype=torch.bfloat16, want_acc=False)
    ref_bits = oracle.f32_to_bf16_bits(y_ref).astype(np.int32)
    assert np.abs(bf16_tensor_bits(yb).astype(np.int32) - ref_bits).max() <= 1


def _random_gemm_shapes(n, seed):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(n):
        T = int(rng.choice([1, 2, 3, 7, 15, 16, 17, 31, 33, 63, 64, 65, 100, 127, 128, 129, 200, 255, 256, 257, 300,
                            511, 513, 700, 1023, 1100]))
        N = 128 * int(rng.integers(1, 9))
        K = 128 * int(rng.integers(1, 25))
        out.append((T, N, K))
    return out


@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("T,N,K", _random_gemm_shapes(24, seed=2024))
def test_gemm_parity_automatic_dispatch_random_shapes(sparse, T, N, K):
    # whatever kernel, tile and split the dispatcher picks for the shape: accumulators bit-exact,
    # outputs within tolerance
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=T + N + K)
    if sparse:
        y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    else:
        y_ref, acc_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"])
    y, acc = gpu_gemm(sparse, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)
    yb, _ = gpu_gemm(sparse, xq, a_scale, g["dev"], out_dtype=torch.bfloat16, want_acc=False)
    ref_bits = oracle.f32_to_bf16_bits(y_ref).astype(np.int32)
    assert np.abs(bf16_tensor_bits(yb).astype(np.int32) - ref_bits).max() <= 1


CLUSTER_CASES = [  # (T, N, K, token tile, cluster size): split-K reduced in distributed shared memory
    (64, 256, 2560, 64, 4), (1, 128, 256, 64, 2), (7, 256, 640, 64, 4),      # 5 k-blocks over 4 CTAs: one empty slice
    (100, 384, 6912, 64, 8), (130, 256, 1280, 128, 8), (200, 128, 384, 128, 2), (33, 512, 128, 64, 8),   # one k-block
    (257, 256, 2560, 128, 4),
    (16, 256, 2560, 32, 4), (1, 128, 256, 32, 2), (31, 384, 6912, 32, 8), (32, 128, 1280, 32, 4), (45, 256, 640, 32, 4),
    (70, 128, 2560, 32, 2),
    (16, 256, 2560, 32, 3), (31, 128, 896, 32, 3), (64, 384, 1280, 64, 3), (50, 128, 4096, 64, 3), (130, 256, 1280, 128, 3),
    (1, 128, 384, 32, 3),
]


@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("T,N,K,tile,cluster", CLUSTER_CASES)
def test_gemm_parity_cluster_split_k(sparse, T, N, K, tile, cluster):
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=cluster + T)
    b.sbn_set_gemm_tuning(tile, -cluster)
    if sparse:
        y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    else:
        y_ref, acc_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"])
    y, acc = gpu_gemm(sparse, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)
    yb, _ = gpu_gemm(sparse, xq, a_scale, g["dev"], out_dtype=torch.bfloat16, want_acc=False)
    ref_bits = oracle.f32_to_bf16_bits(y_ref).astype(np.int32)
    assert np.abs(bf16_tensor_bits(yb).astype(np.int32) - ref_bits).max() <= 1


# Wide token tiles split over clusters: one token in the last tile (CTAs that own none), unequal shares, tiles of the least
# and the greatest width, K-blocks that do not divide by the cluster, one block per CTA, more blocks than stages.
WIDE_CASES = [(81, 128, 512, 80, 4), (65, 256, 384, 80, 3), (201, 256, 1280, 112, 2), (256, 128, 1664, 256, 4), (255, 256, 2560, 256, 2),
              (160, 128, 2176, 160, 3), (300, 128, 768, 208, 6), (97, 384, 256, 112, 2),
              (81, 128, 128, 80, 1), (256, 256, 1664, 256, 1), (300, 128, 2560, 160, 1), (129, 384, 1152, 128, 1), (500, 128, 384, 176, 1)]


@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("T,N,K,tile,cluster", WIDE_CASES)
def test_gemm_parity_cluster_wide_tiles(sparse, T, N, K, tile, cluster):
    test_gemm_parity_cluster_split_k(sparse, T, N, K, tile, cluster)


@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("split", [2, 5, 10])
def test_gemm_parity_split_k(sparse, split):
    T, N, K = 7, 256, 2560
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=split)
    b.sbn_set_gemm_tuning(0, split)
    if sparse:
        y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    else:
        y_ref, acc_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"])
    y, acc = gpu_gemm(sparse, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)


@pytest.mark.parametrize("sparse", [True, False])
def test_gemm_bias_and_bf16_output(sparse):
    T, N, K = 70, 256, 512
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=77)
    bias = np.random.default_rng(78).standard_normal(N).astype(np.float32)
    if sparse:
        y_ref, _ = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"], bias=bias)
    else:
        y_ref, _ = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"], bias=bias)
    y, _ = gpu_gemm(sparse, xq, a_scale, g["dev"], bias=dev(bias))
    _assert_y(y_to_f32_numpy(y), y_ref)
    yb, _ = gpu_gemm(sparse, xq, a_scale, g["dev"], out_dtype=torch.bfloat16, bias=dev(bias))
    ref_bits = oracle.f32_to_bf16_bits(y_ref).astype(np.int32)
    got_bits = bf16_tensor_bits(yb).astype(np.int32)
    # same sign assumed (values are not within one ulp of zero); 1 ulp = 1 step of the pattern
    assert np.abs(got_bits - ref_bits).max() <= 1


@pytest.mark.parametrize("T,N,K", [(200, 6272, 1280), (777, 1664, 1280), (2000, 1920, 6912)])
def test_gemm_dense_plan_of_unsplit_wide_tiles(T, N, K):
    # the library's own choice: accumulators against a product in fp64 (exact), outputs bit for bit in the documented order of roundings
    assert b.sbn_plan_gemm(False, T, N, K)[0] == 4
    g = gpu_quantize_mask_pack(inputs.latent_weights(N, K, seed=T))
    xq, a_scale = gpu_quant_act(inputs.activations_bf16(T, K, seed=T + 1, token_lognormal_sigma=0.5))
    codes = dev(xq_to_numpy(xq, T, K)).double()
    acc_ref = (codes @ dev(g["dense_q"]).double().T).to(torch.int32)
    bias = torch.randn(N, device="cuda", generator=torch.Generator("cuda").manual_seed(K))
    y_ref = acc_ref.float() * (a_scale * g["dev"]["w_scale"])[:, None]
    for out_dtype, with_bias, want_acc in [(torch.float32, True, True), (torch.float32, False, False), (torch.bfloat16, True, False)]:
        y, acc = gpu_gemm(False, xq, a_scale, g["dev"], out_dtype=out_dtype, bias=bias if with_bias else None, want_acc=want_acc)
        if want_acc:
            assert torch.equal(acc, acc_ref)
        assert torch.equal(y, (y_ref + bias if with_bias else y_ref).to(out_dtype))


def test_exact_integer_layer_on_gpu():
    # integer activations and ternary weights: no quantisation error anywhere, acc is the exact
    # integer product and sparse == dense when the pruned entries are zeros
    rng = np.random.default_rng(9)
    T, N, K = 40, 128, 256
    X = rng.integers(-127, 128, size=(T, K)).astype(np.float32)
    X[:, 0] = 127
    tern = np.zeros((N, K), np.int8)
    for g_ in range(K // 4):                                # at most two non-zeros per group
        cols = rng.permuted(np.tile(np.arange(4), (N, 1)), axis=1)[:, :2]
        tern[np.arange(N)[:, None], 4 * g_ + cols] = rng.choice([-1, 1], size=(N, 2))
    W = tern.astype(np.float32) * np.float32(0.5)
    g = gpu_quantize_mask_pack(W)
    xq, a_scale = gpu_quant_act(inputs.f32_to_bf16_bits(X))
    ys, acc_s = gpu_gemm(True, xq, a_scale, g["dev"])
    yd, acc_d = gpu_gemm(False, xq, a_scale, g["dev"])
    ref = X.astype(np.int64) @ tern.astype(np.int64).T
    assert np.array_equal(acc_s.cpu().numpy(), ref)
    assert np.array_equal(acc_d.cpu().numpy(), ref)
    assert torch.equal(ys, yd)


# ------------------------------------------------------------------------------------------------
# full-size shapes in the launch configuration the benchmark times, on sampled outputs
# ------------------------------------------------------------------------------------------------
FULL = [("qkv", 4096, 2560, 3840, 0.02, 0.0, 0.0), ("down", 4096, 6912, 2560, 0.02, 0.0, 0.0),
        ("down_7b", 8192, 11008, 4096, 0.015, 0.05, 0.5)]


@pytest.mark.parametrize("name,T,K,N,sigma,outl,logn", FULL)
def test_full_size_sampled(name, T, K, N, sigma, outl, logn):
    W = inputs.latent_weights(N, K, seed=21, sigma=sigma, outlier_prob=outl)
    x = inputs.activations_bf16(T, K, seed=22, token_lognormal_sigma=logn)
    r = _oracle_pack(W)
    xq_ref, s_ref = oracle.quant_act(x)
    g = gpu_quantize_mask_pack(W)
    assert g["scale"] == r["scale"]
    assert np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])
    assert np.array_equal(g["dense_q"], r["dense_q"])
    xq, a_scale = gpu_quant_act(x)
    assert np.array_equal(xq_to_numpy(xq, T, K), xq_ref) and np.array_equal(a_scale.cpu().numpy(), s_ref)
    t_idx, n_idx = inputs.sample_positions(T, N, 4096, seed=23)
    # corners and tile borders as well
    t_idx[:4] = [0, T - 1, 0, T - 1]
    n_idx[:4] = [0, 0, N - 1, N - 1]
    for sparse in (True, False):
        y, acc = gpu_gemm(sparse, xq, a_scale, g["dev"], out_dtype=torch.bfloat16)
        if sparse:
            acc_ref = oracle.acc_packed_sampled(xq_ref, r["vals"], r["meta"], t_idx, n_idx)
        else:
            acc_ref = oracle.acc_dense_sampled(xq_ref, r["dense_q"], t_idx, n_idx)
        acc_s = acc.cpu().numpy()[t_idx, n_idx]
        assert np.array_equal(acc_s, acc_ref)
        y_ref = oracle.dequant(acc_ref.reshape(-1, 1), r["scale"], s_ref[t_idx]).ravel()
        ref_bits = oracle.f32_to_bf16_bits(y_ref).astype(np.int32)
        got_bits = bf16_tensor_bits(y)[t_idx, n_idx].astype(np.int32)
        assert np.abs(got_bits - ref_bits).max() <= 1
        # property that holds at any size: no output left unwritten, |acc| within its bound
        accn = acc.cpu().numpy()
        bound = 127 * K // 2 if sparse else 127 * K
        assert accn.min() >= -bound and accn.max() <= bound
        assert not torch.isnan(y.float()).any()


@pytest.mark.parametrize("name,T,K,N", [("down", 4096, 6912, 2560), ("down_7b", 8192, 11008, 4096)])
def test_full_size_sampled_68(name, T, K, N):
    # the 6:8 layer at full size, in the configuration bench.py --workload p68 times: pack parity
    # on the whole matrix, activations on the whole batch, accumulators and outputs on samples
    W = inputs.latent_weights(N, K, seed=24)
    x = inputs.activations_bf16(T, K, seed=25, token_lognormal_sigma=0.5)
    g = gpu_quantize_mask_pack68(W)
    r = _assert_pack68(W, g)
    xq_ref, s_ref = oracle.quant_act(x)
    xq, a_scale = gpu_quant_act_expand68(x)
    assert np.array_equal(a_scale.cpu().numpy(), s_ref)
    assert np.array_equal(xq_to_numpy(xq, T, 3 * K // 2), xq_ref[:, expand68_columns(K)])
    t_idx, n_idx = inputs.sample_positions(T, N, 4096, seed=26)
    t_idx[:4] = [0, T - 1, 0, T - 1]
    n_idx[:4] = [0, 0, N - 1, N - 1]
    y, acc = gpu_gemm(True, xq, a_scale, g["dev"], out_dtype=torch.bfloat16)
    acc_ref = oracle.acc_dense_sampled(xq_ref, r["w_eff"], t_idx, n_idx)
    assert np.array_equal(acc.cpu().numpy()[t_idx, n_idx], acc_ref)
    y_ref = oracle.dequant(acc_ref.reshape(-1, 1), r["scale"], s_ref[t_idx]).ravel()
    got_bits = bf16_tensor_bits(y)[t_idx, n_idx].astype(np.int32)
    assert np.abs(got_bits - oracle.f32_to_bf16_bits(y_ref).astype(np.int32)).max() <= 1
    accn = acc.cpu().numpy()
    assert accn.min() >= -127 * 3 * K // 4 and accn.max() <= 127 * 3 * K // 4
    assert not torch.isnan(y.float()).any()


@pytest.mark.parametrize("T,N,K", [(16, 256, 2560), (64, 384, 1280), (300, 256, 2560), (16, 3840, 2560), (1, 2560, 6912)])
def test_gemm_after_repack_sees_the_new_weights(T, N, K):
    # The few-token GEMM fetches weights before its dependency wait; that is only correct because
    # the pack kernel gives its successors no early start.  Re-pack two different matrices into
    # the SAME buffers and run the GEMM right behind each pack, with nothing in between and no
    # synchronisation: every output must belong to the matrix packed just before it.  (A build whose
    # pack kernel signalled early did return stale results on the 3840 x 2560 case.)
    Wa = inputs.latent_weights(N, K, seed=81)
    Wb = inputs.latent_weights(N, K, seed=82)
    bits = inputs.activations_bf16(T, K, seed=83)
    xq_ref, s_ref = oracle.quant_act(bits)
    refs = []
    for W in (Wa, Wb):
        r = _oracle_pack(W)
        refs.append(oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])[1])
    assert not np.array_equal(refs[0], refs[1])
    xq, a_scale = gpu_quant_act(bits)
    Wd = [dev(Wa), dev(Wb)]
    p = b.alloc_packed(N, K)
    ws = b.alloc_gemm_ws(b.OP_SPARSE_BITLINEAR, T, N, K)
    reps = 24
    accs = [torch.zeros((T, N), dtype=torch.int32, device="cuda") for _ in range(reps)]
    y = torch.empty((T, N), dtype=torch.float32, device="cuda")
    for i in range(reps):
        b.sbn_quantize_mask_pack(Wd[i % 2], p["vals"], p["meta"], p["w_scale"], p["ws"])
        b.sbn_sparse_bitlinear(xq, a_scale, p["vals"], p["meta"], p["w_scale"], y, acc_out=accs[i], ws=ws)
    b.sbn_check_status()
    for i in range(reps):
        assert np.array_equal(accs[i].cpu().numpy(), refs[i % 2]), f"launch {i} used stale weights"


# ---- packed weights (2 bits per weight with the metadata) for the few-token regime --------------------
@pytest.mark.parametrize("N,K,seed", [(128, 128, 100), (256, 512, 101), (384, 2560, 102), (128, 6912, 103)])
def test_pack_vals2_parity(N, K, seed):
    W = inputs.latent_weights(N, K, seed=seed)
    r = _oracle_pack(W)
    g = gpu_quantize_mask_pack(W, with_dense=False)
    _, v2 = gpu_pack_vals2(g["dev"])
    assert np.array_equal(v2, oracle.pack_vals2(r["vals"]))


PACKED_GEMM_SHAPES = [(16, 256, 2560), (1, 128, 256), (5, 128, 384), (31, 384, 6912), (32, 128, 1280), (45, 256, 640),
                      (64, 512, 2560), (100, 256, 4096), (7, 128, 11008), (130, 128, 512)]


@pytest.mark.parametrize("T,N,K", PACKED_GEMM_SHAPES)
def test_gemm_parity_packed_weights(T, N, K):
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=T + N + K + 7)
    y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    vals2, _ = gpu_pack_vals2(g["dev"])
    y, acc = gpu_gemm_packed(xq, a_scale, vals2, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)
    bias = np.random.default_rng(T).standard_normal(N).astype(np.float32)
    yb, _ = gpu_gemm_packed(xq, a_scale, vals2, g["dev"], out_dtype=torch.bfloat16, bias=dev(bias), want_acc=False)
    y_ref_b = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"], bias=bias)[0]
    ref_bits = oracle.f32_to_bf16_bits(y_ref_b).astype(np.int32)
    assert np.abs(bf16_tensor_bits(yb).astype(np.int32) - ref_bits).max() <= 1


# ---- activation quantiser + GEMM in one kernel (few tokens) ---------------------------------------------
FUSED_ACT_SHAPES = [(16, 256, 2560), (1, 128, 256), (5, 128, 384), (31, 384, 6912), (32, 128, 1280), (45, 256, 640),
                    (64, 512, 2560), (100, 256, 4096), (7, 128, 11008), (3, 11008 // 128 * 128, 512)]


@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("T,N,K", FUSED_ACT_SHAPES)
def test_fused_quant_act_gemm_parity(sparse, T, N, K):
    W = inputs.latent_weights(N, K, seed=T + N + K + 11)
    bits = inputs.activations_bf16(T, K, seed=T + N + K + 12, token_lognormal_sigma=1.0)
    bits[0, :] = 0                                            # an all-zero token: the 1e-5 clamp
    r = _oracle_pack(W)
    xq_ref, s_ref = oracle.quant_act(bits)
    if sparse:
        y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    else:
        y_ref, acc_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"])
    g = gpu_quantize_mask_pack(W)
    p = g["dev"]
    x = bf16_dev(bits)
    y = torch.full((T, N), float("nan"), dtype=torch.float32, device="cuda")
    acc = torch.full((T, N), -(2 ** 31), dtype=torch.int32, device="cuda")
    a_sc = torch.full((T,), float("nan"), dtype=torch.float32, device="cuda")
    if sparse:
        b.sbn_quant_act_sparse_bitlinear(x, p["vals"], p["meta"], p["w_scale"], y, acc_out=acc, a_scale_out=a_sc)
    else:
        b.sbn_quant_act_bitlinear(x, p["dense_q"], p["w_scale"], y, acc_out=acc, a_scale_out=a_sc)
    b.sbn_check_status()
    assert np.array_equal(a_sc.cpu().numpy(), s_ref)
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)
    # same bits as the two-kernel route of the library itself
    xq, a_scale = gpu_quant_act(bits)
    y2, _ = gpu_gemm(sparse, xq, a_scale, p)
    assert torch.equal(y, y2)


@pytest.mark.parametrize("cluster", [2, 3, 4])
@pytest.mark.parametrize("T,N,K", [(16, 256, 2560), (31, 128, 896), (45, 256, 640), (7, 384, 4096)])
def test_packed_and_fused_kernels_every_cluster_size(T, N, K, cluster):
    # the 32-token kernels with the cluster size forced: 3 takes the select route of the scatter
    W = inputs.latent_weights(N, K, seed=T + N + K + cluster)
    bits = inputs.activations_bf16(T, K, seed=T + N + K + cluster + 1, token_lognormal_sigma=0.5)
    r = _oracle_pack(W)
    xq_ref, s_ref = oracle.quant_act(bits)
    y_ref, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    g = gpu_quantize_mask_pack(W, with_dense=False)
    p = g["dev"]
    vals2, _ = gpu_pack_vals2(p)
    xq, a_scale = gpu_quant_act(bits)
    b.sbn_set_gemm_tuning(0, -cluster)
    y, acc = gpu_gemm_packed(xq, a_scale, vals2, p)
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    _assert_y(y_to_f32_numpy(y), y_ref)
    y2 = torch.full((T, N), float("nan"), dtype=torch.float32, device="cuda")
    acc2 = torch.full((T, N), -(2 ** 31), dtype=torch.int32, device="cuda")
    b.sbn_quant_act_sparse_bitlinear(bf16_dev(bits), p["vals"], p["meta"], p["w_scale"], y2, acc_out=acc2)
    b.sbn_check_status()
    assert np.array_equal(acc2.cpu().numpy(), acc_ref)
    assert torch.equal(y, y2)


# ---- the plain (canonical) layout through the library's own conversion calls ---------------------------
@pytest.mark.parametrize("N,K,seed", [(256, 256, 0), (128, 128, 110), (384, 2560, 111), (640, 6912, 112)])
def test_unpack_canonical_against_oracle(N, K, seed):
    # pack on the GPU, un-tile on the GPU, compare with the oracle's plain arrays: no permutation is
    # restated on the test's side
    W = inputs.latent_weights(N, K, seed=seed)
    r = _oracle_pack(W)
    g = gpu_quantize_mask_pack(W, with_dense=False)
    vals, meta = gpu_unpack_canonical(g["dev"], N, K)
    assert np.array_equal(vals, r["vals"])
    assert np.array_equal(meta, r["meta"])


def test_tile_canonical_round_trip_and_gemm():
    # weights packed by the ORACLE, brought into the library's order by sbn_tile_canonical, then used by
    # the GEMM: accumulators must be the oracle's; and tile -> unpack is the identity
    T, N, K = 70, 384, 1280
    W = inputs.latent_weights(N, K, seed=120)
    bits = inputs.activations_bf16(T, K, seed=121)
    r = _oracle_pack(W)
    xq_ref, s_ref = oracle.quant_act(bits)
    _, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    p = b.alloc_packed(N, K)
    p["vals"].fill_(55)
    p["meta"].fill_(0x55)
    b.sbn_tile_canonical(dev(r["vals"]), dev(r["meta"]), N, K, p["vals"], p["meta"])
    p["w_scale"].copy_(torch.tensor([r["scale"]], dtype=torch.float32))
    assert np.array_equal(p["vals"].cpu().numpy().reshape(-1), tile_vals(r["vals"]))
    assert np.array_equal(p["meta"].cpu().numpy().reshape(-1), tile_meta(r["meta"]))
    vals, meta = gpu_unpack_canonical(p, N, K)
    assert np.array_equal(vals, r["vals"]) and np.array_equal(meta, r["meta"])
    xq, a_scale = gpu_quant_act(bits)
    _, acc = gpu_gemm(True, xq, a_scale, p)
    assert np.array_equal(acc.cpu().numpy(), acc_ref)
    # one pair only
    only_meta = torch.zeros((N, K // 8), dtype=torch.uint8, device="cuda")
    b.sbn_unpack_canonical(None, p["meta"], N, K, None, only_meta)
    b.sbn_check_status()
    assert np.array_equal(only_meta.cpu().numpy(), r["meta"])


# ---- a captured pack call replayed on changed weights ---------------------------------------------------
@pytest.mark.parametrize("N,K", [(2560, 2560), (4096, 4096)])    # 4096 rows: the CTAs also exchange what they have seen under way
def test_quantize_mask_pack_graph_replay_on_changed_weights(N, K):
    # A launch captured in a CUDA graph carries the same host-side nonce at every replay; the slots
    # of the previous replay must still not be taken for this replay's partial sums.  Replays on
    # weights of very different scale: a stale partial sum would give a wrong gamma.
    Ws = [inputs.latent_weights(N, K, seed=130 + i, sigma=0.02 * (3 ** i)) for i in range(3)]
    refs = [_oracle_pack(W) for W in Ws]
    Wd = dev(Ws[0])
    p = b.alloc_packed(N, K)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        b.sbn_quantize_mask_pack(Wd, p["vals"], p["meta"], p["w_scale"], p["ws"])       # set-up outside the capture
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        b.sbn_quantize_mask_pack(Wd, p["vals"], p["meta"], p["w_scale"], p["ws"])
    for rep in range(6):
        i = rep % 3
        Wd.copy_(torch.from_numpy(Ws[i]))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        b.sbn_check_status()
        assert np.float32(p["w_scale"].cpu().numpy()[0]) == refs[i]["scale"], f"replay {rep}"
        vals, meta = gpu_unpack_canonical(p, N, K)
        assert np.array_equal(vals, refs[i]["vals"]), f"replay {rep}"
        assert np.array_equal(meta, refs[i]["meta"]), f"replay {rep}"


# ---- bounded waits that run out --------------------------------------------------------------------------
WAIT_CASES = [("single_cta", 64, 256, 512, (128, 1)), ("pair", 300, 512, 512, (-128, 0)), ("pair_one_m_tile", 300, 256, 512, (-128, 1)),
              ("cluster", 16, 256, 1280, (32, -4)), ("cluster_wide", 100, 256, 1280, (112, -2))]


@pytest.mark.parametrize("sparse", [True, False])
@pytest.mark.parametrize("name,T,N,K,tuning", WAIT_CASES)
def test_gemm_wait_runs_out_and_the_library_recovers(name, T, N, K, tuning, sparse):
    # The load producer is told to issue nothing and the wait limit is 1 ms: the MMA issuer's wait for
    # the first stage runs out, it raises the CTA's abort flag, every role leaves its loop, tensor
    # memory is freed, the kernel returns and the status word says SBN_ERR_TIMEOUT.  Nothing traps
    # and nothing hangs.  The very next ordinary call must be right, bit for bit.
    r, xq_ref, s_ref, g, xq, a_scale = _layer_case(T, N, K, seed=140 + T)
    if sparse:
        _, acc_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"])
    else:
        _, acc_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"])
    b.sbn_set_gemm_tuning(*tuning)
    b.sbn_check_status()
    try:
        b.sbn_set_wait_test(True, 1000)
        with pytest.raises(b.SbnError) as err:
            gpu_gemm(sparse, xq, a_scale, g["dev"])
        assert err.value.code == 7                            # SBN_ERR_TIMEOUT
    finally:
        b.sbn_set_wait_test(False, 0)
    b.sbn_check_status()                                      # the record was cleared by the read above
    _, acc = gpu_gemm(sparse, xq, a_scale, g["dev"])
    assert np.array_equal(acc.cpu().numpy(), acc_ref)


@pytest.mark.parametrize("N,K", [(512, 2560), (4096, 4096)])     # 4096 rows: the CTAs also exchange what they have seen under way
def test_pack_wait_runs_out_and_the_library_recovers(N, K):
    # one CTA of the pack kernel withholds its partial sum: every CTA's bounded wait for that slot runs
    # out, all of them return, the status word says SBN_ERR_TIMEOUT; the next call is exact
    W = inputs.latent_weights(N, K, seed=150)
    r = _oracle_pack(W)
    b.sbn_check_status()
    try:
        b.sbn_set_wait_test(True, 1000)
        with pytest.raises(b.SbnError) as err:
            gpu_quantize_mask_pack(W, with_dense=False)
        assert err.value.code == 7
    finally:
        b.sbn_set_wait_test(False, 0)
    b.sbn_check_status()
    g = gpu_quantize_mask_pack(W, with_dense=False)
    assert g["scale"] == r["scale"]
    assert np.array_equal(g["vals"], r["vals"]) and np.array_equal(g["meta"], r["meta"])


# ---- the streaming pack kernel: hints and very long batches ------------------------------------------------
@pytest.mark.parametrize("hint_factor", [1.0, 1.003, 0.996, 1.02, 2.0, 0.0, -1.0, float("inf")])
def test_quantize_mask_pack_gamma_hint_never_changes_the_result(hint_factor):
    # the hint only decides whether the kernel samples the matrix and whether the bracket holds
    # (within 0.5 % of gamma: the listed values are fixed up; further off: the exact second pass):
    # the bytes must not change
    shapes = [(256, 2560), (640, 256), (128, 128), (384, 1280), (2560, 640), (128, 6912)]
    Ws = [inputs.latent_weights(N, K, seed=160 + i, sigma=0.02 * (i + 1)) for i, (N, K) in enumerate(shapes)]
    refs = [_oracle_pack(W) for W in Ws]
    jobs = []
    for W, r in zip(Ws, refs):
        N, K = W.shape
        bufs = b.alloc_packed(N, K)
        hint = torch.tensor([float(r["scale"]) * hint_factor], dtype=torch.float32, device="cuda")
        jobs.append(dict(W=dev(W), vals=bufs["vals"], meta=bufs["meta"], w_scale=bufs["w_scale"], gamma_hint=hint))
    arr = b.make_pack_jobs(jobs)
    ws = torch.empty(b.sbn_batch_workspace_bytes(len(jobs)), dtype=torch.uint8, device="cuda")
    b.sbn_quantize_mask_pack_batched(arr, ws)
    b.sbn_check_status()
    for job, W, r in zip(jobs, Ws, refs):
        N, K = W.shape
        vals, meta = gpu_unpack_canonical(job, N, K)
        assert np.float32(job["w_scale"].cpu().numpy()[0]) == r["scale"]
        assert np.array_equal(vals, r["vals"]) and np.array_equal(meta, r["meta"])


def test_quantize_mask_pack_hint_in_the_scale_buffer_over_steps():
    # the intended use: w_scale of the previous step is this step's hint, in place, while W drifts
    N, K = 1024, 2560
    W = inputs.latent_weights(N, K, seed=170)
    bufs = b.alloc_packed(N, K)
    bufs["w_scale"].fill_(float("nan"))                          # first step: no usable hint yet
    Wd = dev(W)
    arr = b.make_pack_jobs([dict(W=Wd, vals=bufs["vals"], meta=bufs["meta"], w_scale=bufs["w_scale"], gamma_hint=bufs["w_scale"])])
    ws = torch.empty(b.sbn_batch_workspace_bytes(1), dtype=torch.uint8, device="cuda")
    for step in range(4):
        b.sbn_quantize_mask_pack_batched(arr, ws)
        b.sbn_check_status()
        r = _oracle_pack(W)
        vals, meta = gpu_unpack_canonical(bufs, N, K)
        assert np.float32(bufs["w_scale"].cpu().numpy()[0]) == r["scale"], step
        assert np.array_equal(vals, r["vals"]) and np.array_equal(meta, r["meta"]), step
        W = inputs.perturb_weights(W, seed=171 + step, sigma=1e-4 if step < 2 else 5e-3)   # the last drift breaks the bracket
        Wd.copy_(torch.from_numpy(W))


def test_quantize_mask_pack_batch_longer_than_one_launch_holds():
    # more jobs than one launch of the kernel takes (its per-matrix state on chip is finite): the call
    # splits the batch; every job must still equal the single call
    count = 1030
    base = inputs.latent_weights(128, 128 * count, seed=180).reshape(128, count, 128).transpose(1, 0, 2)
    Ws = [np.ascontiguousarray(base[i]) * np.float32(1 + (i % 7)) for i in range(count)]
    big = {k: torch.empty((count,) + shape, dtype=dt, device="cuda")
           for k, shape, dt in (("vals", (128, 64), torch.int8), ("meta", (128, 16), torch.uint8), ("w_scale", (1,), torch.float32))}
    Wd = torch.from_numpy(np.stack(Ws)).cuda()
    jobs = [dict(W=Wd[i], vals=big["vals"][i], meta=big["meta"][i], w_scale=big["w_scale"][i]) for i in range(count)]
    arr = b.make_pack_jobs(jobs)
    ws = torch.empty(b.sbn_batch_workspace_bytes(count), dtype=torch.uint8, device="cuda")
    b.sbn_quantize_mask_pack_batched(arr, ws)
    b.sbn_check_status()
    for i in list(range(0, count, 97)) + [1023, 1024, 1025, count - 1]:
        r = _oracle_pack(Ws[i])
        vals, meta = gpu_unpack_canonical(dict(vals=big["vals"][i], meta=big["meta"][i]), 128, 128)
        assert np.float32(big["w_scale"][i].cpu().numpy()[0]) == r["scale"], i
        assert np.array_equal(vals, r["vals"]) and np.array_equal(meta, r["meta"]), i


def test_quantize_mask_pack_scale_left_in_the_workspace_never_changes_the_result():
    # A single-matrix call leaves its scale in the workspace, tagged with W and the shape, and the next call
    # for the same buffer on the same workspace starts from it.  Same buffer with weights of another scale,
    # another buffer of the same shape, the same call again, a workspace full of noise: always the oracle's bits.
    N, K = 640, 2560
    Wa = inputs.latent_weights(N, K, seed=410)
    Wb = inputs.latent_weights(N, K, seed=411, sigma=0.31)          # 15 x the scale: the estimate is useless
    Wc = inputs.perturb_weights(Wa, seed=412, sigma=1e-4)           # a training step later: the estimate is good
    refs = {k: _oracle_pack(w) for k, w in (("a", Wa), ("b", Wb), ("c", Wc))}
    buf = dev(Wa)
    other = dev(Wb)
    bufs = b.alloc_packed(N, K)

    def run_and_check(W_dev, r):
        b.sbn_quantize_mask_pack(W_dev, bufs["vals"], bufs["meta"], bufs["w_scale"], bufs["ws"])
        b.sbn_check_status()
        vals, meta = gpu_unpack_canonical(bufs, N, K)
        assert np.float32(bufs["w_scale"].cpu().numpy()[0]) == r["scale"]
        assert np.array_equal(vals, r["vals"]) and np.array_equal(meta, r["meta"])

    bufs["ws"].copy_(torch.randint(0, 256, bufs["ws"].shape, dtype=torch.uint8, device="cuda"))    # noise: no tag
    run_and_check(buf, refs["a"])
    run_and_check(buf, refs["a"])                   # the same matrix again: starts from its own scale
    buf.copy_(torch.from_numpy(Wc).cuda())
    run_and_check(buf, refs["c"])                   # a step later: a good estimate
    buf.copy_(torch.from_numpy(Wb).cuda())
    run_and_check(buf, refs["b"])                   # same buffer, another scale: the estimate misses
    run_and_check(other, refs["b"])                 # another buffer: the tag does not match
    buf.copy_(torch.from_numpy(Wa).cuda())
    run_and_check(buf, refs["a"])


def test_quantize_mask_pack_68_starts_from_a_sample():
    # The scale left in the workspace belongs to the 2:4 calls: a 6:8 call neither takes one that a 2:4 call on the same
    # buffer left (here useless: the weights have changed since) nor leaves its own.
    N, K = 256, 1024
    Wa, Wb = inputs.latent_weights(N, K, seed=420), inputs.latent_weights(N, K, seed=421, sigma=0.31)
    buf = dev(Wa)
    bufs = b.alloc_packed(N, K, n_keep=6, m_group=8)
    b24 = b.alloc_packed(N, K)
    slots_and_generation = 148 * 16 + 8

    def pack68(W):
        b.sbn_quantize_mask_pack(buf, bufs["vals"], bufs["meta"], bufs["w_scale"], bufs["ws"], n_keep=6, m_group=8)
        b.sbn_check_status()
        vals, meta = gpu_unpack_canonical(bufs, N, b.sbn_expanded_k(K, 6, 8))
        _assert_pack68(W, dict(vals=vals, meta=meta, scale=np.float32(bufs["w_scale"].cpu().numpy()[0])))

    bufs["ws"].fill_(0xA5)
    pack68(Wa)
    assert bool((bufs["ws"][slots_and_generation:] == 0xA5).all())
    b.sbn_quantize_mask_pack(buf, b24["vals"], b24["meta"], b24["w_scale"], bufs["ws"])
    left = bufs["ws"][slots_and_generation:].clone()
    assert bool((left != 0xA5).any())                               # the 2:4 call did leave one
    buf.copy_(torch.from_numpy(Wb).cuda())
    pack68(Wb)
    assert torch.equal(bufs["ws"][slots_and_generation:], left)


# ---- the register-fed few-token kernel -----------------------------------------------------------------------------
@pytest.mark.parametrize("T,N,K", [(1, 128, 128), (8, 128, 256), (3, 256, 1152), (5, 4864, 384), (1, 4864, 3328), (9, 640, 1408),
                                   (16, 2560, 256), (16, 128, 128), (5, 7296, 1152), (8, 7296, 2176), (3, 5120, 3328),
                                   (12, 256, 6912), (16, 256, 4352), (2, 128, 8320), (5, 7296, 896), (3, 7296, 1536), (1, 9216, 2304)])
def test_few_token_kernel_all_forms(T, N, K):
    # one token and the last of each group of 8; fewer 128-column blocks than warps, a last round that leaves warps without
    # a block; CTAs with a second row group (7296 / 16 = 456 of them on 444 places, in one and in more rounds over K; fused with
    # K > 3072: 304 and 320 on 296); rows long enough for the early fetch of the next blocks, too long for it; fused calls with a second row
    # group that leave it out (one block per warp; dense, twelve blocks; 2:4, 576 groups on 444 places).  Accumulators exact, outputs as everywhere.
    W = inputs.latent_weights(N, K, seed=200 + T)
    bits = inputs.activations_bf16(T, K, seed=300 + K, token_lognormal_sigma=0.5)
    bias = np.random.default_rng(N).standard_normal(N).astype(np.float32)
    r = _oracle_pack(W)
    xq_ref, s_ref = oracle.quant_act(bits)
    g = gpu_quantize_mask_pack(W)
    p = g["dev"]
    vals2, _ = gpu_pack_vals2(p)
    xq, a_scale = gpu_quant_act(bits)
    x, bias_d = bf16_dev(bits), torch.from_numpy(bias).cuda()
    sparse_ref = oracle.sparse_bitlinear(xq_ref, s_ref, r["vals"], r["meta"], r["scale"], bias)
    dense_ref = oracle.bitlinear(xq_ref, s_ref, r["dense_q"], r["scale"], bias)
    calls = [
        (lambda y, acc: b.sbn_sparse_bitlinear(xq, a_scale, p["vals"], p["meta"], p["w_scale"], y, bias=bias_d, acc_out=acc), sparse_ref),
        (lambda y, acc: b.sbn_bitlinear(xq, a_scale, p["dense_q"], p["w_scale"], y, bias=bias_d, acc_out=acc), dense_ref),
    ]
    if K >= 256:
        calls += [
            (lambda y, acc: b.sbn_sparse_bitlinear_packed(xq, a_scale, vals2, p["meta"], p["w_scale"], y, bias=bias_d, acc_out=acc), sparse_ref),
            (lambda y, acc: b.sbn_quant_act_sparse_bitlinear(x, p["vals"], p["meta"], p["w_scale"], y, bias=bias_d, acc_out=acc), sparse_ref),
            (lambda y, acc: b.sbn_quant_act_bitlinear(x, p["dense_q"], p["w_scale"], y, bias=bias_d, acc_out=acc), dense_ref),
        ]
    for call, (y_ref, acc_ref) in calls:
        y = torch.full((T, N), float("nan"), dtype=torch.float32, device="cuda")
        acc = torch.full((T, N), -(2 ** 31), dtype=torch.int32, device="cuda")
        call(y, acc)
        b.sbn_check_status()
        assert np.array_equal(acc.cpu().numpy(), acc_ref)
        _assert_y(y.cpu().numpy(), y_ref)
        yb = torch.full((T, N), float("nan"), dtype=torch.bfloat16, device="cuda")
        call(yb, None)
        b.sbn_check_status()
        assert torch.equal(yb, y.to(torch.bfloat16))                # bf16 = the fp32 value rounded to nearest even


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_gemm_without_the_workspace_its_split_would_use(dtype):
    # K through global memory is the fastest plan here; a caller without a workspace (or with too little) gets the fastest
    # other one, bit for bit the same
    T, N, K = 9, 2304, 24576
    need = b.sbn_workspace_bytes(b.OP_BITLINEAR, T, N, K)
    assert need > 0
    gen = torch.Generator(device="cuda").manual_seed(1)
    q = torch.randint(-1, 2, (N, K), generator=gen, device="cuda", dtype=torch.int8)
    x = torch.randn((T, K), generator=gen, device="cuda").to(torch.bfloat16)
    xq, a_scale, w_scale = b.alloc_xq(T, K), torch.empty(T, device="cuda"), torch.full((1,), 0.02, device="cuda")
    b.sbn_quant_act(x, xq, a_scale)
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
    ys = []
    for w in (ws, None, ws[:256]):
        y = torch.full((T, N), float("nan"), dtype=dtype, device="cuda")
        b.sbn_bitlinear(xq, a_scale, q, w_scale, y, ws=w)
        b.sbn_check_status()
        ys.append(y)
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])
    assert int(ws.count_nonzero()) == 0                             # zero-kept
