"""GPU parity: the CUDA library (through its C ABI) against the fp64 oracle on the same seeded
inputs.  Flags bit-exact outside the 1e-6 score band; outputs within 1e-5 (fp32) / 2e-2 (bf16)
max relative error |dy| / max(|y_ref|, rms(y_ref[t,:]))."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2501_10054_b200 as T
import workloads as W
from oracle import tardis_oracle as O
from tests import helpers as Hp

pytestmark = pytest.mark.gpu


def _layer(cfg, seed=0):
    return Hp.to_cuda(W.make_layer(cfg, seed))


def _run(cfg, n, calls=None, seed=0, path=0, full_fold=True):
    L = _layer(cfg, seed)
    s = L.numpy64()
    x = W.make_tokens(cfg, n, seed).cuda()
    h = T.fold_layer(L)
    try:
        T.tardis_set_path(h, path)
        y, F, S = Hp.gpu_forward(h, L, x, calls)
        # generic kernels: exact fp64 score; fused decode kernel (calls of up to 8 tokens): exact up to the tracked
        # rounding of tiny x elements; batched path: fp32 tensor-core scores (flags are settled exactly near the
        # range ends, the captured score is the fast one)
        if path == 1 or cfg.dtype == "f32":
            tol = 1e-9
        else:
            # the decode kernel rounds x to a 22-bit grid under the token's largest element
            xmax = x.float().abs().amax(dim=1).cpu().numpy()
            small = np.maximum(5e-7, 4e-6 * xmax)
            fused = path != 3 and cfg.bits == 2
            tol = np.concatenate([np.full(b, 0.0 if (b <= 8 and fused) else 3e-4) for b in (calls or [n])])
            tol = np.where(tol == 0.0, small, tol)
        info = Hp.assert_parity(L, s, x, y, F, S, full_fold=full_fold, label=cfg.name, score_tol=tol)
        st = T.tardis_stats(h)
        assert st["tokens"] == n and st["device_error"] == 0
        assert st["flagged_total"] == int(F.sum())
        assert st["flagged_max"] == int(F.sum(1).max()) if n else True
    finally:
        T.tardis_destroy(h)
    return info


def test_tiny_f32_config_all_tokens():
    cfg = W.CONFIGS["tiny_f32"]
    info = _run(cfg, 64)
    assert 0.02 < info["flag_frac"] < 0.4


def test_tiny_f32_fold_matches_oracle_elementwise():
    cfg = W.CONFIGS["tiny_f32"]
    L = _layer(cfg)
    s = L.numpy64()
    h = T.fold_layer(L)
    Wf = torch.empty(cfg.d_model, cfg.d_model, dtype=torch.float32, device="cuda")
    bf = torch.empty(cfg.d_model, dtype=torch.float32, device="cuda")
    T.tardis_export_folded(h, Wf, bf)
    torch.cuda.synchronize()
    Wf_ref, bf_ref = O.fold(s["W1"], s["W2"], s["a"], s["c"], s["b1"], s["b2"])
    assert np.abs(Wf.double().cpu().numpy() - Wf_ref).max() <= 1e-5 * np.abs(Wf_ref).max()
    assert np.abs(bf.double().cpu().numpy() - bf_ref).max() <= 1e-5 * np.abs(bf_ref).max()
    st = T.tardis_stats(h)
    # footprint accounting: folded matrix d^2 against the 2 d h original weights = 12.5 % at h = 4 d,
    # 2-bit codes = 6.25 % of the original weights
    assert (st["bytes_folded"] - 4 * cfg.d_model) / (st["bytes_w1"] + st["bytes_w2t"]) == 0.125
    assert (cfg.d_ff * cfg.d_model // 4) / st["bytes_w1"] == 2 / 32            # 2-bit codes against fp32 W1
    T.tardis_destroy(h)


@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("shape", [(512, 2048, 64), (1136, 4544, 16), (768, 3072, 128)])
def test_bf16_small_shapes_ragged_batches(shape, path):
    d, hh, G = shape
    cfg = W.LayerConfig("small_%d" % d, d, hh, group=G, n_calib=512, bias=(d != 1136),
                        tokens="mixture" if d == 1136 else "student_t")
    calls = [1, 1, 3, 8, 9, 0, 2, 64, 65, 5]
    info = _run(cfg, sum(calls), calls, path=path)
    assert 0.02 < info["flag_frac"] < 0.5


def test_batched_path_forced_for_calls_of_a_few_tokens():
    # path 3 sends every call through the tensor-core path, also those the per-token kernel would take
    cfg = W.LayerConfig("small_forced", 512, 2048, group=64, n_calib=512)
    calls = [1, 3, 8, 2, 0, 7]
    info = _run(cfg, sum(calls), calls, path=3)
    assert 0.02 < info["flag_frac"] < 0.5


@pytest.mark.parametrize("bits", [3, 4, 8])
def test_wider_predictor_codes(bits):
    # 3- and 4-bit codes: batched tensor-core path (also for calls of a few tokens) and generic kernels; 8-bit codes: generic
    # kernels only.  The paper sweeps the predictor size (Section 7.6); here each width must give the oracle's flags.
    # (3-bit codes are a bit stream: some cross from one 32-bit word into the next.)
    cfg = W.LayerConfig("bits%d" % bits, 512, 2048, group=64, bits=bits, n_calib=512)
    calls = [1, 3, 20, 8]
    info = _run(cfg, sum(calls), calls, path=3 if bits <= 4 else 0)
    assert 0.02 < info["flag_frac"] < 0.5
    _run(cfg, 6, [1, 5], path=1)
    cfg32 = W.LayerConfig("bits%d_f32" % bits, 128, 512, dtype="f32", group=32, bits=bits, n_calib=512)
    _run(cfg32, 7)


@pytest.mark.parametrize("rows", [range(0, 0), range(130, 141), range(0, 2048, 127)])
@pytest.mark.parametrize("n", [3, 20, 150])
def test_predictor_values_of_two_terms_in_some_row_tiles(rows, n):
    # zero-points at the end of the code range make values 3 s, which need a second bf16 term; the fold notes the 128-row tiles
    # that have any: none, one tile, every tile
    cfg = W.LayerConfig("two_terms", 512, 2048, group=64, n_calib=512)
    L = _layer(cfg, 3)
    r = torch.tensor(list(rows), device="cuda", dtype=torch.long)
    L.zero[r] = torch.where(torch.arange(L.zero.shape[1], device="cuda") % 2 == 0, 0, 3).to(torch.uint8)
    L.scale[r] *= 0.4
    s = L.numpy64()
    x = W.make_tokens(cfg, n, 3).cuda()
    for path in (0, 3):
        h = T.fold_layer(L)
        try:
            T.tardis_set_path(h, path)
            y, F, S = Hp.gpu_forward(h, L, x)
            Hp.assert_parity(L, s, x, y, F, S, score_tol=3e-4, label="rows %r path %d" % (rows, path))
        finally:
            T.tardis_destroy(h)


def test_relu_activation_on_every_path():
    # ReLU layer (the OPT model of the paper's evaluation): per-token kernel, batched path, generic kernels, fp32
    cfg = W.LayerConfig("relu", 512, 2048, dtype="bf16", act=W.ACT_RELU, n_calib=512)
    _run(cfg, 30, [1, 5, 24], seed=2)
    _run(cfg, 12, [2, 10], seed=2, path=1)
    cfg = W.LayerConfig("relu32", 128, 512, dtype="f32", act=W.ACT_RELU, n_calib=512)
    _run(cfg, 9, seed=4)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_exact_range_mode_flags_from_true_preactivations(dtype):
    # path 4: the range check runs on z = W1 x + b1 itself (the paper's ablation that takes the predictor out)
    cfg = W.LayerConfig("hybrid_" + dtype, 256, 1024, dtype=dtype, n_calib=512)
    L = _layer(cfg, 1)
    s = L.numpy64()
    x = W.make_tokens(cfg, 11, 1).cuda()
    h = T.fold_layer(L)
    try:
        T.tardis_set_path(h, 4)
        y, F, S = Hp.gpu_forward(h, L, x, [1, 10])
        x64 = x.double().cpu().numpy()
        z = x64 @ s["W1"].T + s["b1"][None, :]
        F_ref = O.flags_from_score(z, s["lo"], s["hi"])
        band = O.near_threshold(z, s["lo"], s["hi"], Hp.BAND)
        assert not ((F != F_ref) & ~band).any()
        assert np.abs(S - z).max() < 1e-9                       # the captured score is the pre-activation
        y_ref = O.direct_partially_linear(x64, np.where(band, F, F_ref), s["W1"], s["W2"], s["a"], s["c"], s["b1"], s["b2"], s["act"])
        assert np.nanmax(O.rel_error(y.double().cpu().numpy(), y_ref)) <= Hp.TOL[dtype]
        # the predictor's flags differ from these on some neurons (that difference is what the mode measures)
        zhat = O.predictor_score(x64, s["codes"], s["scale"], s["zero"], s["group"], s["b1"], s["bits"])
        assert (O.flags_from_score(zhat, s["lo"], s["hi"]) != F_ref).any()
    finally:
        T.tardis_destroy(h)


def test_erf_activation_and_other_seed():
    cfg = W.LayerConfig("erf", 256, 1024, dtype="bf16", act=W.ACT_GELU_ERF, n_calib=512)
    _run(cfg, 17, [1, 16], seed=5)
    cfg = W.LayerConfig("erf32", 128, 512, dtype="f32", act=W.ACT_GELU_ERF, n_calib=512)
    _run(cfg, 9, seed=6)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_degenerate_ranges_all_and_none_flagged(dtype):
    cfg = W.LayerConfig("deg_" + dtype, 256, 1024, dtype=dtype, n_calib=256)
    L = _layer(cfg)
    x = W.make_tokens(cfg, 5, 1).cuda()
    inf = torch.full_like(L.lo, float("inf"))
    for lo, hi, frac in ((inf, inf, 1.0), (-inf, inf, 0.0)):
        L2 = W.Layer(**{**L.__dict__, "lo": lo, "hi": hi})
        s = L2.numpy64()
        h = T.fold_layer(L2)
        y, F, S = Hp.gpu_forward(h, L2, x, [1, 4])
        assert F.mean() == frac
        Hp.assert_parity(L2, s, x, y, F, S, label="degenerate", score_tol=1e-4)
        if frac == 1.0:   # every neuron flagged: the original GELU FFN
            dense = O.dense_ffn(x.double().cpu().numpy(), s["W1"], s["W2"], s["b1"], s["b2"], s["act"])
            assert O.rel_error(y.double().cpu().numpy(), dense).max() <= Hp.TOL[dtype]
        T.tardis_destroy(h)


def test_nan_token_is_flagged_everywhere_and_propagates():
    cfg = W.LayerConfig("nan", 256, 1024, dtype="bf16", n_calib=256)
    L = _layer(cfg)
    x = W.make_tokens(cfg, 3, 2).cuda()
    x[1, 7] = float("nan")
    h = T.fold_layer(L)
    y, F, S = Hp.gpu_forward(h, L, x, [3])
    assert F[1].all() and torch.isnan(y[1]).all()
    assert not torch.isnan(y[0]).any() and not torch.isnan(y[2]).any()
    T.tardis_destroy(h)


def test_forward_argument_errors_and_empty_call():
    cfg = W.LayerConfig("args", 128, 512, dtype="bf16", n_calib=256)
    L = _layer(cfg)
    h = T.fold_layer(L)
    lib = T.load_library()
    x = W.make_tokens(cfg, 2, 0).cuda()
    y = torch.empty_like(x)
    assert lib.tardis_ffn_forward(h, x.data_ptr(), y.data_ptr(), -1, None) == 1
    assert lib.tardis_ffn_forward(h, None, y.data_ptr(), 1, None) == 1
    assert lib.tardis_ffn_forward(h, x.data_ptr() + 2, y.data_ptr(), 1, None) == 1
    assert lib.tardis_ffn_forward(h, None, None, 0, None) == 0          # empty call is a no-op
    assert T.tardis_stats(h)["calls"] == 0
    T.tardis_destroy(h)


def test_run_to_run_flags_identical():
    cfg = W.LayerConfig("rep", 512, 2048, n_calib=512)
    L = _layer(cfg)
    x = W.make_tokens(cfg, 8, 0).cuda()
    h = T.fold_layer(L)
    y1, F1, S1 = Hp.gpu_forward(h, L, x, [8])
    y2, F2, S2 = Hp.gpu_forward(h, L, x, [8])
    # the fused kernel adds its partial scores in a fixed order: the captured scores of two runs are the same numbers
    assert (F1 == F2).all() and (S1 == S2).all()
    assert (y1.float() - y2.float()).abs().max() <= 2e-2 * y1.float().abs().max()
    T.tardis_destroy(h)


@pytest.mark.parametrize("d,h,G", [(512, 2048, 64), (4096, 16384, 128)])
def test_deterministic_mode_same_bits_run_to_run(d, h, G):
    """With tardis_set_deterministic on, y of repeated calls is the same bits (fused path at 1, 3, 4 and 9 tokens, batched
    path at 40 tokens), still agrees with the oracle, and other work in between (a call in the default mode, a call on
    another handle) does not change it."""
    cfg = W.LayerConfig("det", d, h, n_calib=512, group=G)
    L = _layer(cfg)
    s = L.numpy64()
    other = T.fold_layer(L)                                  # a second handle of the same layer, left in the default mode
    hd = T.fold_layer(L)
    try:
        T.tardis_set_deterministic(hd, True)
        for n in (1, 3, 4, 9, 40):
            x = W.make_tokens(cfg, n, 7 + n).cuda()
            outs = []
            for rep in range(4):
                y = torch.empty_like(x)
                T.tardis_ffn_forward(hd, x, y)
                torch.cuda.synchronize()
                outs.append(y.clone())
                yo = torch.empty_like(x)
                T.tardis_ffn_forward(other, x, yo)            # unrelated work between the repetitions
            for y in outs[1:]:
                assert torch.equal(y.view(torch.int16), outs[0].view(torch.int16)), "n = %d" % n
            assert T.tardis_stats(hd)["last_path"] == (2 if n <= 16 else 3)
            yg, F, S = Hp.gpu_forward(hd, L, x, [n])
            assert torch.equal(yg.view(torch.int16), outs[0].view(torch.int16))
            keep = np.arange(n)[: 6]
            ix = torch.as_tensor(keep).cuda()
            Hp.assert_parity(L, s, x[ix], yg[ix], F[keep], S[keep], score_tol=3e-4, label="det n=%d" % n)
        # switching the mode off again gives the default kernels back (same flags, y within the usual tolerance)
        T.tardis_set_deterministic(hd, False)
        x = W.make_tokens(cfg, 4, 99).cuda()
        y0 = torch.empty_like(x); y1 = torch.empty_like(x)
        T.tardis_ffn_forward(hd, x, y0)
        T.tardis_ffn_forward(other, x, y1)
        torch.cuda.synchronize()
        assert (y0.float() - y1.float()).abs().max() <= 2e-2 * y1.float().abs().max()
        assert T.tardis_stats(hd)["device_error"] == 0
    finally:
        T.tardis_destroy(hd)
        T.tardis_destroy(other)


def test_deterministic_mode_refused_where_only_atomic_kernels_serve():
    cfg = W.LayerConfig("detf32", 256, 1024, n_calib=512, dtype="f32")
    L = _layer(cfg)
    h = T.fold_layer(L)
    try:
        with pytest.raises(T.TardisError) as e:
            T.tardis_set_deterministic(h, True)
        assert e.value.status == 2
    finally:
        T.tardis_destroy(h)


@pytest.mark.parametrize("n,normalise,residual", [(1, True, True), (5, True, True), (40, True, True), (3, False, True), (4, True, False)])
def test_stack_forward_layer_by_layer_against_the_oracle(n, normalise, residual):
    """Three independently seeded layers chained on one stream.  With `keep`, every layer's input u_l and output f_l
    are read back: u_l against the oracle's layer normalisation of the stream the GPU itself had (rebuilt from the
    kept outputs, so that a flag that flips downstream of a bf16 rounding does not hide a layer's error), f_l against
    the oracle's forward on exactly u_l (flags and scores captured per layer), the final stream against the rounded
    sums.  The same call without `keep` (two work buffers in turns) gives the same y."""
    cfg = W.LayerConfig("stack", 512, 2048, n_calib=512)
    Ls = [_layer(cfg, seed=10 + l) for l in range(3)]
    hs = [T.fold_layer(L) for L in Ls]
    g = torch.Generator().manual_seed(3)
    gammas = [(1.0 + 0.1 * torch.randn(512, generator=g)).cuda() for _ in Ls]
    betas = [(0.1 * torch.randn(512, generator=g)).cuda() for _ in Ls]
    x = W.make_tokens(cfg, n, 21).cuda()
    try:
        caps = []
        for h in hs:
            bm = torch.zeros(n, 2048 // 32, dtype=torch.int32, device="cuda")
            sc = torch.full((n, 2048), float("nan"), dtype=torch.float64, device="cuda")
            T.tardis_set_debug_capture(h, bm, sc)
            caps.append((bm, sc))
        keep = torch.full((3, 2, n, 512), float("nan"), dtype=x.dtype, device="cuda")
        y = torch.empty_like(x)
        T.tardis_stack_forward(hs, x, y, gammas, betas, 1e-5, normalise, residual, keep=keep)
        torch.cuda.synchronize()
        for h in hs:
            T.tardis_set_debug_capture(h, None, None)
        stream = x.clone()
        for l, L in enumerate(Ls):
            u, f = keep[l, 0], keep[l, 1]
            if normalise:
                ref_u = O.layer_norm(stream.double().cpu().numpy(), gammas[l].double().cpu().numpy(), betas[l].double().cpu().numpy(), 1e-5)
                err = np.abs(u.double().cpu().numpy() - ref_u)
                assert (err <= 2.0 ** -8 * np.abs(ref_u) + 1e-6).all(), "layer %d: normalisation off by %.3e" % (l, err.max())
            else:
                assert torch.equal(u, stream)
            F = Hp.unpack_bitmap(caps[l][0], 2048)
            S = caps[l][1].cpu().numpy()
            Hp.assert_parity(L, L.numpy64(), u, f, F, S, score_tol=3e-4, label="stack layer %d" % l)
            stream = (stream.float() + f.float()).to(x.dtype) if residual else f.clone()
        assert torch.equal(y, stream)
        # without keep: same result from the two work buffers; in place as well
        y2 = torch.empty_like(x)
        T.tardis_stack_forward(hs, x, y2, gammas, betas, 1e-5, normalise, residual)
        x3 = x.clone()
        T.tardis_stack_forward(hs, x3, x3, gammas, betas, 1e-5, normalise, residual)
        torch.cuda.synchronize()
        tol = 2e-2 * float(y.float().abs().max())
        assert float((y2.float() - y.float()).abs().max()) <= tol and float((x3.float() - y.float()).abs().max()) <= tol
        # a buffer that is too small is refused
        with pytest.raises(T.TardisError) as e:
            T.tardis_stack_forward(hs, x, y2, gammas, betas, 1e-5, normalise, residual, work=torch.empty(n * 512, dtype=x.dtype, device="cuda"))
        assert e.value.status == 1
    finally:
        for h in hs:
            T.tardis_destroy(h)


@pytest.mark.parametrize("dtype,d,h", [("bf16", 512, 2048), ("f32", 256, 1024)])
def test_allocation_failures_return_a_status_and_leak_nothing(dtype, d, h):
    """Every device allocation of tardis_fold (and of what it prepares for the kernels) fails once in turn, injected through
    tardis_debug_fail_alloc: the call returns TARDIS_ERR_ALLOC, frees what it had, and a later fold of the same layer works
    and gives correct results.  The same for the buffers of the deterministic mode, the predictor builder and tardis_load."""
    import tempfile, os
    cfg = W.LayerConfig("allocfail", d, h, n_calib=512, dtype=dtype)
    L = _layer(cfg)
    torch.cuda.synchronize()
    live0 = T.tardis_debug_live_allocations()               # (other tests' handles are all destroyed: normally (0, 0))
    failed = 0
    try:
        for nth in range(200):
            T.tardis_debug_fail_alloc(nth)
            try:
                hd = T.fold_layer(L)
            except T.TardisError as e:
                assert e.status == 3, e.status
                failed += 1
                assert T.tardis_debug_live_allocations() == live0, "allocation %d: something left behind" % nth
                continue
            break                                            # nth is past the last allocation of a fold: it went through
        else:
            raise AssertionError("fold never succeeded")
        T.tardis_debug_fail_alloc(-1)
        assert failed >= 10, failed
        x = W.make_tokens(cfg, 3, 1).cuda()
        y, F, S = Hp.gpu_forward(hd, L, x, [3])
        Hp.assert_parity(L, L.numpy64(), x, y, F, S, score_tol=3e-4, label="after failures")
        if dtype == "bf16":
            T.tardis_debug_fail_alloc(0)
            with pytest.raises(T.TardisError):
                T.tardis_set_deterministic(hd, True)
            T.tardis_debug_fail_alloc(-1)
            T.tardis_set_deterministic(hd, True)
            T.tardis_set_deterministic(hd, False)
        path = os.path.join(tempfile.mkdtemp(), "layer.bin")
        T.tardis_save(hd, path)
        T.tardis_destroy(hd)
        hd = None
        assert T.tardis_debug_live_allocations() == live0
        for nth in (0, 3, 9):
            T.tardis_debug_fail_alloc(nth)
            with pytest.raises(T.TardisError) as e:
                T.tardis_load(path)
            assert e.value.status == 3
            assert T.tardis_debug_live_allocations() == live0
        for nth in range(5):
            T.tardis_debug_fail_alloc(nth)
            with pytest.raises(T.TardisError) as e:
                T.tardis_build_predictor(L.W1, None, 2, 64)
            assert e.value.status == 3
        T.tardis_debug_fail_alloc(-1)
        assert T.tardis_debug_live_allocations() == live0
    finally:
        T.tardis_debug_fail_alloc(-1)
        if hd:
            T.tardis_destroy(hd)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_guard_areas_report_a_write_past_a_buffer(dtype):
    """The buffers of a handle lie between guard areas that tardis_stats checks: untouched after real work on every path,
    reported as TARDIS_ERR_CORRUPT once four guard bytes in front of or behind a buffer have changed (changed here by
    tardis_debug_damage_guard, inside the allocation), and fine again after they are restored."""
    cfg = W.LayerConfig("guards", 512, 2048, n_calib=512, dtype=dtype)
    L = _layer(cfg)
    h = T.fold_layer(L)
    try:
        x = W.make_tokens(cfg, 70, 2).cuda()
        y = torch.empty_like(x)
        for n in (1, 4, 9, 70):
            T.tardis_ffn_forward(h, x[:n], y[:n])
        for path in (1, 3, 4, 0):
            T.tardis_set_path(h, path)
            T.tardis_ffn_forward(h, x[:5], y[:5])
        assert T.tardis_stats(h)["device_error"] == 0          # (reads every guard back)
        for front in (True, False):
            T.tardis_debug_damage_guard(h, front, False)
            with pytest.raises(T.TardisError) as e:
                T.tardis_stats(h)
            assert e.value.status == 6
            T.tardis_debug_damage_guard(h, front, True)
            assert T.tardis_stats(h)["device_error"] == 0
        T.tardis_ffn_forward(h, x[:3], y[:3])
        assert T.tardis_stats(h)["device_error"] == 0
    finally:
        T.tardis_destroy(h)


def test_batched_path_chunk_boundary_nan_token_and_empty_ranges():
    """More tokens than one scratch chunk in a single call (chunks hold 1024 tokens while the debug capture is on,
    2048 otherwise), a token holding a NaN in the middle of it, and the result compared token by token with the
    oracle on a seeded sample."""
    cfg = W.LayerConfig("chunks", 256, 1024, n_calib=512)
    L = _layer(cfg)
    s = L.numpy64()
    n = 1030
    x = W.make_tokens(cfg, n, 4).cuda()
    x[1027, 5] = float("nan")
    h = T.fold_layer(L)
    try:
        y, F, S = Hp.gpu_forward(h, L, x, [n])
        assert T.tardis_stats(h)["last_path"] == 3
        assert F[1027].all() and torch.isnan(y[1027]).all()
        keep = np.array([0, 1, 511, 1023, 1024, 1026, 1028, 1029])
        assert not torch.isnan(y[torch.as_tensor(keep).cuda()]).any()
        Hp.assert_parity(L, s, x[torch.as_tensor(keep).cuda()], y[torch.as_tensor(keep).cuda()], F[keep], S[keep],
                         score_tol=3e-4, label="chunks")
        st = T.tardis_stats(h)
        assert st["flagged_total"] == int(F.sum()) and st["device_error"] == 0
        # without the capture the chunks are twice as long: 2055 tokens cross that boundary too, and every token
        # must come out as it does in the captured run (same products, same order of accumulation)
        x2 = torch.cat([x, x[:1025]])
        y2 = torch.empty_like(x2)
        T.tardis_ffn_forward(h, x2, y2)
        torch.cuda.synchronize()
        ref2 = torch.cat([y, y[:1025]])
        ok = (y2 == ref2) | (torch.isnan(y2) & torch.isnan(ref2))
        assert bool(ok.all())
    finally:
        T.tardis_destroy(h)


def test_bounded_wait_runs_out_is_reported_and_cleared():
    """A device-side wait whose data never arrives ends by its limit, sets the error word (no trap, no hang: the kernel
    returns normally), tardis_stats reports the time-out, and after tardis_clear_error the handle works as before."""
    cfg = W.LayerConfig("timeout", 256, 1024, n_calib=256)
    L = _layer(cfg)
    s = L.numpy64()
    x = W.make_tokens(cfg, 3, 4).cuda()
    h = T.fold_layer(L)
    lib = T.load_library()
    y0, F0, _ = Hp.gpu_forward(h, L, x, [3])
    assert lib.tardis_debug_wait_timeout(h, 200000, None) == 0          # about 0.1 ms of waiting
    st = T.Stats()
    assert lib.tardis_stats(h, ctypes.byref(st)) == 5                   # TARDIS_ERR_TIMEOUT
    assert st.device_error == 1
    assert lib.tardis_clear_error(h) == 0
    assert lib.tardis_stats(h, ctypes.byref(st)) == 0 and st.device_error == 0
    y1, F1, _ = Hp.gpu_forward(h, L, x, [3])
    assert (F0 == F1).all()
    Hp.assert_parity(L, s, x, y1, F1, None, score_tol=None, label="after a cleared time-out")
    assert lib.tardis_debug_wait_timeout(h, -1, None) == 1
    T.tardis_destroy(h)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_save_and_load_round_trip(tmp_path, dtype):
    """A handle written to a file and read back gives the same flags and scores bit for bit, outputs within the parity
    tolerance of the oracle, and the same footprint; a damaged file is refused."""
    cfg = W.LayerConfig("saveload_" + dtype, 512, 2048, dtype=dtype, n_calib=512)
    L = _layer(cfg)
    s = L.numpy64()
    x = W.make_tokens(cfg, 21, 6).cuda()
    h = T.fold_layer(L)
    path = str(tmp_path / "layer.tardis")
    T.tardis_save(h, path)
    h2 = T.tardis_load(path)
    calls = [1, 4, 16]
    y1, F1, S1 = Hp.gpu_forward(h, L, x, calls)
    y2, F2, S2 = Hp.gpu_forward(h2, L, x, calls)
    assert (F1 == F2).all() and np.array_equal(S1, S2, equal_nan=True)
    Hp.assert_parity(L, s, x, y2, F2, None, score_tol=None, label="loaded handle")
    st1, st2 = T.tardis_stats(h), T.tardis_stats(h2)
    for k in ("bytes_folded", "bytes_predictor", "bytes_tables", "bytes_w1", "bytes_w2t"):
        assert st1[k] == st2[k]
    Wf1 = torch.empty(cfg.d_model, cfg.d_model, dtype=x.dtype, device="cuda")
    Wf2 = torch.empty_like(Wf1)
    T.tardis_export_folded(h, Wf1, None)
    T.tardis_export_folded(h2, Wf2, None)
    torch.cuda.synchronize()
    assert torch.equal(Wf1, Wf2)
    T.tardis_destroy(h)
    T.tardis_destroy(h2)
    # one flipped byte in the middle, and a truncated file: TARDIS_ERR_CORRUPT (6), no handle
    raw = bytearray(open(path, "rb").read())
    raw[len(raw) // 2] ^= 0x40
    bad = str(tmp_path / "bad.tardis")
    open(bad, "wb").write(raw)
    lib = T.load_library()
    out = ctypes.c_void_p()
    assert lib.tardis_load(bad.encode(), None, ctypes.byref(out)) == 6 and out.value is None
    open(bad, "wb").write(raw[:len(raw) // 3])
    assert lib.tardis_load(bad.encode(), None, ctypes.byref(out)) == 6 and out.value is None


def test_buffers_of_destroyed_layers_are_taken_over_by_new_ones():
    """Layers folded, used and destroyed in turn by two threads on streams of their own, the memory of one going to the next, give the results of a layer folded alone, and nothing stays registered as alive."""
    import threading
    cfgs = [W.LayerConfig("pool%d" % i, 512, 2048, n_calib=256, bias=bool(i)) for i in range(2)]
    Ls = [_layer(c, i) for i, c in enumerate(cfgs)]
    x = W.make_tokens(cfgs[0], 9, 5).cuda()
    want, live0 = [], T.tardis_debug_live_allocations()
    for L in Ls:
        h = T.fold_layer(L)
        want.append(T.tardis_ffn_forward(h, x, torch.empty_like(x)).clone())
        torch.cuda.synchronize()
        T.tardis_destroy(h)
    bad = []

    def work(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(6):
                h = T.fold_layer(Ls[i])
                y = T.tardis_ffn_forward(h, x, torch.empty_like(x))
                s.synchronize()
                if not (y.float() - want[i].float()).abs().max() <= 2e-2 * want[i].float().abs().max() or T.tardis_stats(h)["device_error"]:
                    bad.append(i)
                T.tardis_destroy(h)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad and T.tardis_debug_live_allocations() == live0


@pytest.mark.parametrize("d,h,G,bits", [(64, 32, 16, 2), (136 - 8, 96, 32, 3), (272, 1056, 16, 4), (400, 544, 80, 8), (1040, 160, 16, 2)])
def test_f32_kernels_at_the_edges_of_their_tiles(d, h, G, bits):
    # tiles of 32 outputs, 16 or 8 tokens, passes of 128 channels (a slice of 16 per warp) of d, then of h; 256 tokens per pass
    cfg = W.LayerConfig("f32edge%d" % d, d, h, dtype="f32", group=G, bits=bits, n_calib=256)
    calls = [1, 7, 8, 9, 16, 17, 33, 255, 257]
    _run(cfg, sum(calls), calls)


@pytest.mark.parametrize("d,h,bits,q,calls", [(144, 4800, 2, 0.02, [1, 8, 9, 17, 33]), (144, 4800, 4, 0.12, [3, 16, 40]), (288, 4800, 3, 0.35, [2, 9, 24]),
                                              (144, 2400, 8, 0.3, [16, 17, 32]), (768, 320, 2, 0.1, [40, 48, 64])])
def test_f32_scores_first_then_flagged_pairs_or_a_second_walk(d, h, bits, q, calls):
    # more tiles of 32 neurons and 8 or 16 tokens than SMs (150 of them, or 75 where 16 tokens are one walk and 17 are not), with few
    # pairs flagged in a tile, about the quarter where the second walk begins, and most; output tiles whose parts are a number of CTAs
    # that does not divide them (768 channels x 48 tokens: threes)
    cfg = W.LayerConfig("f32two%d" % d, d, h, dtype="f32", group=16, bits=bits, n_calib=256, q_lo=q, q_hi=1 - q)
    _run(cfg, sum(calls), calls)


@pytest.mark.parametrize("d,h,G,q", [(128, 32, 64, 0.05), (192, 96, 64, 0.2), (576, 2080, 192, 0.05), (1152, 4640, 128, 0.1), (640, 19040, 64, 0.02)])
def test_kernels_for_a_few_tokens_at_the_edges_of_their_tiles(d, h, G, q):
    # columns of 16 (two-term corrections), 32, 64, 128 tokens; neuron tiles of 16 to 128 rows with a short last one, one or several
    # per CTA; output tiles of 128 columns with a short last one; more neuron blocks than CTAs and fewer
    cfg = W.LayerConfig("fewedge%d" % d, d, h, group=G, n_calib=256, q_lo=q, q_hi=1 - q, act=W.ACT_GELU_ERF if d == 192 else W.ACT_GELU_TANH)
    calls = [1, 5, 16, 17, 32, 33, 64, 65, 127, 128, 2]
    _run(cfg, sum(calls), calls, path=3)


@pytest.mark.parametrize("d,bits,n", [(512, 2, 5), (576, 2, 16), (512, 2, 40), (512, 4, 33), (512, 2, 128), (512, 2, 200), (512, 3, 200), (1088, 4, 150)])
def test_scores_near_range_ends_in_every_number_per_tile(d, bits, n):
    # 0 to 20 scores per tile that the fast sums cannot place: a warp for each of eight, the last one to four shared out.  Tiles have 16
    # neurons here (2048 over 148 CTAs); the ends lie 2e-5 above or below scores of two tokens, well inside the allowance and well
    # outside the band in which either outcome is right
    h = 2048
    cfg = W.LayerConfig("nearends", d, h, group=64, n_calib=256, bits=bits)
    L = _layer(cfg, 3)
    x = W.make_tokens(cfg, n, 3).cuda()
    if n > 128:                                                     # (the prompt path: a warp per score of a token)
        x[0, ::7] *= 2.0 ** -30
        x[1, :16] = 0.0
    s = L.numpy64()
    zhat = O.predictor_score(x.double().cpu().numpy(), s["codes"], s["scale"], s["zero"], s["group"], s["b1"], s["bits"])
    lo = np.full(h, -50.0)
    hi = np.full(h, 50.0)
    wanted = 0
    for tile in range(h // 16):
        k = tile % 21
        wanted += k
        for i in range(k):
            j, off = tile * 16 + i % 16, 2e-5 if (tile + i) % 3 else -2e-5
            if i < 16:
                lo[j] = zhat[tile % 2, j] + off
            else:
                hi[j] = max(zhat[n - 1, j] + off, lo[j] + 1e-3)
    L.lo.copy_(torch.from_numpy(lo))
    L.hi.copy_(torch.from_numpy(hi))
    h1 = T.fold_layer(L)
    try:
        T.tardis_set_path(h1, 3)
        y, F, S = Hp.gpu_forward(h1, L, x)
        Hp.assert_parity(L, L.numpy64(), x, y, F, S, label="near ends", score_tol=3e-4)
        assert T.tardis_stats(h1)["exact_rechecks"] >= 0.9 * wanted
    finally:
        T.tardis_destroy(h1)


@pytest.mark.parametrize("d,h,G,q", [(64, 32, 64, 0.4), (192, 160, 64, 0.2), (1088, 4640, 64, 0.05), (1024, 4096, 128, 0.1)])
def test_kernels_for_a_few_tokens_with_4_bit_codes(d, h, G, q):
    # one channel block and several, an odd number of them, tiles with a short last one, every width of the token columns
    cfg = W.LayerConfig("few4bit%d" % d, d, h, group=G, n_calib=256, q_lo=q, q_hi=1 - q, bits=4)
    calls = [1, 3, 16, 17, 33, 64, 65, 128]
    _run(cfg, sum(calls), calls)


@pytest.mark.parametrize("d,h,G,bits", [(16, 32, 16, 2), (80, 96, 16, 4), (160, 224, 32, 3), (208, 1056, 16, 2), (64, 64, 64, 8)])
def test_set_up_kernels_at_the_edges_of_their_tiles(d, h, G, bits):
    # transposes of 64 x 64 tiles, two elements per access, with sides that end inside a tile; dequantised codes of every width
    cfg = W.LayerConfig("setup%d" % d, d, h, group=G, bits=bits, n_calib=256)
    _run(cfg, 9, path=1)
    if bits <= 4:
        _run(cfg, 140, path=3)
    L = _layer(cfg)
    hd = T.fold_layer(L)
    try:
        Wf, bf = torch.empty(d, d, dtype=torch.bfloat16, device="cuda"), torch.empty(d, device="cuda")
        T.tardis_export_folded(hd, Wf, bf)
        ref, bref = O.fold(*[L.numpy64()[k] for k in ("W1", "W2", "a", "c", "b1", "b2")])
        # one rounding to bf16 of sums whose terms keep 16 bits
        assert np.abs(Wf.double().cpu().numpy() - ref).max() <= 2.0 ** -8 * np.abs(ref).max()
        assert np.abs(bf.double().cpu().numpy() - bref).max() <= 1e-5 * max(1.0, np.abs(bref).max())
    finally:
        T.tardis_destroy(hd)


@pytest.mark.parametrize("d,h,G,q", [(64, 32, 64, 0.4), (320, 2400, 64, 0.2), (4096, 16384, 128, 0.05), (4608, 18944, 64, 0.1),
                                     (4672, 4768, 64, 0.1), (8192, 2400, 128, 0.4)])
def test_fused_kernels_at_the_edges_of_their_rings(d, h, G, q):
    # one to four tokens in one launch (three and four: the codes as bf16), one tile in all, tiles that all have a buffer and tiles that
    # share them, as many channels as fit; wider layers: one token per launch, more flagged rows than row slots, CTAs with none
    cfg = W.LayerConfig("fusededge%d" % d, d, h, group=G, n_calib=256, q_lo=q, q_hi=1 - q)
    calls = [1, 3, 4, 2, 3]
    _run(cfg, sum(calls), calls, path=2)


@pytest.mark.parametrize("n", [12, 60, 200])
def test_corrections_of_the_largest_pre_activations_are_finite(n):
    # beyond 2^127 twice a pre-activation is no float; with a bias of 2e38 and output weights of 2^-120 the neuron gives some 150 to every output
    cfg = W.LayerConfig("largest", 256, 512, group=64, n_calib=256)
    L = _layer(cfg, 4)
    L.b1[5], L.a[5], L.W2[:, 5] = 2e38, 0.5, 2.0 ** -120
    x = W.make_tokens(cfg, n, 4).cuda()
    h = T.fold_layer(L)
    try:
        y, F, S = Hp.gpu_forward(h, L, x)
        assert F[:, 5].all()
        Hp.assert_parity(L, L.numpy64(), x, y, F, None, label="largest")
    finally:
        T.tardis_destroy(h)


def test_first_call_of_a_process_may_be_a_chain_under_capture():
    # every kernel of a chain has to be loaded and to have its shared memory when the layers are set up: a process of its own, whose first
    # forward call is captured, and the shape of each of the four sets of kernels
    import subprocess
    import sys
    script = r"""
import sys
import torch
import paper_2501_10054_b200 as T
import workloads as W
for d, G in ((256, 64), (256, 128), (4544, 64), (4224, 128)):
    cfg = W.LayerConfig("capture%d" % d, d, 512, group=G, n_calib=256)
    L = [W.make_layer(cfg, s, device=torch.device("cuda", 0)) for s in (1, 2)]
    handles = [T.fold_layer(l) for l in L]
    for n in (1, 2, 4):
        x = torch.randn(n, d, device="cuda").bfloat16()
        y, work = torch.empty_like(x), torch.empty(2, n, d, dtype=x.dtype, device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            T.tardis_stack_forward(handles, x, y, work=work)
        graph.replay()
        torch.cuda.synchronize()
        captured = y.clone()
        T.tardis_stack_forward(handles, x, y, work=work)
        torch.cuda.synchronize()
        assert T.tardis_stats(handles[0])["last_path"] == 2
        assert (captured.float() - y.float()).abs().max() <= 2e-2 * y.float().abs().max(), (d, G, n)
        del graph
    for h in handles:
        T.tardis_destroy(h)
"""
    r = subprocess.run([sys.executable, "-c", script], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("d,dtype", [(16, "f32"), (1040, "f32"), (4096, "bf16"), (4160, "bf16"), (8256, "bf16")])
def test_stack_normalisation_at_the_edges_of_its_vectors(d, dtype):
    # one, two and three vectors of 8 elements per thread of 512, the last ones partly beyond the row; x apart from y and in place
    cfg = W.LayerConfig("norm%d" % d, d, 32, group=16 if d < 64 else 16 * (2 if d % 32 == 0 else 1), dtype=dtype, n_calib=64)
    L = _layer(cfg, 1)
    x = (W.make_tokens(cfg, 3, 1).cuda().float() * 3 + 0.5).to(L.W1.dtype)
    gam, bet = torch.linspace(0.5, 2, d, device="cuda"), torch.linspace(-1, 1, d, device="cuda")
    h = T.fold_layer(L)
    try:
        for in_place in (False, True):
            xs = x.clone()
            y = xs if in_place else torch.empty_like(x)
            keep = torch.empty(2, 2, 3, d, dtype=x.dtype, device="cuda")
            T.tardis_stack_forward([h, h], xs, y, [gam, bet], [bet, gam], keep=keep)
            torch.cuda.synchronize()
            assert in_place or torch.equal(xs, x)
            s = x
            for l, (a, b) in enumerate(((gam, bet), (bet, gam))):
                u = torch.nn.functional.layer_norm(s.double(), (d,), a.double(), b.double(), 1e-5)
                # one rounding to the dtype (bf16 has 8 significant bits: half a unit in the last is at most 2^-8 of the value; fp32: 2^-24)
                # plus the fp32 mean and deviation (a few 1e-6 of values below 10)
                assert ((keep[l, 0].double() - u).abs() <= (2.0 ** -8 if dtype == "bf16" else 0) * u.abs() + 3e-5).all()
                s = (s.float() + keep[l, 1].float()).to(x.dtype)
            assert torch.equal(y, s)
    finally:
        T.tardis_destroy(h)


@pytest.mark.parametrize("d,group,n", [(64, 64, 1), (320, 64, 2), (1024, 128, 3), (1024, 64, 4), (4096, 128, 1), (4096, 128, 2), (4096, 128, 4), (4544, 64, 2), (4608, 64, 3)])
@pytest.mark.parametrize("aligned", [True, False])
def test_chain_normalised_inside_the_fused_kernel(d, group, n, aligned):
    # the row in less than one warp's vectors, in one vector per thread, several tokens' vectors per thread; tables that 16-byte loads can
    # and cannot read; no tables; the last CTA's addition to the stream, in place and not
    cfg = W.LayerConfig("chain%d" % d, d, 256, group=group, n_calib=64)
    L = _layer(cfg, 1)
    x = (W.make_tokens(cfg, n, 1).cuda().float() * 3 + 0.5).to(L.W1.dtype)
    room = torch.empty(2, d + 1, device="cuda")
    gam, bet = (r[:d] if aligned else r[1:] for r in room)
    gam.copy_(torch.linspace(0.5, 2, d))
    bet.copy_(torch.linspace(-1, 1, d))
    h = T.fold_layer(L)
    try:
        for in_place, ga, be in ((False, [gam, gam], [bet, bet]), (True, None, [bet, bet]), (True, [gam, gam], None)):
            xs = x.clone()
            y = xs if in_place else torch.empty_like(x)
            keep = torch.empty(2, 2, n, d, dtype=x.dtype, device="cuda")
            T.tardis_stack_forward([h, h], xs, y, ga, be, keep=keep)
            torch.cuda.synchronize()
            assert in_place or torch.equal(xs, x)
            s = x
            for l in range(2):
                u = torch.nn.functional.layer_norm(s.double(), (d,), None if ga is None else gam.double(), None if be is None else bet.double(), 1e-5)
                # (one rounding to bf16, plus the fp32 mean and deviation)
                assert ((keep[l, 0].double() - u).abs() <= 2.0 ** -8 * u.abs() + 3e-5).all()
                f = torch.empty_like(x)
                T.tardis_ffn_forward(h, keep[l, 0].contiguous(), f)
                # (the same kernel on the same input: only the order of the sums differs)
                assert (f.float() - keep[l, 1].float()).abs().max() <= 2.0 ** -7 * f.float().abs().max()
                s = (s.float() + keep[l, 1].float()).to(x.dtype)
            assert torch.equal(y, s)
            T.tardis_set_deterministic(h, True)                      # (the small kernels between the layers: the same sums in the same order)
            apart = torch.empty_like(keep)
            T.tardis_stack_forward([h, h], x.clone(), torch.empty_like(x), ga, be, keep=apart)
            torch.cuda.synchronize()
            T.tardis_set_deterministic(h, False)
            assert torch.equal(apart[0, 0], keep[0, 0])
    finally:
        T.tardis_destroy(h)


def _at_range_ends(d, h, bits, group, seed):
    """A ReLU layer without biases whose ranges all end at 0."""
    L = _layer(W.LayerConfig("ends%d" % bits, d, h, bits=bits, group=group, n_calib=128, act=W.ACT_RELU, bias=False), seed)
    L.lo.fill_(float("-inf"))
    L.hi.zero_()
    L.a.zero_()
    L.c.zero_()
    return L


@pytest.mark.parametrize("d,bits,group", [(512, 2, 64), (512, 4, 64), (512, 3, 64), (512, 2, 16), (4672, 2, 64)])
def test_tokens_of_zeros_on_range_ends_need_no_re_evaluation(d, bits, group):
    # such a token's scores are the biases, here exactly the range ends: nothing is uncertain about them
    L = _at_range_ends(d, 2080, bits, group, 7)
    h = T.fold_layer(L)
    try:
        for path in (0, 3):
            T.tardis_set_path(h, path)
            for n in (1, 2, 4, 9, 60, 150):
                y, F, S = Hp.gpu_forward(h, L, torch.zeros(n, d, dtype=L.W1.dtype, device="cuda"))
                assert F.all() and (S == 0).all() and T.tardis_stats(h)["exact_rechecks"] == 0
                assert (y == (0 if L.b2 is None else L.b2.to(y.dtype))).all()
    finally:
        T.tardis_destroy(h)


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("n", [3, 40, 150])
def test_more_scores_on_range_ends_than_are_queued(bits, n):
    # every neuron has the same predictor row, and the ranges end at token 0's score: one neuron below the next above it
    L = _layer(W.LayerConfig("crowd%d" % bits, 512, 2080, bits=bits, group=64, n_calib=128), 9)
    for v in (L.codes, L.scale, L.zero):
        v[:] = v[:1].clone()
    L.b1.zero_()
    s = L.numpy64()
    x = W.make_tokens(L.cfg, n, 9).cuda()
    z = np.float32(O.predictor_score(x[:1].double().cpu().numpy(), s["codes"], s["scale"], s["zero"], s["group"], s["b1"], s["bits"])[0, 0])
    L.lo.fill_(float(z) - 1.0)
    ends = [z, np.nextafter(z, np.float32(np.inf)), np.nextafter(z, np.float32(-np.inf))]
    L.hi[:] = torch.tensor([ends[j % 3] for j in range(2080)], device="cuda")
    s = L.numpy64()
    h = T.fold_layer(L)
    try:
        for path in (0, 3):
            T.tardis_set_path(h, path)
            _, F, _ = Hp.gpu_forward(h, L, x)
            zhat = O.predictor_score(x.double().cpu().numpy(), s["codes"], s["scale"], s["zero"], s["group"], s["b1"], s["bits"])
            sure = np.abs(zhat - s["hi"]) > 1e-9 * np.abs(zhat)      # (fp64 sums in another order: 512 2^-53 of the terms)
            assert (F == O.flags_from_score(zhat, s["lo"], s["hi"]))[sure].all() and sure.mean() > 0.6
    finally:
        T.tardis_destroy(h)


@pytest.mark.parametrize("n", [20, 130])
def test_allowance_of_scores_whose_values_of_three_scales_are_bf16_values(n):
    # scales that are powers of two: 3 s needs no second bf16 term, and yet a term of a score may be 3 s |x|; range ends at 0.8 of the
    # allowance 3 2^-17 max s |x|_1 from the scores of the call's (equal) tokens have to be re-evaluated
    L = _layer(W.LayerConfig("pow2", 512, 2048, group=64, n_calib=128, bias=False), 4)
    L.scale[:] = torch.exp2(torch.floor(torch.log2(L.scale.float()))).to(L.scale.dtype)
    L.zero[:] = torch.where(torch.arange(8, device="cuda") % 2 == 0, 0, 3).to(torch.uint8)
    s = L.numpy64()
    x = W.make_tokens(L.cfg, 1, 4).cuda().expand(n, 512).contiguous()
    z = O.predictor_score(x[:1].double().cpu().numpy(), s["codes"], s["scale"], s["zero"], s["group"], s["b1"], s["bits"])[0]
    tau = 3 * 2.0 ** -17 * np.abs(s["scale"]).max(axis=1) * float(x[0].double().abs().sum())
    L.lo.fill_(float("-inf"))
    L.hi.fill_(float("inf"))
    L.hi[:100] = torch.tensor((z + 0.8 * tau)[:100], dtype=torch.float32, device="cuda")
    h = T.fold_layer(L)
    try:
        T.tardis_set_path(h, 3)
        _, F, _ = Hp.gpu_forward(h, L, x)
        assert not F.any() and T.tardis_stats(h)["exact_rechecks"] == 100 * n
    finally:
        T.tardis_destroy(h)


def test_queue_for_re_evaluation_grows_with_the_layer():
    # 800 of 16384 neurons with a range end on the score of the call's (equal) tokens: those are re-evaluated and no others
    L = _layer(W.LayerConfig("queue", 64, 16384, group=64, n_calib=64), 2)
    x = W.make_tokens(L.cfg, 1, 2).cuda().expand(130, 64).contiguous()
    s = L.numpy64()
    z = O.predictor_score(x[:1].double().cpu().numpy(), s["codes"], s["scale"], s["zero"], s["group"], s["b1"], s["bits"])[0]
    L.lo.fill_(float("-inf"))
    L.hi.fill_(float("inf"))
    L.hi[::20] = torch.tensor(z[::20], dtype=torch.float32, device="cuda")
    h = T.fold_layer(L)
    try:
        _, F, _ = Hp.gpu_forward(h, L, x)
        hi = L.hi.double().cpu().numpy()
        sure = np.abs(z - hi) > 1e-9 * np.abs(z)
        assert (F == (z >= hi))[:, sure].all() and T.tardis_stats(h)["exact_rechecks"] == 820 * 130
    finally:
        T.tardis_destroy(h)


LATE_WRITER = r"""
#include <stddef.h>
// lets the next launch of the stream start at once, writes dst = src only some time later (bounded)
__global__ void k_late(float* dst, const float* src, size_t count, long long cycles) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {}
  for (size_t i = threadIdx.x; i < count; i += blockDim.x) dst[i] = src[i];
}
extern "C" int late_write(float* dst, const float* src, size_t count, long long cycles, void* stream) {
  k_late<<<1, 256, 0, static_cast<cudaStream_t>(stream)>>>(dst, src, count, cycles);
  return cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def late_write(tmp_path_factory):
    """late_write(dst, src, cycles): dst = src on the current stream, written by a kernel that has let the next launch start before."""
    import subprocess
    from paper_2501_10054_b200.build import nvcc_path
    d = tmp_path_factory.mktemp("late")
    (d / "late.cu").write_text(LATE_WRITER)
    subprocess.run([nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-shared", "-Xcompiler", "-fPIC", "-o", str(d / "late.so"), str(d / "late.cu")],
                   check=True)
    fn = ctypes.CDLL(str(d / "late.so")).late_write
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_longlong, ctypes.c_void_p]

    def call(dst, src, cycles):
        n = src.numel() * src.element_size()
        assert n % 4 == 0 and dst.numel() * dst.element_size() == n and 0 <= cycles <= 10 ** 9
        assert fn(dst.data_ptr(), src.data_ptr(), n // 4, cycles, torch.cuda.current_stream().cuda_stream) == 0
    return call


def test_stack_reads_gamma_and_beta_behind_the_launch_that_writes_them(late_write):
    cfg = W.LayerConfig("late", 512, 2048, n_calib=64)
    L = _layer(cfg, 1)
    x = W.make_tokens(cfg, 2, 1).cuda()
    gam, bet = torch.linspace(0.5, 2, 512, device="cuda"), torch.linspace(-1, 1, 512, device="cuda")
    g2, b2 = torch.zeros_like(gam), torch.zeros_like(bet)
    keep, want = (torch.empty(2, 2, 2, 512, dtype=x.dtype, device="cuda") for _ in range(2))
    y = torch.empty_like(x)
    h = T.fold_layer(L)
    try:
        T.tardis_set_deterministic(h, True)
        T.tardis_stack_forward([h, h], x, y, [gam, gam], [bet, bet], keep=want)
        torch.cuda.synchronize()
        for dst, src, ga, be in ((g2, gam, [g2, gam], [bet] * 2), (b2, bet, [gam] * 2, [b2, bet]), (g2, gam, [gam, g2], [bet] * 2), (b2, bet, [gam] * 2, [bet, b2])):
            for cycles in (2000, 20000, 2000000):
                dst.zero_()
                late_write(dst, src, cycles)
                T.tardis_stack_forward([h, h], x, y, ga, be, keep=keep)
                torch.cuda.synchronize()
                assert torch.equal(keep[:, 0], want[:, 0])
    finally:
        T.tardis_destroy(h)


@pytest.mark.parametrize("dtype,bits,d,h", [("bf16", 2, 1024, 8192), ("bf16", 4, 1024, 8192), ("bf16", 2, 4736, 2048), ("f32", 2, 1024, 8192)])
def test_destroy_and_the_builder_give_device_memory_back(dtype, bits, d, h):
    # a small layer first, so that kernels are loaded; then what a layer (over 100 MB) and the builder's scratch (8 d h bytes) take has
    # to be free again when the calls return
    for dd, hh in ((512, 2048), (d, h)):
        L = _layer(W.LayerConfig("back", dd, hh, dtype=dtype, bits=bits, group=64, n_calib=64))
        x = W.make_tokens(L.cfg, 150, 1).cuda()
        y = torch.empty_like(x)
        T.tardis_build_predictor(L.W1, None, bits, 64)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        T.tardis_build_predictor(L.W1, None, bits, 64)
        hd = T.fold_layer(L)
        for n in (1, 4, 40, 150):
            T.tardis_ffn_forward(hd, x[:n], y[:n])
        torch.cuda.synchronize()
        taken = free - torch.cuda.mem_get_info()[0]
        st = T.tardis_stats(hd)
        T.tardis_destroy(hd)
        left = free - torch.cuda.mem_get_info()[0]
    held = sum(v for k, v in st.items() if k.startswith("bytes_"))
    assert taken >= 50 << 20 and held <= taken <= held + (8 << 20) and left <= 2 << 20, (taken, held, left)


@pytest.mark.parametrize("dtype,bits,d,calls", [("bf16", 2, 512, [1, 4, 16, 17, 64, 128, 130]), ("bf16", 4, 512, [1, 33, 128]), ("bf16", 2, 4736, [1, 5]), ("f32", 2, 512, [3])])
def test_calls_behind_a_long_launch_that_lets_them_start_early(late_write, dtype, bits, d, calls):
    # the launch before writes the tokens 0.3 s after it has let the call's kernels start: longer than the kernels' own waits may take
    cfg = W.LayerConfig("patient", d, 2048, dtype=dtype, bits=bits, n_calib=64)
    L = _layer(cfg, 1)
    h = T.fold_layer(L)
    try:
        for n in calls:
            x = W.make_tokens(cfg, n, n).cuda()
            want, y = T.tardis_ffn_forward(h, x, torch.empty_like(x)), torch.empty_like(x)
            late = torch.zeros_like(x)
            torch.cuda.synchronize()
            late_write(late, x, 600000000)
            T.tardis_ffn_forward(h, late, y)
            assert T.tardis_stats(h)["device_error"] == 0
            assert ((y.float() - want.float()).abs() <= 2.0 ** -7 * want.float().abs() + 1e-3).all()   # (bf16 roundings of sums in another order)
    finally:
        T.tardis_destroy(h)


@pytest.mark.parametrize("dtype,bits,d,n", [("bf16", 2, 512, 1), ("bf16", 2, 512, 20), ("bf16", 4, 512, 3), ("bf16", 2, 4736, 2), ("f32", 2, 512, 5)])
def test_first_call_right_behind_the_fold(dtype, bits, d, n):
    # no wait in between, into memory that another layer's state has been in: the call has to find the new layer's state complete
    cfg = W.LayerConfig("behind", d, 2048, dtype=dtype, bits=bits, n_calib=64)
    layers = [_layer(cfg, seed) for seed in (1, 2)]
    x = W.make_tokens(cfg, n, 1).cuda()
    want = []
    for i in range(8):
        L = layers[i % 2]
        h = T.fold_layer(L)
        y = T.tardis_ffn_forward(h, x, torch.empty_like(x)).float()
        torch.cuda.synchronize()
        if i < 2:
            want.append(T.tardis_ffn_forward(h, x, torch.empty_like(x)).float())
        T.tardis_destroy(h)
        assert ((y - want[i % 2]).abs() <= 2.0 ** -7 * want[i % 2].abs() + 1e-3).all()      # (bf16 roundings of sums in another order)


@pytest.mark.parametrize("d,bits,most", [(512, 2, 4), (4736, 2, 3), (512, 4, 0)])
def test_largest_call_that_goes_to_the_decode_kernels(d, bits, most):
    cfg = W.LayerConfig("line%d" % d, d, 2048, bits=bits, n_calib=64)
    L = _layer(cfg, 1)
    s = L.numpy64()
    x = W.make_tokens(cfg, 5, 1).cuda()
    h = T.fold_layer(L)
    try:
        for n in range(1, 6):
            y, F, S = Hp.gpu_forward(h, L, x[:n])
            assert T.tardis_stats(h)["last_path"] == (2 if n <= most else 3)
            Hp.assert_parity(L, s, x[:n], y, F, S, score_tol=3e-4, label="%d tokens" % n)
    finally:
        T.tardis_destroy(h)
