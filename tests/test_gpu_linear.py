"""K3 parity: the GEMM kernels with their fused epilogues against fp64 matrix products."""
import numpy as np
import pytest
import torch

import lsp_synth as S
from oracle import dlm
from gpu_util import DEV

pytestmark = pytest.mark.gpu


def _dec(dtype):
    from paper_2603_05454_b200 import LSPDecoder, SchedCfg
    sh = S.ModelShape(1, 64, 1, 1, 64, 64, 128, dtype=dtype)
    return LSPDecoder(sh, S.make_weights(sh, 0, device=DEV), SchedCfg(), 1, 8, device=DEV)


def _check(dtype, impl, M, N, K, seed):
    tdt = torch.float32 if dtype == "fp32" else torch.bfloat16
    dec = _dec(dtype)
    dec.set_option(0, impl)
    A = S.normal((M, K), seed, 1, 1.0, tdt, DEV)
    W = S.normal((N, K), seed, 2, 0.05, tdt, DEV)
    W2 = S.normal((N, K), seed, 3, 0.05, tdt, DEV)
    X0 = S.normal((M, N), seed, 4, 1.0, tdt, DEV)
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    rnd = dlm.round_bf16 if dtype == "bf16" else (lambda x: x.astype(np.float32).astype(np.float64))
    a, w, w2, x0 = f64(A), f64(W), f64(W2), f64(X0)
    rtol = 2e-5 if dtype == "fp32" else 1.0 / 128   # one bf16 ulp of the result (rounding point may flip)
    out = torch.empty(M, N, dtype=tdt, device=DEV)
    dec.op_linear(0, A, W, None, out)
    ref = a @ w.T
    np.testing.assert_allclose(f64(out), rnd(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05)
    xr = X0.clone()
    dec.op_linear(1, A, W, None, xr)
    ref = x0 + a @ w.T
    np.testing.assert_allclose(f64(xr), rnd(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05)
    dec.op_linear(2, A, W, W2, out)
    g, u = a @ w.T, a @ w2.T
    ref = g / (1 + np.exp(-g)) * u
    np.testing.assert_allclose(f64(out), rnd(ref), rtol=rtol * 2, atol=rtol * np.abs(ref).max() * 0.05)
    dec.close()


@pytest.mark.parametrize("shape", [(1, 64, 64), (70, 144, 192), (129, 256, 128), (300, 512, 1024)])
def test_linear_fp32(shape):
    _check("fp32", 0, *shape, seed=0)


@pytest.mark.parametrize("impl", [0, 1])
@pytest.mark.parametrize("shape", [(1, 64, 64), (70, 144, 192), (129, 256, 128), (300, 512, 1024),
                                   (512, 4096, 4096), (37, 12288, 4096), (257, 4096, 12288)])
def test_linear_bf16(impl, shape):
    _check("bf16", impl, *shape, seed=1)


@pytest.mark.parametrize("grid_mode", [1, 2])
@pytest.mark.parametrize("shape", [(1, 256, 128), (5, 384, 256), (64, 1152, 512), (128, 4096, 4096), (100, 12288, 4096),
                                   (17, 4096, 12288), (129, 384, 256), (200, 4096, 4096), (256, 12288, 4096),
                                   (190, 1152, 576)])
def test_linear_bf16_weight_streaming_kernel(grid_mode, shape):
    """M <= 128 takes the persistent streaming kernel with both ways of dealing out the work: even shares over all SMs (tiles split
    anywhere, partials in scratch, summed by the last arriver) and equal K slices per tile (on clusters).  The row counts above
    that go to the pairs of SMs, beside the line."""
    M, N, K = shape
    tdt = torch.bfloat16
    dec = _dec("bf16")
    dec.debug_set(17, grid_mode)
    A = S.normal((M, K), 2, 1, 1.0, tdt, DEV)
    W = S.normal((N, K), 2, 2, 0.05, tdt, DEV)
    W2 = S.normal((N, K), 2, 3, 0.05, tdt, DEV)
    X0 = S.normal((M, N), 2, 4, 1.0, tdt, DEV)
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    a, w, w2, x0 = f64(A), f64(W), f64(W2), f64(X0)
    rtol = 1.0 / 128
    out = torch.empty(M, N, dtype=tdt, device=DEV)
    outs = []
    for rep in range(2):                       # twice: the tile counters must be back at zero after a launch
        dec.op_linear(0, A, W, None, out)
        ref = a @ w.T
        np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05)
        outs.append(out.clone())
    assert torch.equal(outs[0], outs[1])       # deterministic summation order
    xr = X0.clone()
    dec.op_linear(1, A, W, None, xr)
    ref = x0 + a @ w.T
    np.testing.assert_allclose(f64(xr), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05)
    dec.op_linear(2, A, W, W2, out)
    g, u = a @ w.T, a @ w2.T
    ref = g / (1 + np.exp(-g)) * u
    np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol * 2, atol=rtol * np.abs(ref).max() * 0.05)
    dec.close()


@pytest.mark.parametrize("case", [
    # (M, N, K, options): K slices on clusters of two (64 to 74 tiles of 128 columns), with the half-tile exchange, without it, and
    # below its row count; of four and eight; through global scratch instead of clusters
    (100, 8192, 4096, {}), (100, 8192, 4096, {33: 0}), (128, 8192, 1024, {33: 0}), (33, 8192, 1024, {}), (33, 8192, 1024, {44: 0}),
    (64, 9216, 1088, {33: 0}), (100, 4096, 4096, {}), (128, 1040, 4096, {}), (100, 4096, 4096, {29: 0}), (128, 8192, 1024, {29: 0}),
    (17, 1040, 2048, {29: 0}),
    # SwiGLU GEMM with 192-wide tiles (96 pairs) and a forced 256 for contrast
    (100, 12288, 256, {}), (100, 12288, 256, {32: 256}), (64, 9600, 1024, {32: 192}),
    # more than 128 rows: pairs of SMs, few tiles and many, with and without K slices
    (200, 4096, 4096, {}), (256, 12288, 4096, {}), (130, 4096, 12288, {}), (640, 4096, 12288, {}), (1000, 3584, 3584, {}),
    (300, 2048, 1024, {}), (257, 512, 2048, {}), (640, 4096, 4096, {}), (200, 12288, 1024, {}), (200, 12288, 320, {}),
    (600, 12288, 256, {}), (300, 9600, 192, {}),
])
def test_linear_bf16_split_tiles(case):
    """Every way of splitting a tile's K and of summing the slices, against fp64 products; twice the same bits."""
    M, N, K, opts = case
    tdt = torch.bfloat16
    dec = _dec("bf16")
    for k, v in opts.items():
        dec.debug_set(k, v)
    A = S.normal((M, K), 3, 1, 1.0, tdt, DEV)
    W = S.normal((N, K), 3, 2, 0.05, tdt, DEV)
    W2 = S.normal((N, K), 3, 3, 0.05, tdt, DEV)
    X0 = S.normal((M, N), 3, 4, 1.0, tdt, DEV)
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    a, w, w2, x0 = f64(A), f64(W), f64(W2), f64(X0)
    rtol = 1.0 / 128
    out = torch.empty(M, N, dtype=tdt, device=DEV)
    outs = []
    for rep in range(2):
        dec.op_linear(0, A, W, None, out)
        ref = a @ w.T
        np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05)
        outs.append(out.clone())
    assert torch.equal(outs[0], outs[1])       # rank-order summation: the same bits every time
    xr = X0.clone()
    dec.op_linear(1, A, W, None, xr)
    ref = x0 + a @ w.T
    np.testing.assert_allclose(f64(xr), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05)
    dec.op_linear(2, A, W, W2, out)
    g, u = a @ w.T, a @ w2.T
    ref = g / (1 + np.exp(-g)) * u
    np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol * 2, atol=rtol * np.abs(ref).max() * 0.05)
    dec.close()


def test_linear_bf16_seeded_random_shapes_and_kernel_options():
    """Sixty seeded random (rows, columns, K, option) combinations across the row regimes (one tile; pairs of SMs with one row group
    and several), the split paths (clusters of 2..8, half-tile exchange, global scratch, K slices on pairs) and the tile widths."""
    import random
    rng = random.Random(7)
    dec = _dec("bf16")
    defaults = {29: 1, 33: 1, 23: 0, 32: 0, 17: 2, 41: 0, 42: 0, 46: 0}
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    rows = [1, 2, 5, 17, 32, 33, 64, 100, 128, 129, 190, 256, 257, 300, 400, 512, 640, 768, 1000, 1100, 1536, 2100]
    done = 0
    while done < 60:
        M, N, K = rng.choice(rows), rng.choice([96, 128, 384, 1152, 2048, 3584, 4096, 4608, 9600, 12288]), \
            rng.choice([64, 192, 320, 1024, 2048, 3584, 4096])
        if M * N * K > 2e10:
            continue
        opts = {}
        for key, p, vals in ((29, 0.2, [0]), (33, 0.2, [0]), (41, 0.15, [96, 128, 224]), (23, 0.15, [128, 256]),
                             (32, 0.15, [192, 256]), (17, 0.1, [1]), (42, 0.1, [1, 2]), (46, 0.3, [1, 2, 3])):
            if rng.random() < p:
                opts[key] = rng.choice(vals)
        for k, v in {**defaults, **opts}.items():
            dec.debug_set(k, v)
        A = S.normal((M, K), done, 1, 1.0, torch.bfloat16, DEV)
        W = S.normal((N, K), done, 2, 0.05, torch.bfloat16, DEV)
        W2 = S.normal((N, K), done, 3, 0.05, torch.bfloat16, DEV)
        X0 = S.normal((M, N), done, 4, 1.0, torch.bfloat16, DEV)
        a, w, w2, x0 = f64(A), f64(W), f64(W2), f64(X0)
        rtol = 1.0 / 128
        out = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)
        tag = f"M={M} N={N} K={K} options={opts}"
        dec.op_linear(0, A, W, None, out)
        ref = a @ w.T
        np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05, err_msg=tag)
        xr = X0.clone()
        dec.op_linear(1, A, W, None, xr)
        ref = x0 + a @ w.T
        np.testing.assert_allclose(f64(xr), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05, err_msg=tag)
        dec.op_linear(2, A, W, W2, out)
        g, u = a @ w.T, a @ w2.T
        ref = g / (1 + np.exp(-g)) * u
        np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol * 2, atol=rtol * np.abs(ref).max() * 0.05, err_msg=tag)
        done += 1
    dec.close()


def test_bounded_wait_expiry_is_reported_and_the_context_stays_usable():
    """A device-side wait that runs out (a barrier nothing arrives at, 200 microseconds) comes back as
    LSP_ERR_DEVICE_TIMEOUT with the site in the message; the status word is cleared, and the next GEMM is correct."""
    from paper_2603_05454_b200 import LSPError
    dec = _dec("bf16")
    A = S.normal((70, 192), 3, 1, 1.0, torch.bfloat16, DEV)
    W = S.normal((144, 192), 3, 2, 0.05, torch.bfloat16, DEV)
    out = torch.empty(70, 144, dtype=torch.bfloat16, device=DEV)
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    ref = dlm.round_bf16(f64(A) @ f64(W).T)
    for _ in range(2):
        with pytest.raises(LSPError) as e:
            dec.wait_selftest(200)
        assert e.value.code == -6 and "site 99" in str(e.value)
        dec.op_linear(0, A, W, None, out)               # synchronises and checks the status word: must be clean again
        np.testing.assert_allclose(f64(out), ref, rtol=1.0 / 128, atol=np.abs(ref).max() / 128 * 0.05)
    dec.close()


@pytest.mark.parametrize("M", [1, 48, 128, 200, 256, 384, 640, 1500])
def test_linear_bf16_third_model_shape(M):
    """A model shape none of the tile heuristics were fitted on (d 5120, 40/8 heads of 128, FFN 13824): the fused QKV
    width 7168, the O and down projections, the SwiGLU pair GEMM, at row counts of every regime."""
    dec = _dec("bf16")
    d, qd, kvd, f = 5120, 40 * 128, 8 * 128, 13824
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    rtol = 1.0 / 128
    for (N, K, op) in ((qd + 2 * kvd, d, 0), (d, qd, 1), (f, d, 2), (d, f, 1)):
        A = S.normal((M, K), 5, 1, 1.0, torch.bfloat16, DEV)
        W = S.normal((N, K), 5, 2, 0.03, torch.bfloat16, DEV)
        W2 = S.normal((N, K), 5, 3, 0.03, torch.bfloat16, DEV) if op == 2 else None
        out = S.normal((M, N), 5, 4, 1.0, torch.bfloat16, DEV)
        x0 = f64(out)
        dec.op_linear(op, A, W, W2, out)
        a, w = f64(A), f64(W)
        if op == 0:
            ref = a @ w.T
        elif op == 1:
            ref = x0 + a @ w.T
        else:
            g, u = a @ w.T, a @ f64(W2).T
            ref = g / (1 + np.exp(-g)) * u
        np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol * (2 if op == 2 else 1),
                                   atol=rtol * np.abs(ref).max() * 0.05, err_msg=f"M={M} N={N} K={K} op={op}")
    dec.close()


@pytest.mark.parametrize("M", [1, 16, 17, 100, 129, 144, 177, 200, 256])
def test_linear_bf16_layer_shapes_up_to_256_rows(M):
    """Layer shapes at row counts up to 256, on either side of the line between one SM and pairs of SMs: with and without K slices,
    ragged last tiles, all three epilogues, twice (bit-identical: the K slices are summed in rank order)."""
    dec = _dec("bf16")
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    rtol = 1.0 / 128
    for (N, K) in ((4096, 4096), (12288, 4096), (1152, 512), (384, 256), (3584, 18944), (4608, 3584), (144, 192)):
        A = S.normal((M, K), 7, 1, 1.0, torch.bfloat16, DEV)
        W = S.normal((N, K), 7, 2, 0.03, torch.bfloat16, DEV)
        W2 = S.normal((N, K), 7, 3, 0.03, torch.bfloat16, DEV)
        X0 = S.normal((M, N), 7, 4, 1.0, torch.bfloat16, DEV)
        a, w, w2, x0 = f64(A), f64(W), f64(W2), f64(X0)
        tag = f"M={M} N={N} K={K}"
        out = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)
        outs = []
        for _ in range(2):
            out.fill_(float("nan"))
            dec.op_linear(0, A, W, None, out)
            ref = a @ w.T
            np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05, err_msg=tag)
            outs.append(out.clone())
        assert torch.equal(outs[0], outs[1]), tag
        xr = X0.clone()
        dec.op_linear(1, A, W, None, xr)
        ref = x0 + a @ w.T
        np.testing.assert_allclose(f64(xr), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05, err_msg=tag)
        dec.op_linear(2, A, W, W2, out)
        g, u = a @ w.T, a @ w2.T
        ref = g / (1 + np.exp(-g)) * u
        np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol * 2, atol=rtol * np.abs(ref).max() * 0.05, err_msg=tag)
    dec.close()


@pytest.mark.parametrize("case", [(130, 12288, 256, {}), (150, 12288, 320, {}), (192, 12288, 256, {}), (177, 9600, 192, {}),
                                  (160, 12288, 256, {41: 256}), (193, 12288, 256, {}), (150, 12288, 256, {41: 128}),
                                  (140, 12288, 512, {42: 1})])
def test_linear_bf16_wide_ffn_just_above_one_row_tile(case):
    """130 to 193 rows of a wide FFN: one row group on pairs of SMs, its second half partly or wholly empty, at the automatic tile
    width and others, all three epilogues."""
    M, N, K, opts = case
    dec = _dec("bf16")
    for k, v in opts.items():
        dec.debug_set(k, v)
    A = S.normal((M, K), 9, 1, 1.0, torch.bfloat16, DEV)
    W = S.normal((N, K), 9, 2, 0.05, torch.bfloat16, DEV)
    W2 = S.normal((N, K), 9, 3, 0.05, torch.bfloat16, DEV)
    X0 = S.normal((M, N), 9, 4, 1.0, torch.bfloat16, DEV)
    f64 = lambda t: t.float().cpu().numpy().astype(np.float64)
    a, w, w2, x0 = f64(A), f64(W), f64(W2), f64(X0)
    rtol = 1.0 / 128
    out = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=DEV)
    dec.op_linear(2, A, W, W2, out)
    g, u = a @ w.T, a @ w2.T
    ref = g / (1 + np.exp(-g)) * u
    np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol * 2, atol=rtol * np.abs(ref).max() * 0.05)
    out.fill_(float("nan"))
    dec.op_linear(0, A, W, None, out)
    ref = a @ w.T
    np.testing.assert_allclose(f64(out), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05)
    xr = X0.clone()
    dec.op_linear(1, A, W, None, xr)
    ref = x0 + a @ w.T
    np.testing.assert_allclose(f64(xr), dlm.round_bf16(ref), rtol=rtol, atol=rtol * np.abs(ref).max() * 0.05)
    dec.close()


@pytest.mark.parametrize("case", [
    # (M, N, K, tile width 0 = automatic): row groups of 256 (one row of a second group, a group less one row), a ragged last
    # column tile, a half-empty last K chunk (odd multiples of 64), more tiles than pairs of SMs, several bands
    (257, 64, 64, 0), (511, 1152, 192, 0), (513, 4112, 320, 160), (300, 2048, 1024, 256), (700, 9600, 448, 96),
    (1030, 4096, 512, 224), (4610, 576, 4096, 0), (2600, 1040, 2048, 128),
])
def test_linear_bf16_on_pairs_of_sms(case):
    """More than 256 rows: the GEMM on pairs of SMs, at the edges of its tiles, against fp64 products of the same operands.
    One bf16 ulp of the result (1/128 relative), plus a twentieth of that of the largest, as in the tests above; the SwiGLU
    product has two factors."""
    M, N, K, bn = case
    dec = _dec("bf16")
    dec.debug_set(41, bn)
    A = S.normal((M, K), 11, 1, 1.0, torch.bfloat16, DEV)
    W = S.normal((N, K), 11, 2, 0.05, torch.bfloat16, DEV)
    W2 = S.normal((N, K), 11, 3, 0.05, torch.bfloat16, DEV)
    X0 = S.normal((M, N), 11, 4, 1.0, torch.bfloat16, DEV)
    ref, up = A.double() @ W.double().t(), A.double() @ W2.double().t()
    near = lambda got, want, ulps=1: bool(((got.double() - want).abs() <= ulps / 128 * want.abs() + want.abs().max() / 2560).all())
    out = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device=DEV)
    dec.op_linear(0, A, W, None, out[:M])
    assert near(out[:M], ref) and bool((out[M] == 7.0).all())
    x = torch.cat([X0, out[M:]])
    dec.op_linear(1, A, W, None, x[:M])
    assert near(x[:M], X0.double() + ref) and bool((x[M] == 7.0).all())
    dec.op_linear(2, A, W, W2, out[:M])
    assert near(out[:M], torch.nn.functional.silu(ref) * up, 2) and bool((out[M] == 7.0).all())
    dec.close()


@pytest.mark.parametrize("dh,hq,hkv,bn", [(128, 4, 2, 128), (128, 4, 2, 192), (128, 5, 5, 256), (64, 6, 2, 192), (64, 6, 2, 128),
                                              (128, 4, 2, 96), (128, 5, 5, 160), (64, 6, 2, 224),       # no multiples of 64: automatic
                                              (128, 4, 2, 64), (64, 6, 2, 64)])
def test_rotary_projection_on_pairs_of_sms(dh, hq, hkv, bn):
    """The rotary QKV projection of more than 256 rows (half tiles of whole head halves, or of 32-row pieces of them): the
    first layer's cached keys and values against the CUDA-core GEMM's.  Both round the same fp32 value up to the order of its
    sum, so they differ by at most one bf16 ulp (1/128 relative), with a floor of a ulp of the typical value for sums that
    cancel."""
    from paper_2603_05454_b200 import LSPDecoder, SchedCfg
    d, B, P, G = hq * dh, 2, 170, 9
    sh = S.ModelShape(1, d, hq, hkv, dh, 128, 256, dtype="bf16")
    w = S.make_weights(sh, 5, device=DEV)
    kv = []
    for impl in (1, 0):
        dec = LSPDecoder(sh, w, SchedCfg(), B, P + G, device=DEV)
        dec.set_option(0, impl)
        dec.debug_set(41, bn)
        tokens = torch.zeros(B, P + G, dtype=torch.int32, device=DEV)
        tokens[:, :P] = S.make_prompt(B, P, sh, 6).to(DEV)
        dec.begin(tokens, [P] * B, [G] * B)
        dec.denoise_step()
        dec.commit()
        torch.cuda.synchronize()
        kv.append(dec.kv_view()[0, :, :, :P].double())
        dec.close()
    typical = kv[1].square().mean().sqrt()
    assert bool(((kv[0] - kv[1]).abs() <= (kv[1].abs() + typical) / 128).all())


@pytest.mark.parametrize("P", [5, 28])
@pytest.mark.parametrize("dh,hq,hkv,d", [(128, 32, 32, 4096), (128, 72, 2, 1088), (128, 120, 12, 1152), (64, 64, 64, 1024), (128, 73, 1, 576),
                                         (128, 32, 32, 512), (128, 112, 16, 320), (64, 70, 70, 192)])
def test_rotary_projection_of_few_rows_keeps_its_sums(dh, hq, hkv, d, P):
    """75 to 148 whole tiles of 128 columns add K in the slices, and in the order, of the 256-wide tiles (23 = 256) that would be split over two
    or three CTAs, or not (K <= 512): the cache rows of the two are equal to the bit."""
    from paper_2603_05454_b200 import LSPDecoder, SchedCfg
    G = 4
    sh = S.ModelShape(1, d, hq, hkv, dh, 64, 256, dtype="bf16")
    w = S.make_weights(sh, 3, device=DEV)
    rows = []
    for width in (0, 256):
        dec = LSPDecoder(sh, w, SchedCfg(), 1, P + G, device=DEV)
        dec.debug_set(23, width)
        tokens = torch.zeros(1, P + G, dtype=torch.int32, device=DEV)
        tokens[:, :P] = S.make_prompt(1, P, sh, 7).to(DEV)
        dec.begin(tokens, [P], [G])
        dec.denoise_step()
        dec.commit([1])
        rows.append(dec.kv_view()[:, :, 0, :P].clone())
        dec.close()
    assert rows[0].float().abs().max() > 0.1
    assert torch.equal(*rows), float((rows[0].float() - rows[1].float()).abs().max())


@pytest.mark.parametrize("M,N,K,opts", [(5, 12288, 256, {}), (100, 384, 192, {}), (200, 12288, 320, {}), (128, 1152, 576, {43: 1}),
                                        (200, 12288, 320, {43: 1}), (64, 9600, 1024, {29: 0})])
@pytest.mark.parametrize("up_first", [False, True])
def test_swiglu_weights_by_one_copy_in_either_order(M, N, K, opts, up_first):
    """At most 256 rows: one copy brings a SwiGLU tile's gate and up rows whichever of the two tensors lies first in memory
    (the accumulators then come in that order), and by one copy per half and atom.  Two bf16 ulps: the product has two factors."""
    dec = _dec("bf16")
    for k, v in opts.items():
        dec.debug_set(k, v)
    W = S.normal((2, N, K), 12, 2, 0.05, torch.bfloat16, DEV)
    A = S.normal((M, K), 12, 1, 1.0, torch.bfloat16, DEV)
    gate, up = (W[1], W[0]) if up_first else (W[0], W[1])
    out = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)
    dec.op_linear(2, A, gate, up, out)
    want = torch.nn.functional.silu(A.double() @ gate.double().t()) * (A.double() @ up.double().t())
    assert bool(((out.double() - want).abs() <= want.abs() / 64 + want.abs().max() / 2560).all())
    dec.close()


@pytest.mark.parametrize("up_first", [False, True])
@pytest.mark.parametrize("gap", [0x20000000, 0x46402C00])
def test_swiglu_weights_far_apart(gap, up_first):
    """Gate and up projection half a gigabyte and more apart: no copy spans the two (see ST_MAX_SPAN)."""
    dec = _dec("bf16")
    M, N, K, bf = 26, 192, 512, torch.bfloat16
    A, W, W2 = S.normal((M, K), 3, 1, 1.0, bf, DEV), S.normal((N, K), 3, 2, 0.05, bf, DEV), S.normal((N, K), 3, 3, 0.05, bf, DEV)
    both = torch.empty(gap + N * K * 2, dtype=torch.uint8, device=DEV)
    at = lambda o, t: both[o:o + N * K * 2].view(bf).view(N, K).copy_(t)  # noqa: E731
    w, w2 = at(gap if up_first else 0, W), at(0 if up_first else gap, W2)
    out = torch.empty(M, N, dtype=bf, device=DEV)
    dec.op_linear(2, A, w, w2, out)
    dec.close()
    ref = torch.nn.functional.silu(A.double() @ W.double().t()) * (A.double() @ W2.double().t())
    assert bool(((out.double() - ref).abs() <= ref.abs() / 128 + 1e-3 * ref.abs().max()).all())      # one bf16 ulp, sums that cancel


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("M,N,K", [(1, 16, 64), (31, 48, 64), (33, 1040, 192), (128, 256, 1024), (129, 384, 256),
                                   (1200, 1024, 128), (1217, 1040, 64)])
def test_linear_cuda_core_kernels(dtype, M, N, K):
    """Both CUDA-core kernels (K split over a CTA's warps below two 64 x 64 tiles per SM, one tile per CTA above: the last two)
    at the edges of their tiles, fewer K steps than warps included."""
    _check(dtype, 0, M, N, K, seed=13)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("M,N,K", [(1, 16, 512), (40, 256, 512), (33, 272, 832), (128, 256, 1024), (64, 64, 4096)])
def test_linear_cuda_core_k_slices_on_a_cluster(dtype, M, N, K):
    """Few tiles and a long K: two or four K slices, of unequal length where K is no multiple, summed by the cluster's first CTA."""
    _check(dtype, 0, M, N, K, seed=12)


@pytest.mark.parametrize("M", [129, 187, 256])
@pytest.mark.parametrize("N,K", [(4096, 4096), (1152, 512), (4608, 3584), (7168, 5120), (4096, 12288), (16, 64)])
def test_linear_bf16_one_row_group_on_pairs(M, N, K):
    """129 to 256 rows on the pairs of SMs: one row group, tiles narrower than a box, ragged K, K slices or none."""
    dec = _dec("bf16")
    A = S.normal((M, K), 14, 1, 1.0, torch.bfloat16, DEV)
    W = S.normal((N, K), 14, 2, 0.05, torch.bfloat16, DEV)
    W2 = S.normal((N, K), 14, 3, 0.05, torch.bfloat16, DEV)
    X0 = S.normal((M, N), 14, 4, 1.0, torch.bfloat16, DEV)
    ref, up = A.double() @ W.double().t(), A.double() @ W2.double().t()
    near = lambda got, want, ulps=1: bool(((got.double() - want).abs() <= ulps / 128 * want.abs() + want.abs().max() / 2560).all())
    x = X0.clone()
    dec.op_linear(1, A, W, None, x)
    assert near(x, X0.double() + ref)
    out = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)
    dec.op_linear(2, A, W, W2, out)
    assert near(out, torch.nn.functional.silu(ref) * up, 2)
    dec.close()


@pytest.mark.parametrize("M,N,K", [(1, 512, 64), (64, 1024, 512), (128, 272, 448), (33, 4096, 512), (100, 1024, 576)])
def test_linear_bf16_short_k_without_a_split(M, N, K):
    """At most 512 elements of K: whole tiles per CTA instead of K slices on clusters (the last case is beyond the line)."""
    dec = _dec("bf16")
    A = S.normal((M, K), 16, 1, 1.0, torch.bfloat16, DEV)
    W = S.normal((N, K), 16, 2, 0.05, torch.bfloat16, DEV)
    W2 = S.normal((N, K), 16, 3, 0.05, torch.bfloat16, DEV)
    out = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)
    ref, up = A.double() @ W.double().t(), A.double() @ W2.double().t()
    near = lambda got, want, ulps=1: bool(((got.double() - want).abs() <= ulps / 128 * want.abs() + want.abs().max() / 2560).all())
    dec.op_linear(0, A, W, None, out)
    assert near(out, ref)
    dec.op_linear(2, A, W, W2, out)
    assert near(out, torch.nn.functional.silu(ref) * up, 2)
    dec.close()


def test_tuning_entry_refuses_what_it_does_not_know():
    """Keys that never tuned anything, and widths and splits that the paired GEMM does not have, are errors, not silent defaults."""
    from paper_2603_05454_b200 import LSPError
    dec = _dec("bf16")
    for key, value in ((40, 1), (45, 1), (99, 0), (41, 32), (41, 100), (41, 288), (46, 4), (46, -1)):
        with pytest.raises(LSPError) as e:
            dec.debug_set(key, value)
        assert e.value.code == -1
    for value in (0, 64, 96, 256):
        dec.debug_set(41, value)
    dec.close()


@pytest.mark.parametrize("ctas", [1, 100, 161, 320])
@pytest.mark.parametrize("op,N", [(0, 4096), (2, 1024)])
def test_linear_bf16_forced_cta_count(ctas, op, N):
    """A forced number of CTAs (key 10), below and above what the scratch has room for with 256-wide tiles (160): the count is
    capped, not refused.  One or two bf16 ulps, as above."""
    dec = _dec("bf16")
    dec.debug_set(10, ctas)
    M, K = 64, 4096
    A = S.normal((M, K), 18, 1, 1.0, torch.bfloat16, DEV)
    W = S.normal((N, K), 18, 2, 0.05, torch.bfloat16, DEV)
    W2 = S.normal((N, K), 18, 3, 0.05, torch.bfloat16, DEV)
    out = torch.empty(M, N, dtype=torch.bfloat16, device=DEV)
    dec.op_linear(op, A, W, W2 if op == 2 else None, out)
    want = A.double() @ W.double().t()
    if op == 2:
        want = torch.nn.functional.silu(want) * (A.double() @ W2.double().t())
    assert bool(((out.double() - want).abs() <= (2 if op == 2 else 1) / 128 * want.abs() + want.abs().max() / 2560).all())
    dec.close()


@pytest.mark.parametrize("ks", [0, 2, 3])
@pytest.mark.parametrize("M,N,K", [(187, 4096, 12288), (129, 512, 2048), (257, 272, 3072), (256, 3584, 4032), (700, 1040, 4096)])
def test_linear_bf16_k_slices_on_pairs(M, N, K, ks):
    """K slices of a 256-row tile on clusters of two or three pairs: ragged last column tiles and K chunks, a chunk count that
    the slices do not divide, rows of one CTA of the pair only; against the fp64 product, and twice the same bits."""
    dec = _dec("bf16")
    dec.debug_set(46, ks)
    A = S.normal((M, K), 17, 1, 1.0, torch.bfloat16, DEV)
    W = S.normal((N, K), 17, 2, 0.05, torch.bfloat16, DEV)
    X0 = S.normal((M, N), 17, 4, 1.0, torch.bfloat16, DEV)
    ref = A.double() @ W.double().t()
    near = lambda got, want: bool(((got.double() - want).abs() <= want.abs() / 128 + want.abs().max() / 2560).all())
    x, y = X0.clone(), X0.clone()
    dec.op_linear(1, A, W, None, x)
    dec.op_linear(1, A, W, None, y)
    assert near(x, X0.double() + ref) and torch.equal(x, y)
    out = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device=DEV)
    dec.op_linear(0, A, W, None, out[:M])
    assert near(out[:M], ref) and bool((out[M] == 7.0).all())
    dec.close()


@pytest.mark.parametrize("M", [257, 320, 384, 385, 1032])
@pytest.mark.parametrize("N,K,bn", [(272, 192, 0), (1040, 4032, 64), (4096, 576, 128), (1536, 512, 192), (3584, 4096, 256), (1024, 512, 224)])
def test_linear_bf16_half_row_group_on_pairs(M, N, K, bn):
    """A last row group of at most 128 rows (the fourth row count and the last width are beyond the line) on 128-row MMAs: ragged
    last column tiles and K chunks, rows of one CTA of the pair only; against the fp64 product."""
    dec = _dec("bf16")
    dec.debug_set(46, 1)
    dec.debug_set(41, bn)
    A = S.normal((M, K), 19, 1, 1.0, torch.bfloat16, DEV)
    W = S.normal((N, K), 19, 2, 0.05, torch.bfloat16, DEV)
    W2 = S.normal((N, K), 19, 3, 0.05, torch.bfloat16, DEV)
    X0 = S.normal((M, N), 19, 4, 1.0, torch.bfloat16, DEV)
    ref, up = A.double() @ W.double().t(), A.double() @ W2.double().t()
    for op, want, ulps in ((0, ref, 1), (1, X0.double() + ref, 1), (2, torch.nn.functional.silu(ref) * up, 2)):
        out = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device=DEV)
        out[:M] = X0
        dec.op_linear(op, A, W, W2 if op == 2 else None, out[:M])
        # one bf16 rounding per stored value (two ulps with the 2-ulp division) and the fp32 sums' absolute error
        assert bool(((out[:M].double() - want).abs() <= ulps / 128 * want.abs() + want.abs().max() / 2560).all())
        assert bool((out[M] == 7.0).all())
    dec.close()
