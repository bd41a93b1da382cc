"""Cache build from the F_pos / F_dir MLPs on the tensor cores, through the C ABI.

Checked against the FP64 oracle's MLP evaluated at the same grid samples:
(i) with the same bf16 weights and bf16 rounding of the network input and of
every hidden activation (as the tensor-core chain stores them), per output
channel: relative L2 error <= 2.5e-3, at least 99% of the values within
1e-2 * rms(channel), and max |error| <= 0.13 * rms(channel). The chain rounds
fp32 accumulators to bf16 where the oracle rounds FP64 ones. The fp32 sum of
256 exact bf16 products differs from the FP64 one by ~1e-6 relative, so about
one activation in 2,000 lies close enough to a bf16 rounding boundary to land
one bf16 ulp (2^-8 relative) apart; F_pos has 2,048 hidden activations per
point, so most points carry a flip or two through the later layers. That sets
the bulk (measured at 1,048,576 points: relative L2 1.3e-3, 99.65% of values
within 1e-2 rms in the worst channel) and the rare large outliers (measured
max 8.7e-2 rms); the bounds above were frozen from that run with headroom.
(ii) against pure FP64 activations: relative L2 <= 5e-2. A single linear layer
(no hidden rounding) is checked tightly (FP32 accumulation only), which pins
the operand layouts. The full-size build (F_pos over 512^3, F_dir over 512^2)
is checked on 1,048,576 random grid points and 65,536 random direction bins."""

import numpy as np
import pytest

import oracle
import scenegen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fnr():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2103_10380_gb300 as fnr
    torch.cuda.set_device(0)
    return fnr


def device_bytes(ptr, nbytes):
    import torch

    class _V:
        __cuda_array_interface__ = {"shape": (nbytes,), "typestr": "|u1", "data": (ptr, False), "version": 3}

    return torch.as_tensor(_V(), device="cuda").cpu().numpy()


def to_device(layers):
    import torch
    return [(torch.from_numpy(W.view(np.int16)).cuda(), torch.from_numpy(b).cuda()) for W, b in layers]


def as_fp64(layers):
    return [(scenegen.bf16_value(W).astype(np.float64), b.astype(np.float64)) for W, b in layers]


def read_cache(fnr, cache, k, D, l, prec=0, dprec=0):
    lay = fnr.fnr_cache_get_layout(cache)
    k3 = k ** 3
    es = 4 if prec == 0 else 2
    sdt = np.float32 if prec == 0 else np.float16
    sig = device_bytes(lay.sigma_dev, k3 * es).view(sdt).astype(np.float64)
    rec = device_bytes(lay.uvw_dev, k3 * lay.record_stride).reshape(k3, lay.record_stride)
    uvw = np.ascontiguousarray(rec[:, :3 * D * es]).view(sdt).astype(np.float64).reshape(k3, 3 * D)
    bes = 4 if dprec == 0 else 2
    bdt = np.float32 if dprec == 0 else np.float16
    beta = device_bytes(lay.beta_dev, l * l * D * bes).view(bdt).astype(np.float64).reshape(l * l, D)
    return sig, uvw, beta


def build(fnr, ctx, k, l, D, pos, dirn, prec=0, dprec=0):
    desc = fnr.make_desc(k, D, l, prec, dprec)
    return fnr.fnr_build_cache_mlp(ctx, desc, to_device(pos), to_device(dirn))


def check_channels(got, ref, l2_rel=2.5e-3, max_rel=0.13, bulk_rel=1e-2, bulk_frac=0.99):
    rms = np.sqrt(np.mean(ref ** 2, axis=0)) + 1e-12
    err = np.abs(got - ref) / rms
    l2 = np.sqrt(np.mean(err ** 2, axis=0))
    mx = np.max(err, axis=0)
    within = np.mean(err <= bulk_rel, axis=0)
    tail = {t: float(np.mean(err <= t, axis=0).min()) for t in (2e-2, 3e-2, 5e-2)}
    print(f"per-channel relative L2 max {l2.max():.2e}, max |err|/rms {mx.max():.2e}, "
          f"fraction within {bulk_rel:g} rms min {within.min():.6f}, within 2e-2/3e-2/5e-2 "
          f"{tail[2e-2]:.6f}/{tail[3e-2]:.6f}/{tail[5e-2]:.6f} ({got.shape[0]} points)")
    assert np.all(l2 <= l2_rel), l2.max()
    assert np.all(within >= bulk_frac), within.min()
    assert np.all(mx <= max_rel), mx.max()
    return {"rel_l2_max": float(l2.max()), "max_abs_over_rms": float(mx.max()),
            "frac_within_bulk_min": float(within.min())}


def test_single_linear_layer(fnr):
    """One linear layer per MLP: only FP32 accumulation separates GPU and FP64."""
    k, l, D = 8, 8, 8
    pos = scenegen.mlp_weights(1, [60, 25], bias_scale=0.5)
    dirn = scenegen.mlp_weights(2, [24, 8], bias_scale=0.5)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        cache = build(fnr, ctx, k, l, D, pos, dirn)
        sig, uvw, beta = read_cache(fnr, cache, k, D, l)
        xyz = oracle.cell_centres(k, np.arange(k ** 3))
        out = oracle.mlp_eval(as_fp64(pos), xyz, 10, True)
        np.testing.assert_allclose(sig, np.maximum(out[:, 0], 0), atol=2e-4)
        np.testing.assert_allclose(uvw, out[:, 1:], atol=2e-4)
        dirs = oracle.bin_directions(l, np.arange(l * l))
        bout = oracle.mlp_eval(as_fp64(dirn), dirs, 4, True)
        np.testing.assert_allclose(beta, bout, atol=2e-4)
    finally:
        fnr.fnr_context_destroy(ctx)


@pytest.mark.parametrize("prec", [0, 1])
def test_full_architecture_small_grid(fnr, prec):
    """8 x 256 ReLU F_pos (+ head) and 4 x 128 ReLU F_dir (+ head), k=16, l=16 (ragged last tile of F_dir)."""
    k, l, D = 16, 12, 8
    pos = scenegen.mlp_weights(3, scenegen.FPOS_DIMS_D8, bias_scale=0.05)
    dirn = scenegen.mlp_weights(4, scenegen.FDIR_DIMS_D8, bias_scale=0.05)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        cache = build(fnr, ctx, k, l, D, pos, dirn, prec, prec)
        sig, uvw, beta = read_cache(fnr, cache, k, D, l, prec, prec)
        xyz = oracle.cell_centres(k, np.arange(k ** 3))
        ref_b = oracle.mlp_eval(as_fp64(pos), xyz, 10, True)
        got = np.concatenate([sig[:, None], uvw], axis=1)
        ref = np.concatenate([np.maximum(ref_b[:, :1], 0), ref_b[:, 1:]], axis=1)
        check_channels(got, ref, 2.5e-3 if prec == 0 else 3e-3)
        ref64 = oracle.mlp_eval(as_fp64(pos), xyz, 10, False)
        rel = np.linalg.norm(uvw - ref64[:, 1:]) / np.linalg.norm(ref64[:, 1:])
        assert rel < 5e-2, rel
        dirs = oracle.bin_directions(l, np.arange(l * l))
        check_channels(beta, oracle.mlp_eval(as_fp64(dirn), dirs, 4, True), 2.5e-3 if prec == 0 else 3e-3)
    finally:
        fnr.fnr_context_destroy(ctx)


def test_cache_build_config_sampled(fnr):
    """F_pos over 512^3 and F_dir over 512^2 (He-uniform, seeds 0 and 100), checked on 1,048,576 random grid
    points (seed 1) and 65,536 random direction bins against the FP64 oracle MLP."""
    import torch
    k, l, D = 512, 512, 8
    pos = scenegen.mlp_weights(0, scenegen.FPOS_DIMS_D8)
    dirn = scenegen.mlp_weights(100, scenegen.FDIR_DIMS_D8)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        cache = build(fnr, ctx, k, l, D, pos, dirn)
        torch.cuda.synchronize()
        rng = np.random.default_rng(1)
        cells = rng.integers(0, k ** 3, 1 << 20)
        lay = fnr.fnr_cache_get_layout(cache)
        sig_all = device_bytes(lay.sigma_dev, k ** 3 * 4).view(np.float32)
        ref = oracle.mlp_eval(as_fp64(pos), oracle.cell_centres(k, cells), 10, True)
        rec = torch.as_tensor(type("V", (), {"__cuda_array_interface__": {
            "shape": (k ** 3, lay.record_stride // 4), "typestr": "<f4", "data": (lay.uvw_dev, False),
            "version": 3}})(), device="cuda")
        uvw = rec[torch.from_numpy(cells).cuda()].cpu().numpy().astype(np.float64)[:, :3 * D]
        got = np.concatenate([sig_all[cells].astype(np.float64)[:, None], uvw], axis=1)
        check_channels(got, np.concatenate([np.maximum(ref[:, :1], 0), ref[:, 1:]], axis=1))
        bins = rng.integers(0, l * l, 65536)
        beta_all = device_bytes(lay.beta_dev, l * l * D * 4).view(np.float32).reshape(l * l, D)
        check_channels(beta_all[bins].astype(np.float64),
                       oracle.mlp_eval(as_fp64(dirn), oracle.bin_directions(l, bins), 4, True))
    finally:
        fnr.fnr_context_destroy(ctx)


def test_render_mlp_built_cache(fnr):
    """A cache built by the MLP kernel renders like the oracle rendering the same cache values."""
    import torch
    k, l, D = 32, 16, 8
    pos = scenegen.mlp_weights(5, scenegen.FPOS_DIMS_D8, bias_scale=0.5)
    dirn = scenegen.mlp_weights(6, scenegen.FDIR_DIMS_D8, bias_scale=0.5)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        cache = build(fnr, ctx, k, l, D, pos, dirn)
        sig, uvw, beta = read_cache(fnr, cache, k, D, l)
        oc = oracle.Cache(k, D, l, sig.astype(np.float32), uvw.astype(np.float32), beta.astype(np.float32))
        cam = scenegen.cameras(9, 1, 48, 40)[0]
        p = fnr.make_params(64)
        rgba = torch.zeros(48 * 40 * 4, device="cuda")
        st = torch.zeros(48 * 40 * 4, device="cuda", dtype=torch.int32)
        fnr.fnr_render(ctx, cache, [cam], p, rgba, st)
        torch.cuda.synchronize()
        ref, rst, _ = oracle.render_image(oc, cam, oracle.params_struct(64))
        assert np.array_equal(st.cpu().numpy().reshape(40, 48, 4), rst)
        assert np.max(np.abs(rgba.cpu().numpy().reshape(40, 48, 4) - ref)) <= 1e-5
    finally:
        fnr.fnr_context_destroy(ctx)


def test_widths_not_multiple_of_64(fnr):
    """Hidden widths of 80 and 48: the K padding of the next layer's input (to 64-column blocks) must read
    as zeros."""
    k, l, D = 8, 8, 8
    pos = scenegen.mlp_weights(5, [60, 80, 48, 25], bias_scale=0.3)
    dirn = scenegen.mlp_weights(6, [24, 40, 8], bias_scale=0.3)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        cache = build(fnr, ctx, k, l, D, pos, dirn)
        sig, uvw, beta = read_cache(fnr, cache, k, D, l)
        xyz = oracle.cell_centres(k, np.arange(k ** 3))
        ref_b = oracle.mlp_eval(as_fp64(pos), xyz, 10, True)
        got = np.concatenate([sig[:, None], uvw], axis=1)
        ref = np.concatenate([np.maximum(ref_b[:, :1], 0), ref_b[:, 1:]], axis=1)
        check_channels(got, ref)
        dirs = oracle.bin_directions(l, np.arange(l * l))
        check_channels(beta, oracle.mlp_eval(as_fp64(dirn), dirs, 4, True))
    finally:
        fnr.fnr_context_destroy(ctx)


def test_encoded_width_above_64_rejected(fnr):
    """The encoded input must fit one 64-column staging chunk: dims[0] = 128 is refused before any launch."""
    pos = scenegen.mlp_weights(5, [128, 32, 25], bias_scale=0.3)
    dirn = scenegen.mlp_weights(6, [24, 16, 8], bias_scale=0.3)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        with pytest.raises(fnr.FnrError) as ei:
            build(fnr, ctx, 8, 8, 8, pos, dirn)
        assert ei.value.status == fnr.FNR_ERR_UNSUPPORTED
    finally:
        fnr.fnr_context_destroy(ctx)


@pytest.mark.parametrize("k,l,pos_dims,dir_dims", [
    (37, 13, scenegen.FPOS_DIMS_D8, scenegen.FDIR_DIMS_D8),   # ragged last tile of 128 and of 256 points
    (64, 64, scenegen.FPOS_DIMS_D8, scenegen.FDIR_DIMS_D8),   # whole tiles, several per CTA pair
    (9, 8, [60, 80, 48, 25], [24, 40, 8]),                    # narrow layers: chunk halves of 40, 24, 16, 8 rows
])
def test_cta_pair_form_bit_identical(fnr, k, l, pos_dims, dir_dims):
    """The CTA-pair form of the build kernel (two SMs per M=256 MMA, each holding half of every weight chunk,
    one load of each layer's weights for both tiles in flight) computes every product in the same order as
    the single-CTA form: the caches are equal byte for byte, and so is an uncached render."""
    import torch
    D = 8
    pos = to_device(scenegen.mlp_weights(7, pos_dims, bias_scale=0.3))
    dirn = to_device(scenegen.mlp_weights(8, dir_dims, bias_scale=0.3))
    desc = fnr.make_desc(k, D, l)
    ctx = fnr.fnr_context_create(0, 0)
    cam = scenegen.cameras(4, 1, 40, 28)[0]
    try:
        outs = []
        for pair in (False, True):
            fnr.fnr_testing_mlp_cta_pair(pair)
            c = fnr.fnr_build_cache_mlp(ctx, desc, pos, dirn)
            lay = fnr.fnr_cache_get_layout(c)
            raw = (device_bytes(lay.sigma_dev, k ** 3 * 4).copy(),
                   device_bytes(lay.uvw_dev, k ** 3 * lay.record_stride).copy(),
                   device_bytes(lay.beta_dev, l * l * D * 4).copy())
            fnr.fnr_cache_free(ctx, c)
            img = torch.zeros(40 * 28 * 4, device="cuda")
            if pos_dims is scenegen.FPOS_DIMS_D8:
                fnr.fnr_render_mlp(ctx, pos, dirn, D, cam, fnr.make_params(24), img)
                torch.cuda.synchronize()
            outs.append(raw + (img.cpu().numpy(),))
        for a, b in zip(*outs):
            assert np.array_equal(a, b)
    finally:
        fnr.fnr_testing_mlp_cta_pair(False)
        fnr.fnr_context_destroy(ctx)


@pytest.mark.parametrize("k,l,D,pos_dims,dir_dims", [
    (37, 300, 8, scenegen.FPOS_DIMS_D8, scenegen.FDIR_DIMS_D8),          # a last pair of one tile; narrow, many rounds
    (30, 150, 16, [60, 256, 49], [60, 16]),                              # two passes of a head; one layer
    (20, 200, 4, [60, 144, 200, 64, 16, 25], [24, 16, 8]),               # halves of 16 and 72 outputs, padded inputs
    (11, 9, 8, [60] + [256] * 15 + [25], [64, 256, 256, 30]),            # the deepest network; outputs not stored
    (70, 20, 2, [24, 128, 129, 128, 7], [24, 32, 2]),                    # widths at a half's edge
])
def test_forms_agree_over_shapes(fnr, k, l, D, pos_dims, dir_dims):
    """The single-CTA form (activations in tensor memory, outputs in halves of 128) against the CTA-pair form
    (activations in shared memory, all outputs at once), both accumulating each output over the inputs in the
    same order: caches equal byte for byte."""
    pos = to_device(scenegen.mlp_weights(17, pos_dims, bias_scale=0.3))
    dirn = to_device(scenegen.mlp_weights(18, dir_dims, bias_scale=0.3))
    pos_freqs, dir_freqs = pos_dims[0] // 6, min(dir_dims[0] // 6, 10)
    ctx = fnr.fnr_context_create(0, 0)
    try:
        for prec in (fnr.FNR_PREC_FP32, fnr.FNR_PREC_FP16):
            outs = []
            for pair in (True, False):
                fnr.fnr_testing_mlp_cta_pair(pair)
                c = fnr.fnr_build_cache_mlp(ctx, fnr.make_desc(k, D, l, prec, prec), pos, dirn, pos_freqs, dir_freqs)
                outs.append(read_cache(fnr, c, k, D, l, prec, prec))
                fnr.fnr_cache_free(ctx, c)
            for a, b in zip(*outs):
                assert np.array_equal(a, b)
    finally:
        fnr.fnr_testing_mlp_cta_pair(False)
        fnr.fnr_context_destroy(ctx)
