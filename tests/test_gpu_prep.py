"""The weight-side and preparation kernels at the sizes and values where their fast forms could go
wrong, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import jab_oracle as O
from tests.harness import J, np64
from workloads import BlockShape

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_34866_gb300 import build
    build.build()
    J().jab_get_device_status()


def _weights(d, kind, seed=3):
    """[256, d] weights (a 2-head block of 64): normal, on the grid of some trial scale, heavy-tailed
    with all-zero groups, or with a scale outside the fp32 window of the search."""
    g = torch.Generator().manual_seed(seed)
    w = torch.randn((256, d), generator=g)
    if kind == "grid":  # exact multiples: several trials share codes, one has error 0
        w = torch.round(w * 2).clamp(-3, 3) * 0.25
    elif kind == "tails":
        w = w / torch.rand((256, d), generator=g).clamp_min(1e-3)
        w[::5] = 0
    elif kind == "tiny":
        w = w * 1e-33
    return w.to(torch.bfloat16)


# The fp32 stage only discards trials that its bound rules out, so the chosen scale is the fp64
# search's: its criterion equals the oracle's minimum to fp64 summation order, G 2^-53 at most.
@pytest.mark.parametrize("bits", [2, 3, 8])
@pytest.mark.parametrize("kind", ["normal", "grid", "tails", "tiny"])
@pytest.mark.parametrize("d,G", [(64, 64), (384, 192), (1024, 1024)])
def test_minmse_scales_are_the_fp64_choice(d, G, kind, bits):
    w = _weights(d, kind)
    desc = J().desc_from_shape(BlockShape(d, 2, 1, 64, False), G)
    s = torch.empty((256, d // G), dtype=torch.float32, device="cuda")
    J().jab_init_scales(desc, bits, 1, w.cuda(), s)
    w64, s = np64(w), s.cpu().numpy()
    so = O.init_scales_minmse(w64, bits, G)

    def crit(sc):
        _, wh, _ = O.quantize(w64, sc, bits, G)
        return ((wh - w64) ** 2).reshape(256, -1, G).sum(axis=2)

    assert (s > 0).all()
    assert np.all(crit(s) <= crit(so) * (1 + 4 * G * 2.0 ** -53))


@pytest.mark.parametrize("bits", [2, 8])
@pytest.mark.parametrize("kind", ["normal", "grid", "tiny"])
def test_omega_error_sum_in_pairs(kind, bits):
    """Omega's squared error from unevaluated float pairs equals the fp64 sum: 2^-46 per term, and the
    fp64 additions of 4096-term threads at most 4096 2^-53 of the (positive) total."""
    d, G = 512, 64
    w = _weights(d, kind)
    desc = J().desc_from_shape(BlockShape(d, 2, 1, 64, False), G)
    s = torch.from_numpy(O.init_scales_absmax(np64(w), bits, G) * np.float32(0.93)).cuda()
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    c1 = torch.empty(1, dtype=torch.float64, device="cuda")
    J().jab_omega_scores(desc, w.cuda(), [bits], [s], one, 1, c1, J().Workspace(desc, 1, 1, 1, False))
    want, _ = O.omega_scores(1.0, np64(w), s.cpu().numpy(), bits, G, layers_after=1)
    np.testing.assert_allclose(c1.item(), want, rtol=2.0 ** -46 + 4096 * 2.0 ** -53)
    assert J().jab_get_device_status() == 0


@pytest.mark.parametrize("bits", [2, 3, 8])
@pytest.mark.parametrize("w_mul,s_mul", [(1.0, 1.0), (1e-25, 1e-25), (1e30, 1e30), (1e-30, 1.0)])
def test_codes_bit_exact_in_and_out_of_the_quotient_window(w_mul, s_mul, bits):
    """The corrected-reciprocal quotient inside its window, the division outside it, and chunks that mix
    zeros and both: the codes of the fp32 quotient, ties included (weights on half steps)."""
    d, G = 256, 64
    g = torch.Generator().manual_seed(5)
    s = (torch.rand((256, d // G), generator=g) + 0.5).numpy().astype(np.float32)
    s[::2] = 0.25                                      # exact ties below
    w = torch.randint(-9, 10, (256, d), generator=g).float() * 0.125
    w[:, ::7] = torch.randn((256, (d + 6) // 7), generator=g)
    w = (w * w_mul).to(torch.bfloat16)
    s = (s * np.float32(s_mul)).astype(np.float32)
    desc = J().desc_from_shape(BlockShape(d, 2, 1, 64, False), G)
    codes = torch.empty(w.shape, dtype=torch.int8, device="cuda")
    w_hat = torch.empty(w.shape, dtype=torch.float32, device="cuda")
    J().jab_quantize(desc, bits, w.cuda(), torch.from_numpy(s).cuda(), codes=codes, w_hat=w_hat)
    oc, ow, _ = O.quantize(np64(w), s, bits, G)
    np.testing.assert_array_equal(codes.cpu().numpy(), oc)
    np.testing.assert_array_equal(w_hat.cpu().numpy(), ow.astype(np.float32))
    assert J().jab_get_device_status() == 0


@pytest.mark.parametrize("shape,T", [(BlockShape(256, 4, 1, 64, True, 500.0), 65),
                                     (BlockShape(512, 4, 2, 128, True, 1e4), 33)])
def test_ten_candidates_in_one_call_equal_single_calls(shape, T):
    """More candidates than one preparation launch takes (8): each loss has the bits of a call of its
    own, with an odd number of rows for the last run of the RoPE table."""
    from dataclasses import replace
    from tests.harness import Case
    from workloads import WORKLOADS
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=shape), 2, T, 64)
    bits = [2, 3, 4, 5, 8, 2, 3, 4, 5, 8]
    scales = [c.gpu_scales(b) * f for b, f in zip(bits, [1.0] * 5 + [0.7] * 5)]
    ws = c.workspace(n_cand=10, with_bwd=False)
    A, _, _ = c.gpu_teacher(ws)
    loss = torch.empty(10, dtype=torch.float64, device="cuda")
    J().jab_loss_forward(c.desc, c.B, c.T, c.X, c.W, A, bits, scales, loss, ws)
    one = torch.empty(1, dtype=torch.float64, device="cuda")
    for i in range(10):
        J().jab_loss_forward(c.desc, c.B, c.T, c.X, c.W, A, bits[i:i + 1], scales[i:i + 1], one, ws)
        assert one.item() == loss[i].item(), i
    assert J().jab_get_device_status() == 0


def test_scale_gradient_where_the_quotient_takes_the_division():
    """Chunks with zero weights and groups of tiny ones (quotients outside the corrected reciprocal's
    window): the LSQ factor of the weight-gradient epilogue against the oracle's."""
    from dataclasses import replace
    from tests.harness import COS_MIN, Case, cosine
    from workloads import WORKLOADS
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=BlockShape(256, 4, 1, 64, True, 500.0)), 2, 65, 64)
    g = torch.Generator().manual_seed(2)
    w = c.W.float().cpu()
    w[torch.rand(w.shape, generator=g) < 0.02] = 0
    w[:, 64:128] *= 1e-25
    w = w.to(torch.bfloat16)
    s = (torch.rand((c.D, 4), generator=g) * 0.02 + 0.01).numpy()
    W, S = w.cuda(), torch.from_numpy(s).cuda()
    ws = c.workspace()
    A = torch.empty((c.B, c.T, c.Hq * c.dh), dtype=torch.float32, device="cuda")
    J().jab_reference_forward(c.desc, c.B, c.T, c.X, W, A, ws)
    loss = torch.empty(1, dtype=torch.float64, device="cuda")
    grad = torch.empty_like(S)
    J().jab_loss_backward_scales(c.desc, c.B, c.T, c.X, W, A, 3, S, 1.0, loss, grad, ws)
    r = O.jab_loss_and_grad(c.x64, np64(w), s, 3, c.odesc, kappa=1.0)
    assert cosine(grad.cpu().numpy(), r["grad_s"]) >= COS_MIN
    assert J().jab_get_device_status() == 0


@pytest.mark.parametrize("B,T", [(3, 65), (1, 257), (2, 1)])
def test_weight_gradient_norm_and_loss_parts_of_odd_batches(B, T):
    """||dW||^2 from float pairs against the fp64 sum of the returned dW (2^-46 per term, 256-thread fp64
    sums), alone and beside dW, and the loss as the fixed-order sum of its (sequence, head) parts over
    numbers of partials that are no power of two."""
    from dataclasses import replace
    from tests.harness import Case
    from workloads import WORKLOADS
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=BlockShape(256, 4, 1, 64, True, 500.0)), B, T, 64)
    ws = c.workspace()
    A, _, _ = c.gpu_teacher(ws)
    s = c.gpu_scales(2)
    loss, sq, sq2 = (torch.empty(1, dtype=torch.float64, device="cuda") for _ in range(3))
    dw = torch.empty((c.D, 256), dtype=torch.float32, device="cuda")
    J().jab_set_deterministic(True)
    try:
        J().jab_loss_backward_weights(c.desc, B, T, c.X, c.W, A, 2, s, loss, grad_w=dw, grad_sqnorm=sq, ws=ws)
        J().jab_loss_backward_weights(c.desc, B, T, c.X, c.W, A, 2, s, loss, grad_sqnorm=sq2, ws=ws)
    finally:
        J().jab_set_deterministic(False)
    np.testing.assert_allclose(sq.item(), (dw.double() ** 2).sum().item(), rtol=1e-12)
    assert sq.item() == sq2.item()
    parts = torch.empty((1, B, 4), dtype=torch.float64, device="cuda")
    J().jab_loss_forward(c.desc, B, T, c.X, c.W, A, [2], [s], loss, ws, sse_parts=parts)
    np.testing.assert_allclose(loss.item(), parts.sum().item() / (B * T * 4 * 64), rtol=1e-13)
    assert J().jab_get_device_status() == 0


@pytest.mark.parametrize("shape,B,T", [(BlockShape(768, 12, 12, 64, False), 1, 70),
                                       (BlockShape(768, 12, 12, 64, False), 1, 1337),
                                       (BlockShape(512, 4, 2, 128, True, 1e4), 3, 43),
                                       (BlockShape(512, 20, 2, 128, True, 1e4), 4, 301),
                                       (BlockShape(256, 3, 1, 128, True, 1e4), 2, 65),
                                       (BlockShape(256, 3, 1, 128, True, 1e4), 16, 395),
                                       (BlockShape(256, 4, 1, 64, True, 500.0), 2, 65)])
def test_projection_with_narrow_and_wide_tiles(shape, B, T):
    """[Q | K | V] with RoPE from 128- and 256-column tiles (few tiles, or most of a round of CTA pairs),
    ragged in rows and in the last column tile. Against float64 on the fp16 operands: half an ulp of the
    fp16 result, and for the fp32 sums of K products K 2^-24 of the sum of their magnitudes, of both
    halves of a rotated pair."""
    from dataclasses import replace
    from tests.harness import Case
    from workloads import WORKLOADS
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=shape), B, T, 64)
    out = torch.empty((B, T, c.D), dtype=torch.float16, device="cuda")
    J().jab_reference_projection(c.desc, B, T, c.X, c.W, out, c.workspace())
    assert J().jab_get_device_status() == 0
    x, w = np64(c.X.half()), np64(c.W.half())
    ref, mag = x @ w.T, np.abs(x) @ np.abs(w).T
    if shape.use_rope:
        cos, sin = O.rope_tables(T, c.dh, shape.rope_theta)
        nr = (c.Hq + shape.n_kv_heads) * c.dh
        rot = ref[..., :nr].reshape(B, T, -1, c.dh)
        ref[..., :nr] = O.apply_rope(rot, cos, sin).reshape(B, T, nr)
        m = mag[..., :nr].reshape(B, T, -1, 2, c.dh // 2).sum(3, keepdims=True)
        mag[..., :nr] = np.broadcast_to(m, (B, T, m.shape[2], 2, c.dh // 2)).reshape(B, T, nr)
    # (the rotation's own roundings and the tables': four more of 2^-24)
    bound = 2.0 ** -11 * np.abs(ref) + (shape.d_model + 4) * 2.0 ** -24 * mag + 2.0 ** -25
    err = np.abs(np64(out) - ref)
    assert (err <= bound).all(), (err / bound).max()


@pytest.mark.parametrize("shape,B,T", [(BlockShape(256, 4, 1, 64, True, 500.0), 96, 128),
                                       (BlockShape(256, 4, 1, 64, True, 500.0), 96, 333),
                                       (BlockShape(512, 4, 2, 128, True, 1e4), 96, 128),
                                       (BlockShape(512, 4, 2, 128, True, 1e4), 96, 333),
                                       (BlockShape(256, 4, 1, 64, True, 500.0), 320, 333),
                                       (BlockShape(256, 6, 2, 128, True, 1e4), 216, 333)])
def test_persistent_maps_equal_single_sequences(shape, B, T):
    """KL maps and Hessian products of a batch with several tiles per persistent CTA (of several lengths
    where T > 128; in the last two cases with more than 24 tiles per SM, so that tiles go by KV head and not
    by length, the last with three query heads per KV head): every KL row has the bits of a call with that sequence alone, and the
    probes' v^T H v, sums of per-sequence values over n, agree to the fp64 sums' 2^-52 a term."""
    from dataclasses import replace
    from tests.harness import Case
    from workloads import WORKLOADS
    bits = [2, 4]
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=shape), B, T, 64)

    def run(X):
        n = X.shape[0]
        ws = J().Workspace(c.desc, n, T, 2, True)
        A = torch.empty((n, T, c.Hq * c.dh), dtype=torch.float32, device="cuda")
        lse = torch.empty((n, c.Hq, T), dtype=torch.float32, device="cuda")
        qkv = torch.empty((n, T, c.D), dtype=torch.float16, device="cuda")
        rows = torch.empty((2, n, c.Hq, T), dtype=torch.float32, device="cuda")
        loss, kl = (torch.empty(2, dtype=torch.float64, device="cuda") for _ in range(2))
        vhv, trace = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (2, 1))
        J().jab_reference_forward(c.desc, n, T, X, c.W, A, ws, lse=lse)
        J().jab_reference_projection(c.desc, n, T, X, c.W, qkv, ws)
        J().jab_loss_forward_kl(c.desc, n, T, X, c.W, A, qkv, bits, [c.gpu_scales(b) for b in bits], 0.1,
                                loss, ws, kl=kl, kl_rows=rows)
        J().jab_hutchinson_trace(c.desc, n, T, X, c.W, A, lse, 2, 7, trace, ws, vhv=vhv)
        assert J().jab_get_device_status() == 0
        return rows, vhv

    rows, vhv = run(c.X)
    ones = [run(c.X[b:b + 1].contiguous()) for b in range(B)]
    assert torch.equal(rows, torch.cat([r for r, _ in ones], 1))
    np.testing.assert_allclose(vhv.cpu(), torch.stack([v for _, v in ones]).mean(0).cpu(), rtol=1e-12)


@pytest.mark.parametrize("d,G", [(768, 192), (960, 320), (768, 384), (1024, 512), (1280, 640), (768, 768), (768, 256)])
@pytest.mark.parametrize("T", [65, 2600])
def test_scale_gradient_of_groups_over_several_tiles(d, G, T):
    """Groups that begin and end inside 256-column tiles or span several, with one K range and with
    several (2600 tokens): the scale gradient against sums over each group of dL/dW times the LSQ factor,
    dW from the weight-gradient call. The factors are exact fp32 and the sums over G products in fp32 differ
    in order only: (G + 1) 2^-23 of the sum of magnitudes, and the splits' atomic order in dW as much again."""
    from dataclasses import replace
    from tests.harness import Case
    from workloads import WORKLOADS
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=BlockShape(d, 4, 1, 64, True, 500.0)), 1, T, G)
    ws = c.workspace()
    A, _, _ = c.gpu_teacher(ws)
    s = c.gpu_scales(3)
    loss = torch.empty(1, dtype=torch.float64, device="cuda")
    grad, dw = torch.empty_like(s), torch.empty((c.D, d), dtype=torch.float32, device="cuda")
    J().jab_loss_backward_scales(c.desc, 1, T, c.X, c.W, A, 3, s, 1.0, loss, grad, ws)
    again = torch.empty_like(grad)
    J().jab_loss_backward_scales(c.desc, 1, T, c.X, c.W, A, 3, s, 1.0, loss, again, ws)
    J().jab_loss_backward_weights(c.desc, 1, T, c.X, c.W, A, 3, s, loss, grad_w=dw, ws=ws)
    assert J().jab_get_device_status() == 0
    assert torch.equal(grad, again)
    q = (c.W.float().view(c.D, -1, G) / s[:, :, None]).double()
    r = torch.where(q.abs() <= 3, torch.round(q) - q, torch.sign(q) * 3)
    terms = r * dw.double().view(c.D, -1, G)
    bound = 2 * (G + 1) * 2.0 ** -23 * terms.abs().sum(2)
    err = (terms.sum(2) - grad.double()).abs()
    assert bool((err <= bound).all()), (err / bound).max().item()


def test_omega_scores_keep_the_prepared_x():
    """jab_prepare_x, jab_omega_scores and the prepared fit on one workspace: Omega's partials lie behind
    the converted X, and the fit has the plain call's bits. Where the workspace given to Omega is too small
    for that, the prepared call is refused."""
    from dataclasses import replace
    from tests.harness import Case
    from workloads import WORKLOADS
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=BlockShape(256, 4, 1, 64, True, 500.0)), 8, 256, 64)
    ws = c.workspace(n_cand=2)
    A, _, _ = c.gpu_teacher(ws)
    s = c.gpu_scales(3)
    bits, scales = [3, 4], [s, c.gpu_scales(4)]
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    want, got = torch.empty(2, dtype=torch.float64, device="cuda"), torch.empty(2, dtype=torch.float64, device="cuda")
    J().jab_omega_scores(c.desc, c.W, bits, scales, one, 1, want, J().Workspace(c.desc, 1, 1, 2, False))
    l0, l1 = (torch.empty(1, dtype=torch.float64, device="cuda") for _ in range(2))
    g0, g1 = torch.empty_like(s), torch.empty_like(s)
    J().jab_loss_backward_scales(c.desc, c.B, c.T, c.X, c.W, A, 3, s, 0.0, l0, g0, ws)
    J().jab_prepare_x(c.desc, c.B, c.T, c.X, ws)
    J().jab_omega_scores(c.desc, c.W, bits, scales, one, 1, got, ws)
    J().jab_loss_backward_scales_prepared(c.desc, c.B, c.T, c.X, c.W, A, 3, s, 0.0, l1, g1, ws)
    assert l0.item() == l1.item() and torch.equal(g0, g1) and torch.equal(want, got)
    small = J().Workspace(c.desc, 1, 1, 2, False)
    small.buf = ws.buf                                 # the same memory, fewer bytes of it
    assert small.nbytes < c.B * c.T * 256 * 2
    J().jab_prepare_x(c.desc, c.B, c.T, c.X, ws)
    J().jab_omega_scores(c.desc, c.W, bits, scales, one, 1, got, small)
    with pytest.raises(J().JabError) as e:
        J().jab_loss_backward_scales_prepared(c.desc, c.B, c.T, c.X, c.W, A, 3, s, 0.0, l1, g1, ws)
    assert e.value.status == 1 and torch.equal(want, got)
    assert J().jab_get_device_status() == 0


@pytest.mark.parametrize("bits", [2, 8])
@pytest.mark.parametrize("s_mul", [1.0, 1e-25])
def test_w_hat_of_small_negative_weights_is_negative_zero(bits, s_mul):
    """A weight below half a step has the code 0, and fl32(0 s) the weight's sign as rint gives it, by the
    corrected reciprocal (scale 1) and by the division (scale 1e-25) alike."""
    d, G = 128, 64
    g = torch.Generator().manual_seed(7)
    w = torch.randn((256, d), generator=g) * 0.5
    w[:, ::5] *= 0.0                                   # +0 and -0
    w = (w * s_mul).to(torch.bfloat16)
    s = np.full((256, d // G), s_mul, dtype=np.float32)
    desc = J().desc_from_shape(BlockShape(d, 2, 1, 64, False), G)
    w_hat = torch.empty(w.shape, dtype=torch.float32, device="cuda")
    J().jab_quantize(desc, bits, w.cuda(), torch.from_numpy(s).cuda(), w_hat=w_hat)
    _, ow, _ = O.quantize(np64(w), s, bits, G)
    want = ow.astype(np.float32)
    assert (np.signbit(want) & (want == 0)).any()
    np.testing.assert_array_equal(w_hat.cpu().numpy().view(np.uint32), want.view(np.uint32))
    assert J().jab_get_device_status() == 0


def test_weight_gradient_norm_is_not_biased():
    """||dW||^2 against the exact sum of the returned dW's squares (fp32 squares are exact in fp64): eight
    batches' errors are independent roundings of about 2^-53 in the last additions, so that their mean is
    below 2^-52; low parts that are dropped would all fall on one side."""
    import math
    from dataclasses import replace
    from tests.harness import Case
    from workloads import WORKLOADS
    errors = []
    for seed in range(8):
        wl = replace(WORKLOADS["gpt2_smoke"], shape=BlockShape(256, 4, 1, 64, True, 500.0), seed=seed)
        c = Case(wl, 2, 65, 64)
        ws = c.workspace()
        A, _, _ = c.gpu_teacher(ws)
        loss, sq = (torch.empty(1, dtype=torch.float64, device="cuda") for _ in range(2))
        dw = torch.empty((c.D, 256), dtype=torch.float32, device="cuda")
        J().jab_loss_backward_weights(c.desc, 2, 65, c.X, c.W, A, 2, c.gpu_scales(2), loss, grad_w=dw, grad_sqnorm=sq,
                                      ws=ws)
        exact = math.fsum((np64(dw).ravel() ** 2).tolist())
        errors.append(sq.item() / exact - 1)
    assert J().jab_get_device_status() == 0
    assert abs(np.mean(errors)) <= 2.0 ** -52, errors
