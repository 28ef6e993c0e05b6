"""The attention kernels at the points where their fast forms could go wrong: rounding of the forward's
probabilities, extreme softmax scales, odd head ratios, grouped tile orders."""
import numpy as np
import pytest
import torch

from tests.harness import J
from workloads import WORKLOADS, BlockShape

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2609_34866_gb300 import build
    build.build()
    J().jab_get_device_status()


def _blockwise(qkv, shape, threshold):
    """Causal attention of [T, D] fp16 projections over key blocks of 128 in float64, with the forward's one
    rounding that is seen: P to fp16 relative to a running row maximum (log2 units) that moves to the
    block's when it is exceeded by more than `threshold`; the row sums take P unrounded."""
    T, (hq, hkv, dh) = qkv.shape[0], (shape.n_q_heads, shape.n_kv_heads, shape.head_dim)
    y = qkv.double().reshape(T, -1, dh).transpose(0, 1)
    q, k, v = y[:hq], y[hq:hq + hkv].repeat_interleave(hq // hkv, 0), y[hq + hkv:].repeat_interleave(hq // hkv, 0)
    sl2 = float(np.float32(np.float32(1 / np.sqrt(dh)) * np.float32(1.4426950408889634)))
    m = torch.full((hq, T, 1), -torch.inf, dtype=torch.float64, device=qkv.device)
    den = torch.zeros_like(m)
    out = torch.zeros((hq, T, dh), dtype=torch.float64, device=qkv.device)
    for k0 in range(0, T, 128):
        s = q @ k[:, k0:k0 + 128].transpose(1, 2)
        hidden = torch.arange(k0, min(k0 + 128, T), device=s.device)[None, :] > torch.arange(T, device=s.device)[:, None]
        s.masked_fill_(hidden, -torch.inf)
        top = (s.amax(2, keepdim=True).float() * sl2).double()  # (float, as the kernel forms it)
        moved = torch.maximum(m, top)
        new = torch.where(moved > m + threshold, moved, m)
        p = torch.where(hidden, 0.0, torch.exp2(s * sl2 - new))
        old = torch.where(new > m, torch.exp2(m - new), 1.0)
        den = den * old + p.sum(2, keepdim=True)
        out = out * old + p.half().double() @ v[:, k0:k0 + 128]
        m = new
    return (out / den).transpose(0, 1).reshape(T, hq * dh)


@pytest.mark.parametrize("shape", [BlockShape(256, 4, 1, 64, False), BlockShape(256, 3, 1, 128, False)])
def test_forward_rounds_p_at_a_maximum_moved_beyond_two_to_the_eight(shape):
    """Later key blocks have larger scores, so that row maxima grow by 2^8 .. 2^12 from one block to the
    next. The output is that of P rounded to fp16 relative to a maximum that has moved, not one that has
    stayed: in rows where the two differ they are independent roundings of 2^-11, while the fp32 scores
    and exponentials (about 1e-5 relative here) turn a few roundings in a hundred."""
    from dataclasses import replace
    from tests.harness import Case
    T = 384
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=shape), 2, T, 64)
    c.X.mul_(torch.tensor([1.0, 2.0, 3.0], device="cuda").repeat_interleave(128)[None, :, None])
    c.W.mul_(3.0)
    A, _, _ = c.gpu_teacher()
    qkv = torch.empty((c.B, T, c.D), dtype=torch.float16, device="cuda")
    J().jab_reference_projection(c.desc, c.B, T, c.X, c.W, qkv, c.workspace())
    assert J().jab_get_device_status() == 0
    eight, twelve = (torch.stack([_blockwise(qkv[b], shape, th) for b in range(c.B)]) for th in (8.0, 12.0))
    differ = (eight != twelve).reshape(c.B, T, c.Hq, -1).any(-1, keepdim=True)
    assert differ.float().mean() > 0.02, differ.float().mean()

    def distance(e):
        return ((A.double() - e).reshape(c.B, T, c.Hq, -1) * differ).norm().item()

    assert distance(eight) < 0.5 * distance(twelve), (distance(eight), distance(twelve))


@pytest.mark.parametrize("scale", [1e-6, 1e-9, 1e-30, 1e-37])
@pytest.mark.parametrize("T", [5, 200])
def test_kl_rows_vanish_with_the_softmax_scale(scale, T):
    """With a softmax scale near 0 both maps are uniform over the visible keys: the KL of a row is of the
    size of the squared score differences, 1e-11 at most here, and the difference form rounds to 1e-7 of
    its terms. Hidden keys keep no weight, however small the scale that multiplies their score."""
    from dataclasses import replace
    from tests.harness import KL_ROW_ATOL, Case
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=BlockShape(256, 4, 1, 64, True, 500.0)), 2, T, 64)
    c.desc.softmax_scale = scale
    ws = c.workspace(with_bwd=False)
    A, _, _ = c.gpu_teacher(ws)
    qkv = torch.empty((c.B, T, c.D), dtype=torch.float16, device="cuda")
    rows = torch.empty((1, c.B, c.Hq, T), dtype=torch.float32, device="cuda")
    loss, kl = (torch.empty(1, dtype=torch.float64, device="cuda") for _ in range(2))
    J().jab_reference_projection(c.desc, c.B, T, c.X, c.W, qkv, ws)
    J().jab_loss_forward_kl(c.desc, c.B, T, c.X, c.W, A, qkv, [3], [c.gpu_scales(3)], 0.1, loss, ws, kl=kl,
                            kl_rows=rows)
    assert J().jab_get_device_status() == 0
    assert rows.abs().max().item() <= KL_ROW_ATOL, rows.abs().max()
    np.testing.assert_allclose(kl.item(), rows.double().sum().item() / c.B, rtol=1e-6, atol=1e-12)
    v = qkv[..., -c.dh:].double()  # (one KV head) the uniform map's output: the mean of the visible values
    mean = (v.cumsum(1) / torch.arange(1, T + 1, device="cuda")[:, None]).repeat(1, 1, c.Hq)
    assert (A.double() - mean).abs().max() <= 2e-3 * mean.abs().max()


@pytest.mark.parametrize("shape,B,T,bits", [(BlockShape(768, 6, 2, 128, True, 1e4), 2, 171, 3),
                                            (BlockShape(384, 6, 2, 64, False), 1, 300, 2)])
def test_three_query_heads_per_kv_head(shape, B, T, bits):
    """An odd head ratio above 1 at both head sizes (tiles of 128 rows of one head): the teacher's output,
    the candidates' losses, the KL maps, the Hessian products and the gradients with and without the KL term
    against the oracle, with the bars of the other head ratios."""
    from dataclasses import replace
    from tests import test_gpu_parity as P
    from tests.harness import Case
    name = f"ratio3_dh{shape.head_dim}_T{T}"
    P._cases[name] = Case(replace(WORKLOADS["gpt2_smoke"], shape=shape), B, T, 64)
    try:
        P.test_teacher_output_parity(name)
        P.test_loss_forward_parity(name)
        P.test_kl_forward_parity(name)
        P.test_hutchinson_trace_parity(name)
        P.test_backward_parity(name, bits)
        P.test_weight_gradient_and_fisher_coupling_score(name, bits)
        for regime in ("default", "balanced"):
            P.test_backward_kl_parity(name, bits, regime)
    finally:
        del P._cases[name]


@pytest.mark.parametrize("shape", [BlockShape(256, 4, 1, 64, True, 500.0), BlockShape(256, 3, 1, 128, False)])
def test_row_sum_of_do_and_o_is_a_tree(shape):
    """D = rowsum(dO * O) of the backward, as the call leaves it in its workspace slot: every fp32 rounding in
    its place (column groups of four, the chunks of 32 columns in order, then a tree over the eight groups).
    The student's weights are multiples of 2^-6, which bf16 holds, so that a teacher pass on them returns O
    itself. (The products' sums are rounded by way of float64 here: equal but for double roundings.)"""
    from dataclasses import replace
    from tests.harness import Case
    B, T, dh = 2, 333, shape.head_dim
    c = Case(replace(WORKLOADS["gpt2_smoke"], shape=shape), B, T, 64)
    ws = c.workspace()
    A, _, _ = c.gpu_teacher(ws)
    s = torch.full((c.D, shape.d_model // 64), 2.0 ** -6, device="cuda")
    w_hat = (torch.clamp(torch.round(c.W.float() * 64), -3, 3) / 64).to(torch.bfloat16)
    O = torch.empty_like(A)
    J().jab_reference_forward(c.desc, B, T, c.X, w_hat, O, ws)
    loss = torch.empty(1, dtype=torch.float64, device="cuda")
    J().jab_loss_backward_scales(c.desc, B, T, c.X, c.W, A, 3, s, 1.0, loss, torch.empty_like(s), ws)
    assert J().jab_get_device_status() == 0
    N, tp, at = B * T, (T + 127) // 128 * 128, 0  # the slots before D's, in the order of csrc/workspace.h
    for n in (64, N * shape.d_model * 2, c.D * shape.d_model * 2, N * c.D * 2, T * dh * 4, B * c.Hq * ((T + 63) // 64) * 8,
              16, 1024 * 8, N * c.Hq * dh * 2, B * c.Hq * tp * 4):
        at += (n + 255) // 256 * 256
    d = ws.buf[at:at + B * c.Hq * tp * 4].view(torch.float32).view(B, c.Hq, tp)[..., :T]
    o = O.view(B, T, c.Hq, dh // 32, 8, 4).cpu()
    f = (O - A).half().float().view(o.shape).cpu()
    low = f[..., :2] * o[..., :2]
    pairs = (f[..., 2:].double() * o[..., 2:].double() + low.double()).float()
    groups = pairs[..., 0] + pairs[..., 1]
    t = groups[..., 0, :]
    for ch in range(1, dh // 32):
        t = t + groups[..., ch, :]
    while t.shape[-1] > 1:
        t = t[..., 0::2] + t[..., 1::2]
    same = t[..., 0].permute(0, 2, 1) == d.cpu()
    assert same.float().mean() >= 0.999, same.float().mean()
