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
