"""On-the-fly applies with and without the leg workspace (needs a GB300)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2202_09703_gb300 import synth as S
from tests.helpers import many_layer_scene, ragged_scene, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2202_09703_gb300 import build as B  # noqa: E402

B.build()
from paper_2202_09703_gb300 import mbir as M  # noqa: E402

DEV = torch.device("cuda:0")


def _irregular(n_tx, n_rx, w, h, n_layers):
    """Transmitters at positions of no common step: every (position, column) has its own |x_c - u|."""
    s = S.small_scene(n_layers=n_layers, w=w, h=h, n_tx=n_tx, n_rx=n_rx, M=200, name="tiny_irregular")
    u = S.SplitMix64(5).integers(0, 10 ** 6, n_tx) * 1e-6
    return s.copy(tx_x=np.sort(w * s.pitch * u), rx_offset=s.rx_offset * 1.0371)


# Side by side: positions on the pixel grid (few distinct |x_c - u|, both signs), none shared but within 64 MB of
# legs, one pixel column and one row, two to eight layers, and (the last two) more legs than the workspace holds,
# which the applies solve pair by pair.
SCENES = [
    (ragged_scene, True),
    (lambda: many_layer_scene(8), True),
    (lambda: _irregular(5, 3, 1, 33, 2), True),
    (lambda: _irregular(4, 4, 37, 1, 3), True),
    (lambda: _irregular(12, 6, 48, 40, 4), True),
    (lambda: _irregular(96, 7, 96, 72, 2), False),
    (lambda: _irregular(96, 7, 96, 72, 4), False),
]


@pytest.mark.parametrize("precision,bound", [("fp32", 1e-5), ("bf16", 1e-2)])
@pytest.mark.parametrize("scene_fn,fits", SCENES)
def test_otf_applies(scene_fn, fits, precision, bound):
    """A x and A^T r of the on-the-fly form against the FP64 oracle, twice, the second time on other inputs (the
    workspace is solved again)."""
    s = scene_fn().copy(precision=precision)
    geo = M.Geometry(s, mode="otf")
    legs = 16 * s.img_h * s.img_w * s.n_tx * (s.n_rx + 1)       # with no |x_c - u| shared
    assert fits or legs > (64 << 20)
    plan = O.Plan(s)
    dt = torch.bfloat16 if precision == "bf16" else torch.float32
    for seed in (61, 62):
        x = S.random_vector(s.N, seed).astype(np.float32)
        r = torch.as_tensor(S.random_vector(s.K * s.M, seed + 10), dtype=dt, device=DEV)
        y, b = torch.empty(s.K * s.M, dtype=dt, device=DEV), torch.empty(s.N, device=DEV)
        geo.forward(torch.as_tensor(x, device=DEV), y)
        geo.backproject(r, b)
        torch.cuda.synchronize()
        want = plan.forward(x.astype(np.float64))
        assert np.linalg.norm(want) > 0
        assert rel_l2(y.float().cpu().numpy(), want) <= bound
        assert rel_l2(b.cpu().numpy(), plan.backproject(r.float().cpu().numpy().astype(np.float64))) <= bound
