"""Relative accuracy of the applies without stored records where the weights, or the image, are small beside the
largest of the geometry or the call (needs a GB300).

The FP32 form's bound (relative L2 of 1e-5) is asked of the weak part by itself."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2202_09703_gb300 import synth as S
from tests.helpers import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2202_09703_gb300 import build as B  # noqa: E402

B.build()
from paper_2202_09703_gb300 import mbir as M  # noqa: E402

DEV = torch.device("cuda:0")


def _wide():
    """Transducers at one end of a wide, shallow image: the far columns' weights fall to about 1e-16."""
    s = S.small_scene(n_layers=1, w=300, h=24, n_tx=2, n_rx=2, M=2048, name="tiny_wide")
    return s.copy(tx_x=np.array([2e-3, 4e-3]))


def _geo(s, mode):
    return M.Geometry(s, mode="otf") if mode == "otf" else M.Geometry(s, mode="tab", records=False)


def _forward(geo, x):
    y = torch.empty(geo.scene.K * geo.scene.M, device=DEV)
    geo.forward(torch.as_tensor(x, device=DEV), y)
    torch.cuda.synchronize()
    return y.cpu().numpy().reshape(geo.scene.K, geo.scene.M)


@pytest.mark.parametrize("mode", ["otf", "norec"])
def test_forward_of_far_columns(mode):
    s = _wide()
    x = S.random_vector(s.N, 101).astype(np.float32).reshape(s.img_h, s.img_w)
    x[:, :260] = 0.0
    x = x.reshape(-1)
    y, want = _forward(_geo(s, mode), x), O.Plan(s).forward(x.astype(np.float64)).reshape(s.K, s.M)
    assert 0.0 < np.abs(want).max() < 1e-12
    for k in range(s.K):
        assert rel_l2(y[k], want[k]) <= 1e-5


@pytest.mark.parametrize("mode", ["otf", "norec"])
def test_forward_beside_an_outlier(mode):
    """One pixel 1e15 times the others: the samples that its pulses do not reach (nor share a tile with) are those of
    the other pixels."""
    s = S.small_scene(n_layers=3, w=24, h=90, n_tx=2, n_rx=2, M=800, name="tiny_outlier")
    x = S.random_vector(s.N, 102).astype(np.float32)
    plan = O.Plan(s)
    v = 3 * s.img_w + 11
    one = np.zeros(s.N)
    one[v] = 1.0
    reach = plan.forward(one).reshape(s.K, s.M) != 0.0
    last = max(np.flatnonzero(reach[k])[-1] for k in range(s.K))
    n = (last // 128 + 2) * 128
    assert n < s.M - 128
    x[v] = 1e15
    y, want = _forward(_geo(s, mode), x)[:, n:], plan.forward(x.astype(np.float64)).reshape(s.K, s.M)[:, n:]
    assert 0.0 < np.abs(want).max() < 1e3
    assert rel_l2(y, want) <= 1e-5


@pytest.mark.parametrize("mode", ["otf", "norec"])
def test_adjoint_of_far_columns(mode):
    s = _wide()
    r = S.random_vector(s.K * s.M, 103).astype(np.float32)
    b = torch.empty(s.N, device=DEV)
    _geo(s, mode).backproject(torch.as_tensor(r, device=DEV), b)
    torch.cuda.synchronize()
    got = b.cpu().numpy().reshape(s.img_h, s.img_w)
    want = O.Plan(s).backproject(r.astype(np.float64)).reshape(s.img_h, s.img_w)
    for c in (260, 280, 299):
        assert 0.0 < np.abs(want[:, c]).max() < 1e-12
        assert rel_l2(got[:, c], want[:, c]) <= 1e-5


@pytest.mark.parametrize("mode", ["otf", "norec"])
def test_adjoint_beside_an_outlier(mode):
    """One sample 1e12 times the others: the pixels whose pulses do not come near it are those of the other samples."""
    s = S.small_scene(n_layers=3, w=24, h=90, n_tx=2, n_rx=2, M=800, name="tiny_outlier")
    r = S.random_vector(s.K * s.M, 104).astype(np.float32)
    plan = O.Plan(s)
    at = s.M + 100
    near = np.zeros(s.K * s.M)
    near[at - 5:at + 6] = 1.0
    far = plan.backproject(near) == 0.0
    assert 0.25 * s.N < far.sum() < s.N
    r[at] = 1e12
    b = torch.empty(s.N, device=DEV)
    _geo(s, mode).backproject(torch.as_tensor(r, device=DEV), b)
    torch.cuda.synchronize()
    want = plan.backproject(r.astype(np.float64))[far]
    assert 0.0 < np.abs(want).max() < 1e3
    assert rel_l2(b.cpu().numpy()[far], want) <= 1e-5
