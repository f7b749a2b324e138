"""A x and A^T r from the leg table without stored records, at the edges of their tiles and chunks (needs a GB300)."""
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


def _forward(geo, x):
    s = geo.scene
    dt = torch.bfloat16 if geo.precision == "bf16" else torch.float32
    y = torch.empty(s.K * s.M, dtype=dt, device=DEV)
    geo.forward(torch.as_tensor(np.asarray(x, dtype=np.float32), device=DEV), y)
    torch.cuda.synchronize()
    return y.float().cpu().numpy().astype(np.float64).reshape(s.K, s.M)


# records of one tile, one sample more and less, chunks of four tiles with and without a last one cut short, more
# (column, layer) cursors than threads, one attenuation plane, no distinct transmitters
@pytest.mark.parametrize("precision,bound", [("fp32", 1e-5), ("bf16", 1e-2)])
@pytest.mark.parametrize("mode", ["otf", "norec"])
@pytest.mark.parametrize("w,h,layers,n_tx,n_rx,samples,atten", [
    (17, 30, 2, 2, 3, 127, True), (17, 30, 2, 2, 3, 128, True), (17, 30, 2, 2, 3, 129, True),
    (24, 97, 3, 1, 1, 512, True), (24, 97, 3, 1, 2, 641, True), (24, 160, 3, 2, 2, 1280, False),
    (1100, 3, 1, 1, 2, 300, True), (400, 30, 4, 1, 2, 260, True)])
def test_forward_from_legs(w, h, layers, n_tx, n_rx, samples, atten, mode, precision, bound):
    s = S.small_scene(n_layers=layers, w=w, h=h, n_tx=n_tx, n_rx=n_rx, M=samples, atten=atten,
                      name="tiny_legs").copy(precision=precision)
    if samples > 400:
        s = s.copy(pitch=2e-3, tx_x=s.tx_x + 0.75e-3 * w)
    geo = M.Geometry(s, mode="otf") if mode == "otf" else M.Geometry(s, mode="tab", records=False)
    plan = O.Plan(s)
    for scale, seed in ((1.0, 71), (3e-30, 72), (0.0, 73)):
        x = (scale * S.random_vector(s.N, seed)).astype(np.float32)
        y, want = _forward(geo, x), plan.forward(x.astype(np.float64)).reshape(s.K, s.M)
        if scale == 0.0:
            assert not y.any()
        else:
            assert np.linalg.norm(want) > 0
            assert rel_l2(y, want) <= bound
            assert np.array_equal(y, _forward(geo, x))


def _backproject(geo, r):
    dt = torch.bfloat16 if geo.precision == "bf16" else torch.float32
    rd, b = torch.as_tensor(np.asarray(r), dtype=dt, device=DEV), torch.empty(geo.scene.N, device=DEV)
    geo.backproject(rd, b)
    torch.cuda.synchronize()
    return b.cpu().numpy().astype(np.float64), rd.float().cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("precision,bound", [("fp32", 1e-5), ("bf16", 1e-2)])
@pytest.mark.parametrize("mode", ["otf", "norec"])
@pytest.mark.parametrize("w,h,layers,n_tx,n_rx,samples,atten", [
    (17, 30, 2, 2, 3, 127, True), (17, 30, 2, 2, 3, 128, True), (17, 30, 2, 2, 3, 129, True),
    (24, 97, 3, 1, 2, 641, True), (24, 160, 3, 2, 2, 1280, False), (1100, 3, 1, 1, 2, 300, True),
    (400, 30, 4, 1, 2, 260, True)])
def test_adjoint_from_legs(w, h, layers, n_tx, n_rx, samples, atten, mode, precision, bound):
    s = S.small_scene(n_layers=layers, w=w, h=h, n_tx=n_tx, n_rx=n_rx, M=samples, atten=atten,
                      name="tiny_legs").copy(precision=precision)
    if samples > 400:
        s = s.copy(pitch=2e-3, tx_x=s.tx_x + 0.75e-3 * w)
    geo = M.Geometry(s, mode="otf") if mode == "otf" else M.Geometry(s, mode="tab", records=False)
    plan = O.Plan(s)
    for scale, seed in ((1.0, 81), (3e-30, 82), (0.0, 83)):
        b, r = _backproject(geo, scale * S.random_vector(s.K * s.M, seed))
        want = plan.backproject(r)
        if scale == 0.0:
            assert not b.any()
        else:
            assert np.linalg.norm(want) > 0
            assert rel_l2(b, want) <= bound
            assert np.array_equal(b, _backproject(geo, r)[0])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_adjoint_from_legs_non_finite(bad):
    """A sample that is not finite spoils the pixels whose pulses reach it (or end within four taps of it), and no
    other."""
    s = S.small_scene(n_layers=3, w=24, h=40, n_tx=2, n_rx=2, M=400, name="tiny_legs")
    geo, plan = M.Geometry(s, mode="otf"), O.Plan(s)
    r = S.random_vector(s.K * s.M, 84)
    at = 2 * s.M + 150
    one = np.zeros(s.K * s.M)
    near = np.zeros(s.N, bool)
    for d in range(5):
        one[:] = 0.0
        one[at - d] = 1.0
        near |= plan.backproject(one) != 0.0
        if d == 0:
            reach = near.copy()
    r[at] = 0.0
    rest, _ = _backproject(geo, r)
    r[at] = bad
    b, _ = _backproject(geo, r)
    assert reach.any() and not near.all()
    assert not np.isfinite(b[reach]).any()
    # the other pixels: the same sums (their scale does not depend on the sample)
    assert np.array_equal(b[~near], rest[~near])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_forward_from_legs_non_finite(bad):
    """A pixel that is not finite spoils the samples its pulses reach, and no other."""
    s = S.small_scene(n_layers=3, w=24, h=40, n_tx=2, n_rx=2, M=400, name="tiny_legs")
    geo = M.Geometry(s, mode="otf")
    x = S.random_vector(s.N, 74).astype(np.float32)
    v = 20 * s.img_w + 11
    x[v] = 0.0
    rest = _forward(geo, x)
    one = np.zeros(s.N)
    one[v] = 1.0
    reach = O.Plan(s).forward(one).reshape(s.K, s.M) != 0.0
    x[v] = bad
    y = _forward(geo, x)
    assert reach.any()
    assert not np.isfinite(y[reach]).any()
    tw = geo.info.pulse_support
    for k in range(s.K):
        n = np.flatnonzero(reach[k])
        if n.size == 0:
            assert np.array_equal(y[k], rest[k])
            continue
        outside = np.ones(s.M, bool)
        outside[max(n[-1] - tw, 0):n[0] + tw + 1] = False
        assert np.array_equal(y[k][outside], rest[k][outside])
