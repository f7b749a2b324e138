"""A x and A^T r where rows lie on layer interfaces, where tiles of samples stay empty between others, and where a
tile reaches too many attenuation planes for the tiled kernels (needs a GB300)."""
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


def _on_interface(pitch, z0, water, first_angle):
    """A slow layer over a fast one with the centres of one row exactly on the interface: that row's delay is the
    direct path through the slow layer, later (past the critical angle) than the refracted one of the rows below."""
    fc = 2e6
    w = 64
    s = S.Scene(name="interface_row", layers=[S.material_layer("water", water, fc), S.material_layer("steel", 50e-3, fc)],
                img_w=w, img_h=64, pitch=pitch, x0=0.0, z0=z0, tx_x=S.centred_positions(4, 3e-3, w * pitch / 2),
                rx_offset=S.centred_positions(3, 5e-3), fs=20e6, n_samples=1024, fc=fc, apod_first_angle=first_angle)
    assert (z0 + (np.arange(64) + 0.5) * pitch == water).any()
    return s


def _sparse_rows():
    """Rows about two tiles of 128 samples apart: most tiles, and the first of most chunks of tiles, hold no pair."""
    s = S.small_scene(n_layers=1, w=3, h=6, n_tx=2, n_rx=2, M=4000, name="tiny_sparse_rows")
    return s.copy(pitch=40e-3, tx_x=np.array([60e-3, 62e-3]))


def _all_planes():
    """Every attenuation plane within one tile."""
    s = S.small_scene(n_layers=3, w=17, h=30, n_tx=2, n_rx=3, M=128, name="tiny_all_planes")
    return s.copy(gamma_max=O.Geometry(s).gamma_max() / 8)


SCENES = [lambda: _on_interface(1e-3, 0.0, 10.5e-3, False), lambda: _on_interface(1e-3, 0.0, 10.5e-3, True),
          lambda: _on_interface(0.5e-3, 0.25e-3, 20e-3, True), _sparse_rows, _all_planes]


@pytest.mark.parametrize("precision,bound", [("fp32", 1e-5), ("bf16", 1e-2)])
@pytest.mark.parametrize("mode", ["otf", "norec", "tab"])
@pytest.mark.parametrize("scene_fn", SCENES)
def test_applies(scene_fn, mode, precision, bound):
    s = scene_fn().copy(precision=precision)
    geo = M.Geometry(s, mode="tab", records=False) if mode == "norec" else M.Geometry(s, mode=mode)
    plan = O.Plan(s)
    dt = torch.bfloat16 if precision == "bf16" else torch.float32
    x = S.random_vector(s.N, 91).astype(np.float32)
    r = torch.as_tensor(S.random_vector(s.K * s.M, 92), dtype=dt, device=DEV)
    y, b = torch.empty(s.K * s.M, dtype=dt, device=DEV), torch.empty(s.N, device=DEV)
    geo.forward(torch.as_tensor(x, device=DEV), y)
    geo.backproject(r, b)
    torch.cuda.synchronize()
    want = plan.forward(x.astype(np.float64))
    assert np.linalg.norm(want) > 0
    assert rel_l2(y.float().cpu().numpy(), want) <= bound
    assert rel_l2(b.cpu().numpy(), plan.backproject(r.float().cpu().numpy().astype(np.float64))) <= bound


def _grazing(pitch):
    """Rows a few micrometres apart below an interface into a faster layer, seen from far to the side: a pair's delay
    grows by less per row than its rounding error.  The delay of the first row below the interface is a multiple of
    128 samples in the middle column, and the 64 receivers 20 nm apart sample the delays around it in steps of 7e-5, so
    that pairs out of order meet a tile's bound."""
    fc, water, w = 2e6, 10e-3, 128

    def scene(dist):
        return S.Scene(name="grazing", layers=[S.material_layer("water", water, fc), S.material_layer("steel", 50e-3, fc)],
                       img_w=w, img_h=64, pitch=pitch, x0=0.0, z0=water - 4 * pitch, tx_x=np.array([-dist]),
                       rx_offset=20e-9 * np.arange(64), fs=20e6, n_samples=1000, fc=fc, apod_first_angle=True)

    lo, hi = 60e-3, 80e-3
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        s = scene(mid)
        if 2 * O.Geometry(s).leg(mid + 0.5 * w * pitch, water + 0.5 * pitch)[0] * s.fs < 768.0:
            lo = mid
        else:
            hi = mid
    return scene(lo)


@pytest.mark.parametrize("pitch", [1e-6, 2e-6, 5e-6, 1e-5])
@pytest.mark.parametrize("mode", ["otf", "norec"])
def test_grazing_rows(mode, pitch):
    """Every pair is taken: the applies without stored records against those of the sorted record list, which makes no
    use of an order (the same pairs, FP32 sums in another order)."""
    s = _grazing(pitch)
    geo = M.Geometry(s, mode="tab", records=False) if mode == "norec" else M.Geometry(s, mode=mode)
    ref = M.Geometry(s, mode="tab", tensor_cores=False)
    assert ref.info.n_records > 0
    x = torch.as_tensor(S.random_vector(s.N, 93), dtype=torch.float32, device=DEV)
    r = torch.as_tensor(S.random_vector(s.K * s.M, 94), dtype=torch.float32, device=DEV)
    out = []
    for g in (geo, ref):
        y, b = torch.empty(s.K * s.M, device=DEV), torch.empty(s.N, device=DEV)
        g.forward(x, y)
        g.backproject(r, b)
        torch.cuda.synchronize()
        out.append((y.cpu().numpy(), b.cpu().numpy()))
    (y, b), (y_ref, b_ref) = out
    assert np.linalg.norm(y_ref) > 0 and np.linalg.norm(b_ref) > 0
    assert rel_l2(y, y_ref) <= 1e-5
    assert rel_l2(b, b_ref) <= 1e-5
