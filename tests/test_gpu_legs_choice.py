"""Which kernels an unstored geometry runs, read off its device memory (needs a GB300).

A leg table is H x (distinct |x_c - u|) x 16 B, of TAB mode always and of the on-the-fly form up to 64 MB; the tiled
kernels of that table add 17 B per pixel and more (sums, marks, scales)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2202_09703_gb300 import synth as S
from tests.helpers import many_layer_scene, ragged_scene

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2202_09703_gb300 import build as B  # noqa: E402

B.build()
from paper_2202_09703_gb300 import mbir as M  # noqa: E402


def _leg_bytes(s):
    xc = s.x0 + (np.arange(s.img_w) + 0.5) * s.pitch
    pos = np.unique(np.concatenate([s.tx_x] + [s.tx_x + o for o in s.rx_offset]))
    d = np.sort(np.abs(xc[None, :] - pos[:, None]).reshape(-1))
    return 16 * s.img_h * (1 + int((np.diff(d) > 1e-9 * s.pitch).sum()))


def _irregular(n_tx, n_rx, w, h):
    s = S.small_scene(n_layers=2, w=w, h=h, n_tx=n_tx, n_rx=n_rx, M=200, name="tiny_irregular")
    u = S.SplitMix64(5).integers(0, 10 ** 6, n_tx) * 1e-6
    return s.copy(tx_x=np.sort(w * s.pitch * u), rx_offset=s.rx_offset * 1.0371)


@pytest.mark.parametrize("scene_fn,fits", [(ragged_scene, True), (lambda: many_layer_scene(8), True),
                                           (lambda: _irregular(12, 6, 48, 40), True),
                                           (lambda: _irregular(96, 7, 96, 72), False)])
def test_leg_workspace(scene_fn, fits):
    s = scene_fn()
    legs = _leg_bytes(s)
    assert (legs <= 64 << 20) == fits
    otf, tab = M.Geometry(s, mode="otf").info.device_bytes, M.Geometry(s, mode="tab", records=False).info.device_bytes
    assert tab > legs
    if fits:
        assert otf >= tab                 # the same tables, and the list of offsets
    else:
        assert otf < tab - legs


@pytest.mark.parametrize("mode", ["otf", "norec"])
def test_tiled_kernels_refuse_a_tile_of_too_many_planes(mode):
    """Every attenuation plane in one tile: 272 columns of sums do not fit in shared memory (the same scene with the
    default range of planes is taken)."""
    s = S.small_scene(n_layers=3, w=40, h=60, n_tx=2, n_rx=3, M=128, name="tiny_planes")
    wide = s.copy(gamma_max=O.Geometry(s).gamma_max() / 16)
    make = lambda sc: M.Geometry(sc, mode="otf") if mode == "otf" else M.Geometry(sc, mode="tab", records=False)
    assert make(s).info.device_bytes - make(wide).info.device_bytes >= 17 * s.N
