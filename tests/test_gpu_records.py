"""Record order of the tensor-core A^T at the edges of its pixel bitmap (needs a GB300)."""
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


def _scene(w, h, pitch, samples):
    s = S.small_scene(n_layers=3, w=w, h=h, n_tx=2, n_rx=3, M=samples, name="tiny_records")
    return s.copy(pitch=pitch, tx_x=S.centred_positions(2, 2e-3, w * pitch / 2))


# pixel counts on both sides of a 128-pixel group of the bitmap, one row or column of pixels, and the largest
# image the tensor-core records take (2^20 pixels; its pixels reach few tiles, many of them in one)
@pytest.mark.parametrize("w,h,pitch,samples", [(1, 127, 0.2e-3, 300), (129, 1, 0.2e-3, 260), (16, 8, 0.5e-3, 128),
                                               (43, 3, 0.4e-3, 131), (64, 2, 0.3e-3, 150),
                                               (1024, 1024, 0.02e-3, 700)])
@pytest.mark.parametrize("precision,cc_bound,bound", [("fp32", 1e-6, 1e-5), ("bf16", 1e-3, 1e-2)])
def test_adjoint_in_pixel_order(w, h, pitch, samples, precision, cc_bound, bound):
    """A^T from the pixel-ordered records against the CUDA-core A^T (same pairs, FP32 sums in another order;
    the BF16 form's packed weights are rounded to 2^-12) and, on the small images, the FP64 oracle."""
    s = _scene(w, h, pitch, samples).copy(precision=precision)
    tc, cc = M.Geometry(s, mode="tab"), M.Geometry(s, mode="tab", tensor_cores=False)
    if not tc.info.adjoint_tensor_cores:
        pytest.skip("a tile of this scene reaches more attenuation planes than the tensor-core A^T holds")
    r = S.random_vector(s.K * s.M, 51)
    dt = torch.bfloat16 if precision == "bf16" else torch.float32
    rd = torch.as_tensor(r, dtype=dt, device=DEV)
    b_tc, b_cc = torch.empty(s.N, device=DEV), torch.empty(s.N, device=DEV)
    tc.backproject(rd, b_tc)
    cc.backproject(rd, b_cc)
    torch.cuda.synchronize()
    a, b = b_tc.cpu().numpy(), b_cc.cpu().numpy()
    assert np.linalg.norm(b) > 0
    assert rel_l2(a, b) <= cc_bound
    if s.N <= 4096:
        assert rel_l2(a, O.Plan(s).backproject(rd.float().cpu().numpy().astype(np.float64))) <= bound
