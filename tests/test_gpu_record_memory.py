"""Device memory of the two packed record lists of the tensor-core applies (needs a GB300)."""
import pytest

from oracle import oracle as O
from paper_2202_09703_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2202_09703_gb300 import build as B  # noqa: E402

B.build()
from paper_2202_09703_gb300 import mbir as M  # noqa: E402

DEV = torch.device("cuda:0")


def test_no_second_list_for_a_cuda_core_adjoint():
    """A tile of the BF16 form that reaches more than 256 table columns keeps A x on the tensor cores and A^T off
    them: the geometry then holds one packed list (12 B per pair) where the CUDA-core forms hold 24 B."""
    s = S.small_scene(n_layers=3, w=64, h=64, n_tx=32, n_rx=16, M=512, name="tiny_planes").copy(precision="bf16")
    s = s.copy(gamma_max=O.Geometry(s).gamma_max() / 16)
    tc, cc = M.Geometry(s, mode="tab"), M.Geometry(s, mode="tab", tensor_cores=False)
    n = tc.info.n_records
    assert tc.info.forward_tensor_cores and not tc.info.adjoint_tensor_cores
    assert n == cc.info.n_records and n > 400000
    assert cc.info.device_bytes - tc.info.device_bytes > 6 * n


@pytest.mark.parametrize("precision,per_pair", [("fp32", 51), ("bf16", 49)])
def test_record_lists_fit_in_the_admitted_memory(precision, per_pair):
    """Records are admitted where the sorted list (24 B per pair) takes at most half the free memory; the packed lists
    of both applies are then built within that memory."""
    s = S.cfg1().copy(precision=precision)
    n = M.Geometry(s).info.n_records
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info(DEV)
    left = per_pair * n + (64 << 20)           # and the run bounds, tables and tuning buffers
    ballast = torch.empty(free - left, dtype=torch.uint8, device=DEV)
    info = M.Geometry(s).info
    del ballast
    torch.cuda.empty_cache()
    assert info.n_records == n
    assert info.forward_tensor_cores and info.adjoint_tensor_cores
