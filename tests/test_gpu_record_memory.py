"""Device memory of the two packed record lists of the tensor-core applies (needs a GB300)."""
import pytest

from paper_2202_09703_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2202_09703_gb300 import build as B  # noqa: E402

B.build()
from paper_2202_09703_gb300 import mbir as M  # noqa: E402

DEV = torch.device("cuda:0")


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
