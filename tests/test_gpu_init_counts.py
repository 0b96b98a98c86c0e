"""Initial counts on the GPU against the oracle's, exactly: laws whose table of
sums is one entry, a few, hundreds, and ends at its last one."""
import numpy as np
import pytest

import oracle as O
from paper_1806_10889_gb300.workloads import TissueSpec
from tests._util import orc_desc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1806_10889_gb300.tissue import Tissue  # noqa: E402


@pytest.mark.parametrize("lam", [(0.0, 1e-9, 0.1), (5.0, 5.0, 5.0), (60.0, 30.0, 10.0),
                                 (300.0, 700.0, 690.5)])
@pytest.mark.parametrize("w,h,n", [(1, 1, 2), (5, 3, 7), (40, 30, 16)])
def test_initial_counts_match_oracle(w, h, n, lam):
    spec = TissueSpec(w, h, n, seed=17, tissue_id=5, init_lambda=lam)
    g = Tissue(spec)
    assert np.array_equal(g.read_counts(), O.init_counts(orc_desc(spec)))
    g.close()
