"""Batches whose first cell-size class leaves no room for helper warps: the small
classes beside it, one to twelve cells an SM, of every model, against the
oracle, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1806_10889_gb300 import workloads as W
from paper_1806_10889_gb300.batching import Batch
from paper_1806_10889_gb300.workloads import TissueSpec
from tests._util import orc_desc, orc_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1806_10889_gb300.tissue import Tissue  # noqa: E402

SMS = torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("model", ["plain", "binding", "promoter"])
def test_small_classes_beside_a_full_chip_match_the_oracle(model):
    def small(w, h, n, tissue_id):
        if model == "promoter":
            rates = W.promoter_model(n)
            rates["kd"] = 3.0
            return TissueSpec(w, h, n, seed=61, tissue_id=tissue_id, init_lambda=(0.6, 0.4, 0.0),
                              model=rates)
        spec = TissueSpec(w, h, n, seed=61, tissue_id=tissue_id)
        return spec.with_model(k_in=0.02, k_off=0.7) if model == "binding" else spec

    # 32 lanes (1 to 4 cells an SM) and 16 lanes (up to 12) of cells in every tree depth
    specs = [TissueSpec(10, SMS, 32, seed=61, tissue_id=0), small(2, SMS, 31, 1), small(3, SMS, 16, 2),
             small(7, SMS, 15, 3), small(1, 5, 8, 4), small(10, SMS, 7, 5)]
    members = [Tissue(s) for s in specs]
    refs = [O.init_counts(orc_desc(s)) for s in specs]
    b = Batch(members)
    dt = 0.004
    for k in range(2):
        b.step(dt, 1)
        b.sync()
        for g, s, ref in zip(members, specs, refs):
            ne, tl = O.step(orc_desc(s), orc_model(s), ref, k, 1, dt)
            assert np.array_equal(g.read_counts(), ref), (s, k)
            gne, gtl = g.read_stats()
            assert np.array_equal(gne, ne), (s, k)
            assert np.array_equal(gtl.view(np.uint64), tl.view(np.uint64)), (s, k)
    b.close()
    for g in members:
        g.close()
