"""Steps of no to a dozen events a cell, on small cells in every form the sum-tree
kernel runs them in, where a batch is cut to the events likely left.  Against
the oracle, bit for bit."""
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


def _spec(per_sm, n, model, tissue_id=1):
    kw = {}
    if model == "promoter":
        kw = dict(model=dict(W.promoter_model(n), kd=3.0), init_lambda=(0.6, 0.4, 0.0))
    spec = TissueSpec(per_sm, SMS - 3, n, seed=43, tissue_id=tissue_id, **kw)
    return spec.with_model(k_in=0.02, k_off=0.7) if model == "binding" else spec


def _same(g, spec, ref, k, dt):
    ne, tl = O.step(orc_desc(spec), orc_model(spec), ref, k, 1, dt)
    assert np.array_equal(g.read_counts(), ref), (spec, dt, k)
    gne, gtl = g.read_stats()
    assert np.array_equal(gne, ne) and np.array_equal(gtl.view(np.uint64), tl.view(np.uint64))


# lanes per cell 32, 16, 8 (with a helper and without), 4 and 1 (with one and without)
@pytest.mark.parametrize("model", ["plain", "binding", "promoter"])
@pytest.mark.parametrize("per_sm,n", [(2, 3), (8, 4), (24, 2), (28, 5), (45, 7), (90, 3), (150, 2),
                                      (150, 5), (200, 8), (330, 4), (700, 2)])
def test_short_steps_of_small_cells_match_the_oracle(per_sm, n, model):
    spec = _spec(per_sm, n, model)
    rate = 60.0 * n * n  # events a cell and unit of time, at most
    ref = O.init_counts(orc_desc(spec))
    g = Tissue(spec)
    for k, events in enumerate((0.01, 2.0, 12.0)):
        dt = events / rate
        g.step(dt, 1)
        _same(g, spec, ref, k, dt)
    g.close()


def test_members_of_a_batch_share_a_warp():
    """Cells of many small tissues in one class: a warp's lanes hold cells of
    different tissues, with counts past the packed range and without."""
    specs = [TissueSpec(17, 13 + i, 3, seed=43, tissue_id=i).with_model(kD=5.0 + i) for i in range(100)]
    members = [Tissue(s) for s in specs]
    refs = []
    for g, s in zip(members, specs):
        x = O.init_counts(orc_desc(s)).reshape(s.cells, 3, s.V)
        x[s.tissue_id % s.cells, 0, 1] = 70000
        x[(7 * s.tissue_id) % s.cells, 2, 0] = 5000
        x[3, 1, 2] = 200000 if s.tissue_id % 9 == 0 else 4
        refs.append(np.ascontiguousarray(x.ravel()))
        g.write_counts(refs[-1], 0)
    b = Batch(members)
    assert len(b.classes()) == 1 and b.chi_info(0)["lanes_per_cell"] == 1
    for k, dt in enumerate((1e-6, 0.002)):
        b.step(dt, 1)
        b.sync()
        for g, s, x in zip(members, specs, refs):
            _same(g, s, x, k, dt)
    b.close()
    for g in members:
        g.close()
