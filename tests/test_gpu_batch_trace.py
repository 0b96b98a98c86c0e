"""Event logs of batch members: a class whose members are traced logs every
event the oracle fires, whatever its model; the members beside it, of other
cell sizes and not traced, run as always."""
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


def _promoter(n, tissue_id):
    model = W.promoter_model(n)
    model["kd"] = 3.0
    return TissueSpec(4, 3, n, seed=53, tissue_id=tissue_id, init_lambda=(0.6, 0.4, 0.0), model=model)


@pytest.mark.parametrize("specs", [
    [_promoter(8, 1)],                                         # a class of the promoter model only
    [TissueSpec(3, 3, 8, seed=53, tissue_id=2)],               # Notch-Delta only
    [_promoter(8, 3), TissueSpec(3, 3, 8, seed=53, tissue_id=4)],  # both in one class
], ids=["promoter", "notch_delta", "both"])
def test_traced_members_log_every_event(specs):
    dt, steps = 0.1, 3
    other = TissueSpec(3, 2, 16, seed=53, tissue_id=9)
    members = [Tissue(s) for s in specs + [other]]
    for g in members[:-1]:
        g.trace_begin(1 << 20)
    b = Batch(members)
    b.step(dt, steps)
    b.sync()
    for g, s in zip(members, specs + [other]):
        ref = O.init_counts(orc_desc(s))
        want = O.step_traced(orc_desc(s), orc_model(s), ref, 0, steps, dt, trace_cap=1 << 20)
        assert np.array_equal(g.read_counts(), ref)
        if s is other:
            continue
        got = g.trace_read()
        want = np.sort(want, order=["step", "kind", "unit", "e"])
        assert got.size == want.size, (got.size, want.size)
        for f in ("step", "kind", "unit", "e", "site", "channel"):
            assert np.array_equal(got[f], want[f]), f
        assert np.array_equal(got["t"].view(np.uint64), want["t"].view(np.uint64))
    b.close()
    for g in members:
        g.close()
