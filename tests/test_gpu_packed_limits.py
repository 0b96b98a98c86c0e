"""Cells with packed counts past the tissue's common limits: counts whose voxel
totals are a fraction of 2^52 (fast hops), and bound or free receptors near the
end of the Hill table.  Such a cell goes on with limits of its own, or, where
there are none, is run again by the 32-bit pass; in every packed form the
results are the oracle's, bit for bit."""
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

from paper_1806_10889_gb300 import tissue as T  # noqa: E402
from paper_1806_10889_gb300.tissue import Tissue  # noqa: E402

SMS = torch.cuda.get_device_properties(0).multi_processor_count
# (cells per SM, n): planes at 16 (three forms), 8 and 4 lanes; records at 16, 8, 4
# and 1; sectors at 1 (V = 81 and 289)
PACKED = [(9, 31), (15, 26), (20, 26), (45, 16), (90, 16), (110, 8), (30, 32), (45, 32), (120, 16), (140, 8),
          (140, 9), (112, 17)]


def _tissue(per_sm, n, **kw):
    h = max(2, int((per_sm * SMS) ** 0.5))
    return TissueSpec(per_sm * SMS // h, h, n, seed=97, tissue_id=n, **kw)


def _same(spec, x, dt, steps=2):
    d, m = orc_desc(spec), orc_model(spec)
    ref = np.ascontiguousarray(x.ravel())
    g = Tissue(spec)
    g.write_counts(ref, 0)
    for k in range(steps):
        ne, tl = O.step(d, m, ref, k, 1, dt)
        g.step(dt, 1)
        got = g.read_counts()
        assert np.array_equal(got, ref), f"cell {np.flatnonzero(got != ref)[0] // (3 * spec.V)}"
        gne, gtl = g.read_stats()
        assert np.array_equal(gne, ne) and np.array_equal(gtl.view(np.uint64), tl.view(np.uint64))
    g.close()
    return ref


@pytest.mark.parametrize("model", ["plain", "binding", "promoter"])
@pytest.mark.parametrize("per_sm,n", PACKED)
def test_cells_past_the_common_limit_match_the_oracle(per_sm, n, model):
    # hops at 1000: totals reach 2^52 at 262 molecules of one species; the common
    # limit is 64 (promoter: 128)
    if model == "promoter":
        spec = _tissue(per_sm, n, model=dict(W.promoter_model(n), hop=1000.0, kd=3.0),
                       init_lambda=(0.6, 0.4, 0.0))
    else:
        spec = _tissue(per_sm, n).with_model(hopD=1000.0, hopN=1000.0, hopR=1000.0)
        if model == "binding":
            spec = spec.with_model(k_in=0.02, k_off=0.7)
    x = O.init_counts(orc_desc(spec)).reshape(spec.cells, 3, spec.V)
    x[0::8, 0] = 110            # past the limit from the start
    x[1::8, 0] = 124            # ... and meets its own
    x[2::8, 0] = 63             # passes the limit within the step
    x[3::8, 1] = 126            # nothing left above it: run again
    x[4::8, 0, :2] = 200        # run again from the start
    x[5::8, 1, -2:] = 100
    _same(spec, x, 200.0 / (4000.0 * 80.0 * spec.V))


@pytest.mark.parametrize("model", ["plain", "binding"])
@pytest.mark.parametrize("per_sm,n", PACKED)
def test_receptors_up_to_the_end_of_the_hill_table_match_the_oracle(per_sm, n, model):
    spec = _tissue(per_sm, n)
    if model == "binding":
        spec = spec.with_model(k_in=0.02, k_off=0.7)
    x = O.init_counts(orc_desc(spec)).reshape(spec.cells, 3, spec.V)
    x[0::16, 2, 3] = 2047
    x[1::16, 2, :] = 2500
    x[2::16, 2, :4] = 4093      # passes the table within the step
    x[3::16, 2, -2:] = 4094
    x[4, 2, 1] = 4095
    x[5, 2, 1] = 4096
    x[6, 2, 0] = 9000
    _same(spec, x, 150.0 / (4.0 * 2500.0 * spec.V))


@pytest.mark.parametrize("per_sm,n", [(45, 16), (120, 16), (140, 9)])
def test_a_total_past_its_limit_is_reported(per_sm, n):
    spec = _tissue(per_sm, n).with_model(hopD=1000.0, hopN=1000.0, hopR=1000.0)
    x = O.init_counts(orc_desc(spec)).reshape(spec.cells, 3, spec.V)
    x[7, 0] = 261
    x[7, 1:] = 0                # a hop takes a neighbour to 262 and more
    with pytest.raises(O.OracleError):
        O.step(orc_desc(spec), orc_model(spec), x.ravel().copy(), 0, 1, 2e-6)
    g = Tissue(spec)
    g.write_counts(x.ravel(), 0)
    g.step(2e-6, 1)
    with pytest.raises(T.TissueError) as e:
        g.read_counts()
    assert e.value.code == T.E_OVERFLOW
    g.close()


def test_packed_classes_of_a_batch_share_the_redo_list():
    """Three classes with packed counts (sectors, planes, records) in one batch, some
    cells of each past their range from the start and within the step."""
    specs = [_tissue(112, 17), _tissue(45, 16), TissueSpec(140, SMS, 8, seed=97, tissue_id=1),
             TissueSpec(3, 2, 16, seed=97, tissue_id=2)]
    dt = 0.004
    states = []
    for s in specs:
        x = O.init_counts(orc_desc(s)).reshape(s.cells, 3, s.V)
        x[0, 0, 0] = 70000
        x[1, 2, 1] = 5000
        x[2, 1, :2] = 65533
        x[3, 2, :3] = 4094
        x[4, 0, 0] = 200000
        states.append(np.ascontiguousarray(x.ravel()))
    members = [Tissue(s) for s in specs]
    for g, x in zip(members, states):
        g.write_counts(x, 0)
    b = Batch(members)
    assert [b.chi_info(i)["launches"] for i in range(3)] == [2, 2, 2]
    for k in range(2):
        b.step(dt, 1)
        b.sync()
        for g, s, x in zip(members, specs, states):
            ne, tl = O.step(orc_desc(s), orc_model(s), x, k, 1, dt)
            assert np.array_equal(g.read_counts(), x), (s, k)
            gne, gtl = g.read_stats()
            assert np.array_equal(gne, ne) and np.array_equal(gtl.view(np.uint64), tl.view(np.uint64))
    b.close()
    for g in members:
        g.close()
