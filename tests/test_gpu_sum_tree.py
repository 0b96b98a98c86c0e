"""The sum-tree chi kernel in every form its launch plan picks -- 32 to 1
lanes per cell, leaves in shared memory, in planes, records or sectors --
against the oracle, bit for bit: counts, per-cell event counts and
binary64 times.  The plan follows from the cell size and the cells per SM, so
the tissues here are just wide enough, with cells of ragged sizes.  Some
cells hold counts past what the packed records and the unchecked Hill lookups
take, from the start or from within the step."""
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
BIND = dict(k_in=0.02, k_off=0.7)


def _spec(per_sm, n, model):
    """A tissue of about per_sm cells per SM (never more)."""
    h = max(2, int((per_sm * SMS) ** 0.5))
    w = per_sm * SMS // h
    if model == "promoter":
        rates = W.promoter_model(n)
        rates["kd"] = 3.0
        return TissueSpec(w, h, n, seed=91, tissue_id=n, init_lambda=(0.6, 0.4, 0.0), model=rates)
    spec = TissueSpec(w, h, n, seed=91, tissue_id=n)
    return spec.with_model(**BIND) if model == "binding" else spec


def _plant(x, spec):
    """Counts past the limits that keep a voxel's total below 2^52 unchecked
    (2^16 with these rates) and R within the unchecked Hill lookups (2048) or
    the table (4096), and just below them beside another full voxel, whose
    molecules hop in during the first step."""
    v = spec.V - 1
    x[1, 0, 0] = 70000
    x[2, 2, v] = 2048
    x[3, 2, 0:2] = 2047
    x[4, 2, v - 1:] = 4095
    x[5, 1, 2:4] = 65535


def _compare(g, spec, ref, ne, tl, ctx):
    got = g.read_counts()
    assert np.array_equal(got, ref), f"{ctx}: first cell {np.flatnonzero(got != ref)[0] // (3 * spec.V)}"
    gne, gtl = g.read_stats()
    assert np.array_equal(gne, ne), f"{ctx}: event counts"
    assert np.array_equal(gtl.view(np.uint64), tl.view(np.uint64)), f"{ctx}: event times"


# (cells per SM, n, dt): shared leaves at 32, 16, 8 and 4 lanes; planes at 16, 8
# and 4; records at 16, 8, 4 and 1; sectors at 1 (V = 4 to 1,024)
FORMS = [(1, 2, 0.3), (8, 5, 0.1), (20, 7, 0.1), (100, 5, 0.02), (8, 16, 0.02), (30, 9, 0.02),
         (28, 8, 0.02), (28, 16, 0.01), (40, 9, 0.02), (90, 8, 0.01), (140, 9, 0.01), (50, 17, 0.01),
         (45, 16, 0.01), (98, 9, 0.01), (120, 2, 0.1), (120, 8, 0.01), (120, 9, 0.01),
         (3, 17, 0.02), (9, 18, 0.02), (30, 17, 0.01), (85, 17, 0.005), (112, 17, 0.005),
         (2, 32, 0.01), (16, 32, 0.005), (11, 32, 0.005), (24, 31, 0.005), (60, 15, 0.01),
         (120, 16, 0.004), (30, 32, 0.002)]


@pytest.mark.parametrize("model", ["plain", "binding", "promoter"])
@pytest.mark.parametrize("per_sm,n,dt", FORMS)
def test_every_form_matches_oracle(per_sm, n, dt, model):
    spec = _spec(per_sm, n, model)
    d, m = orc_desc(spec), orc_model(spec)
    ref = O.init_counts(d)
    if model == "plain" and n > 2 and spec.cells > 5:
        _plant(ref.reshape(spec.cells, 3, spec.V), spec)
    g = Tissue(spec)
    g.write_counts(ref, 0)
    for k in range(2):
        ne, tl = O.step(d, m, ref, k, 1, dt)
        g.step(dt, 1)
        _compare(g, spec, ref, ne, tl, f"{spec.width}x{spec.height}x{n} {model} step {k}")
    g.close()


def test_no_scratch_or_a_capture_runs_the_segmented_kernel():
    """A tissue or batch that cannot have the records' scratch gives the same
    results by the other kernel; so does a step captured into a graph."""
    spec = _spec(140, 9, "plain")
    dt = 0.01
    ref = Tissue(spec)
    ref.step(dt, 2)
    want, (wne, wtl) = ref.read_counts(), ref.read_stats()
    ref.close()

    a = Tissue(spec)
    a.sync()
    T.debug_fail_allocs(1)
    try:
        a.step(dt, 1)  # its scratch allocation fails
    finally:
        T.debug_fail_allocs(0)
    a.step(dt, 1)
    _compare(a, spec, want, wne, wtl, "no scratch")
    a.close()

    b = Tissue(spec)
    b.sync()
    T.debug_fail_allocs(1)
    try:
        bt = Batch([b])  # its scratch allocation fails, its tables' does not
    finally:
        T.debug_fail_allocs(0)
    bt.step(dt, 2)
    bt.sync()
    _compare(b, spec, want, wne, wtl, "batch")
    bt.close()
    b.close()

    # captured: the large tissue without scratch, a small one with early launches
    # and one whose planes need none
    for sp, steps in ((spec, 1), (_spec(60, 15, "plain"), 1), (TissueSpec(3, 3, 8, seed=93), 3)):
        ref = Tissue(sp)
        ref.step(dt, 2 * steps)
        want, (wne, wtl) = ref.read_counts(), ref.read_stats()
        ref.close()
        s = torch.cuda.Stream()
        c = Tissue(sp, stream=s)
        c.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            c.step(dt, steps)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        _compare(c, sp, want, wne, wtl, "captured")
        c.close()


def test_two_streams_step_large_tissues_at_once():
    """Two tissues on two streams, each with its own scratch in flight."""
    specs = [_spec(140, 9, "plain"), _spec(140, 8, "binding")]
    dt = 0.01
    want = []
    for s in specs:
        t = Tissue(s)
        t.step(dt, 3)
        want.append(t.read_counts())
        t.close()
    ts = [Tissue(s, stream=torch.cuda.Stream()) for s in specs]
    for _ in range(3):
        for t in ts:
            t.step(dt, 1)
    for t, x in zip(ts, want):
        assert np.array_equal(t.read_counts(), x)
        t.close()


@pytest.mark.parametrize("per_sm,n,dt", [(60, 15, 0.002), (70, 16, 0.002), (11, 32, 0.001)])
def test_planes_meet_their_range_within_a_step(per_sm, n, dt):
    """Counts just below what 16 bits hold, whose neighbours' molecules hop in:
    some cells pass the range within the step (and are run again by the 32-bit
    pass), others only in the events that the end of the step undoes."""
    spec = _spec(per_sm, n, "plain")
    d, m = orc_desc(spec), orc_model(spec)
    ref = O.init_counts(d)
    x = ref.reshape(spec.cells, 3, spec.V)
    for c in range(8):
        x[c, c % 2, 2 * c:2 * c + 2] = 65534 - c
    g = Tissue(spec)
    g.write_counts(ref, 0)
    for k in range(2):
        ne, tl = O.step(d, m, ref, k, 1, dt)
        g.step(dt, 1)
        _compare(g, spec, ref, ne, tl, f"{spec.width}x{spec.height}x{n} step {k}")
    g.close()
