"""The segmented chi kernel in the forms its default launch shapes name, which the
library runs with the sum-tree kernel: the same instantiations with another
number of warps a block, against the oracle, bit for bit.  It still runs traces,
mixed models, captures without scratch and the cells past packed ranges."""
import numpy as np
import pytest

import oracle as O
from paper_1806_10889_gb300.workloads import TissueSpec
from tests._util import orc_desc, orc_model

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1806_10889_gb300 import tissue as T  # noqa: E402
from paper_1806_10889_gb300.tissue import Tissue  # noqa: E402

P, PRE, REC = T.KERNEL_PERSISTENT, T.LAYOUT_PREFIX, T.LAYOUT_RECOMPUTE


def _run(spec, dt, steps, config, x=None):
    d, m = orc_desc(spec), orc_model(spec)
    ref = O.init_counts(d) if x is None else x
    g = Tissue(spec)
    g.set_launch_config(*config)
    assert not g.chi_info()["sum_tree"]
    g.write_counts(ref, 0)
    for k in range(steps):
        ne, tl = O.step(d, m, ref, k, 1, dt)
        g.step(dt, 1)
        assert np.array_equal(g.read_counts(), ref), (config, k)
        gne, gtl = g.read_stats()
        assert np.array_equal(gne, ne) and np.array_equal(gtl.view(np.uint64), tl.view(np.uint64))
    g.close()
    return ref


@pytest.mark.parametrize("config", [(P, 32, 1, 0, PRE), (P, 16, 2, 0, PRE), (P, 8, 2, 0, PRE),
                                    (P, 8, 1, 0, REC)])
@pytest.mark.parametrize("w,h,n,dt", [(5, 3, 16, 0.1), (3, 2, 10, 0.1), (4, 1, 2, 0.5),
                                      (1, 3, 7, 0.2), (7, 5, 8, 1.0)])
def test_the_default_shapes_kernels_match_the_oracle(config, w, h, n, dt):
    spec = TissueSpec(w, h, n, seed=2000 + w * 100 + n, tissue_id=w * h).with_model(k_bind=0.05)
    _run(spec, dt, 3, config)


@pytest.mark.parametrize("side,n,config", [(47, 32, (P, 16, 1, 0, REC)), (78, 16, (P, 8, 1, 0, REC))])
def test_whole_tissues_of_the_counts_only_layout_match_the_oracle(side, n, config):
    _run(TissueSpec(side, side, n, seed=40 + n, tissue_id=side), 0.1, 2, config)


@pytest.mark.parametrize("n", [20, 21])
@pytest.mark.parametrize("config", [(P, 16, 1, 0, REC), (P, 32, 1, 0, PRE)])
def test_counts_past_16_bits_are_handed_back(n, config):
    spec = TissueSpec(3, 2, n, seed=71, tissue_id=3).with_model(hopD=0.0, k_off=1.0, k_in=0.0)
    x = O.init_counts(orc_desc(spec)).reshape(spec.cells, 3, spec.V)
    x[1, 0, 0] = 70000          # from the start
    x[4, 0, 5] = 65000          # within the step: R -> D + N releases it faster than it decays
    x[4, 2, 5] = 0xFFFF
    ref = _run(spec, 0.05, 3, config, x.ravel().copy()).reshape(spec.cells, 3, spec.V)
    assert ref[4, 0, 5] > 0xFFFF
