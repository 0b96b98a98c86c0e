"""A step of a tissue that takes scratch, while the program captures another
stream into a graph: neither disturbs the other, in every capture mode, from the
capturing thread and from another."""
import threading

import numpy as np
import pytest

from paper_1806_10889_gb300.workloads import TissueSpec

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1806_10889_gb300.tissue import Tissue  # noqa: E402

SMS = torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("other_thread", [False, True])
@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
def test_stepping_a_large_tissue_beside_a_capture(mode, other_thread):
    large, small = TissueSpec(140, SMS, 9, seed=7), TissueSpec(3, 3, 8, seed=7)
    want = []
    for spec, steps in ((large, 2), (small, 3)):
        t = Tissue(spec)
        t.step(0.01, steps)
        want.append(t.read_counts())
        t.close()  # gives the scratch back: the steps below take it anew
    a = Tissue(small, stream=torch.cuda.Stream())
    b = Tissue(large, stream=torch.cuda.Stream())
    assert b.chi_info()["scratch_bytes"] > 0
    torch.cuda.synchronize()
    errors = []

    def step():
        try:
            b.step(0.01, 2)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=a.stream, capture_error_mode=mode):
        a.step(0.01, 2)
        if other_thread:
            th = threading.Thread(target=step)
            th.start()
            th.join()
        else:
            step()
        a.step(0.01, 1)
    assert not errors
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(b.read_counts(), want[0])
    assert np.array_equal(a.read_counts(), want[1])
    a.close()
    b.close()
