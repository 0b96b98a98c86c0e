"""The memory of a batch's sum-tree launches: reported, kept to a limit without a
change of results, and part of what a server's budget bounds."""
import numpy as np
import pytest

from paper_1806_10889_gb300.batching import Batch
from paper_1806_10889_gb300.workloads import Request, TissueSpec

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1806_10889_gb300.serving import Server, request_bytes  # noqa: E402
from paper_1806_10889_gb300.tissue import KERNEL_WARP, Tissue  # noqa: E402

SMS = torch.cuda.get_device_properties(0).multi_processor_count


def test_a_limit_moves_classes_to_their_shape_s_kernel():
    specs = [TissueSpec(120, SMS, 16, seed=41, tissue_id=0), TissueSpec(140, SMS, 8, seed=41, tissue_id=1)]
    outs, held = [], []
    for limit in (None, 0, 80 << 20):
        ms = [Tissue(s) for s in specs]
        b = Batch(ms, scratch_limit=limit)
        info = [b.chi_info(i) for i in range(2)]
        held.append([i["scratch_bytes"] for i in info])
        assert b.scratch_bytes() == sum(held[-1]) <= (limit if limit is not None else 1 << 62)
        assert [i["sum_tree"] for i in info] == [bool(h) for h in held[-1]]
        b.step(0.005, 2)
        b.sync()
        outs.append([m.read_counts() for m in ms])
        b.close()
        for m in ms:
            m.close()
    assert held[0][0] > 1 << 26 and held[0][1] > 1 << 24  # records of both classes
    assert held[1] == [0, 0] and held[2] == [held[0][0], 0]
    for o in outs[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(o, outs[0]))


def test_a_tissue_reports_what_its_step_takes():
    t = Tissue(TissueSpec(120, SMS, 16, seed=41))
    info = t.chi_info()
    assert info["sum_tree"] and info["launches"] == 2 and info["scratch_bytes"] > 1 << 26
    t.set_launch_config(KERNEL_WARP, 32, 4, 0, 0)
    assert t.chi_info() == {"sum_tree": False, "lanes_per_cell": 32, "launches": 1,
                            "scratch_bytes": 0}
    t.close()
    t = Tissue(TissueSpec(2, 2, 8, seed=41))
    assert t.chi_info() == {"sum_tree": True, "lanes_per_cell": 32, "launches": 1,
                            "scratch_bytes": 0}
    t.close()


def test_a_server_s_budget_holds_the_batch_s_scratch_too():
    reqs = [Request(0, 0.0, 1, 135, 16, 4, 0.002)]
    need = request_bytes(reqs[0])
    seen = []

    def serve(budget):
        srv = Server(budget_bytes=budget, chunk_steps=2, keep_counts=True)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        out = srv.run(reqs, on_round=lambda s, i: seen.append(free - torch.cuda.mem_get_info()[0]))
        assert srv.peak_used <= budget and all(r.digest and not r.rejected for r in out)
        return [r.digest for r in out]

    want = serve(1 << 33)
    for budget in (need, need + (40 << 20), need + (80 << 20)):
        del seen[:]
        assert serve(budget) == want
        # beside the budget: what a context, a graph and the allocators round up
        assert max(seen) <= budget + (24 << 20), (budget, seen)
