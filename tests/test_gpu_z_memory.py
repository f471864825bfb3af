"""The z vectors of a mixed handle take room for its update group, no more (batch handles have smaller
groups than single ones), and st_workspace_bytes stays an upper bound."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_each_pending_z_is_one_padded_vector(monkeypatch):
    import paper_2201_10062_gb300 as P
    from paper_2201_10062_gb300 import build

    build.build()
    P.load_library()
    # mx = 3: the padding is a third of the unknowns
    spec = P.ProblemSpec(2, 3, 1023, 1024, 1.0, "theta", 0.5, None, "PH", "mixed")
    used = {}
    P.Solver(spec).close()  # what the first handle of a process brings along
    for group in (1, 8):
        monkeypatch.setenv("ST_UPDATE_GROUP", str(group))
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        s = P.Solver(spec)
        used[group] = free - torch.cuda.mem_get_info()[0]
        # the allocator's granularity of 2 MB for each of some fifteen allocations
        assert used[group] <= P.st_workspace_bytes(spec) + (30 << 20)
        s.close()
    padded = 4 * 4 * 1023 * 1024
    assert abs(used[8] - used[1] - 7 * padded) <= 4 << 20
