"""A context whose device memory is the caller's workspace holds no other until its links are changed, whatever creation and other changes of
the policy of many workers borrow; then the block of that search, once, until it is destroyed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2009_05766_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("M", [320, 700, 1500])
def test_nothing_else_is_held_beside_the_workspace(nm, M):
    import torch
    rng = np.random.default_rng(M)
    links = [np.exp(rng.uniform(0.0, 3.0, (M, M))) for _ in range(2)]
    links = [np.triu(s, 1) + np.triu(s, 1).T for s in links]
    P = np.full((M, M), 1.0 / M)
    size = nm.Netmax.workspace_size(M, 64)
    workspace = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
    base = (workspace.data_ptr() + 255) // 256 * 256

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def walk():
        seen = []
        sim = nm.Netmax(M=M, d=64, lr=0.05, prob=P, link_speed_gbps=links[0], policy_K=2, policy_R=2, seed=1, workspace=base, workspace_bytes=size)
        seen.append(free())
        for change in ({"prob": P}, {}, {"link_speed_gbps": links[1]}, {"prob": P}, {"link_speed_gbps": links[0]}):
            sim.set_policy(**change)
            seen.append(free())
        sim.close()
        return seen + [free()]

    walk()                              # (kernels are loaded, and the like)
    before = free()
    seen = walk()
    assert seen[:3] == [before] * 3 and seen[-1] == before       # (allocations come in pieces of 2 MB: none is too small to be seen)
    assert len(set(seen[3:6])) == 1 and 0 <= before - seen[3] <= 17 * M * M + (305 * 8 * M) + (4 << 20)
