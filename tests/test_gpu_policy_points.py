"""The device generator's row solver, bounds and in-place Y_P over sizes at which its loops can go wrong: odd and even rows,
fewer and more links than threads, links in one direction only, equal times, grids of more points than one launch takes;
against the host generator (same readings, other code: both settle lambda_2 to 1e-13, P to 1e-10)."""
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


def _speeds(M, seed, missing=0.0, spread=100.0):
    rng = np.random.default_rng(seed)
    s = np.exp(rng.uniform(0.0, np.log(spread), (M, M)))
    s[rng.random((M, M)) < missing] = 0.0
    s[np.arange(M), (np.arange(M) + 1) % M] = 2.0     # a ring keeps the graph connected
    s = np.triu(s, 1) + np.triu(s, 1).T
    s[0, M - 1] = s[M - 1, 0] = 2.0
    return s


@pytest.mark.parametrize("M,K,R,missing,spread", [(2, 3, 5, 0.0, 100.0), (3, 4, 70, 0.0, 100.0), (33, 5, 33, 0.0, 100.0), (64, 3, 4, 0.9, 10.0),
                                                  (97, 4, 4, 0.0, 1.0), (255, 3, 6, 0.3, 1000.0), (300, 2, 40, 0.0, 100.0), (514, 3, 3, 0.0, 100.0)])
def test_device_generator_matches_host_generator(nm, M, K, R, missing, spread):
    t, adj = nm.netmax_iteration_times(_speeds(M, M + R, missing, spread), 4096)
    outcome = []
    for generate in (nm.netmax_policy_generate, nm.netmax_policy_generate_device):
        try:
            outcome.append(generate(t, adj, 0.05, K, R))
        except nm.NetmaxError as e:
            outcome.append(e.code)
    if isinstance(outcome[0], int):
        assert outcome[0] == outcome[1]
        return
    (Ph, rhoh, infoh), (Pd, rhod, infod) = outcome
    assert (infod["k"], infod["r"]) == (infoh["k"], infoh["r"]) and rhod == rhoh
    np.testing.assert_allclose(Pd, Ph, atol=1e-10)
    assert infod["lam2"] == pytest.approx(infoh["lam2"], abs=1e-10)


def test_changes_of_links_in_several_contexts(nm):
    """Changes of either kind in several contexts, in turn, with the searches' device memory borrowed and given back each time."""
    sizes = (190, 400, 613)
    sims = [nm.Netmax(M=M, d=64, lr=0.05, prob=np.full((M, M), 1.0 / M), link_speed_gbps=_speeds(M, 1), policy_K=3, policy_R=3, seed=M)
            for M in sizes]
    for turn in range(3):
        for M, sim in zip(sizes, sims):
            if turn == 1:
                sim.set_policy(prob=np.full((M, M), 1.0 / M))
            else:
                sim.set_policy(link_speed_gbps=_speeds(M, 2 + turn))
                P, rho = sim.get_policy()
                t, adj = nm.netmax_iteration_times(_speeds(M, 2 + turn), 64)
                Ph, rhoh, _ = nm.netmax_policy_generate(t, adj, 0.05, 3, 3)
                assert rho == pytest.approx(rhoh, rel=1e-12)
                np.testing.assert_allclose(P, Ph, atol=1e-10)
            sim.round(2)
    for sim in sims:
        sim.close()


def test_first_change_without_device_memory_to_spare(nm):
    """In a program that has handed out all device memory the policy is searched on the host (590 workers: tables come from the host
    at creation)."""
    import torch
    M, d = 590, 64     # the search wants 7 MB
    kw = dict(M=M, d=d, lr=0.05, prob=np.full((M, M), 1.0 / M), link_speed_gbps=_speeds(M, 1), policy_K=3, policy_R=3, seed=2)
    with_block, without = nm.Netmax(**kw), nm.Netmax(**kw)
    with_block.set_policy(link_speed_gbps=_speeds(M, 3))      # (every kernel has run before the memory is gone)
    for sim in (with_block, without):
        sim.round(2)
        sim.peer_trace(0, 2)
    held, step = [], 1 << 36
    try:
        while step >= 1 << 18:
            try:
                held.append(torch.cuda.caching_allocator_alloc(step))
            except torch.cuda.OutOfMemoryError:
                step >>= 1
        assert torch.cuda.cudart().cudaMemGetInfo(0)[0] < 7 << 20
        without.set_policy(link_speed_gbps=_speeds(M, 3))
    finally:
        for p in held:
            torch.cuda.caching_allocator_delete(p)
        torch.cuda.empty_cache()
    P, rho = with_block.get_policy()
    Pw, rhow = without.get_policy()
    assert rhow == pytest.approx(rho, rel=1e-12)
    np.testing.assert_allclose(Pw, P, atol=1e-10)
    for sim in (with_block, without):
        sim.round(3)
    assert (with_block.peer_trace(2, 3) == without.peer_trace(2, 3)).mean() > 0.999
    with_block.close()
    without.close()
