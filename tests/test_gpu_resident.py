"""GPU parity of the launch shape for short vectors that keeps whole columns (all M rows of a few
column groups) resident in shared memory for every round of a call.  Replicas and peer traces
must equal, bit for bit, those of the launch shapes that keep nothing on chip across rounds
(fuse_rounds = 1), and match the CPU oracle within the fp32 tolerance; telemetry sums are
accumulated in a different order and agree to fp32 rounding."""
import numpy as np
import pytest

from oracle import oracle

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def nm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2009_05766_b200 import binding
    binding.lib()
    return binding


def full_adj(M):
    return (1 - np.eye(M)).astype(np.uint8)


def random_policy(M, rng, zeros=0.0):
    P = rng.random((M, M)) + 0.05
    if zeros > 0:
        mask = rng.random((M, M)) < zeros
        mask[np.arange(M), (np.arange(M) + 1) % M] = False
        P[mask] = 0.0
    return P / P.sum(axis=1, keepdims=True)


# a thread per column group (small M), rows split over threads (larger M), ragged tails, one column,
# more tiles than resident CTAs, the largest M that still fits (a 4-element column of 4700 rows)
SHAPES = [(2, 1), (3, 9), (4, 4096), (7, 4099), (5, 67), (2, 280_001), (66, 515), (67, 515), (130, 37), (300, 1030),
          (512, 1024), (1000, 131), (4096, 64), (4700, 7)]


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("M,d", SHAPES)
def test_resident_columns_change_no_bit(nm, M, d, storage):
    rng = np.random.default_rng(M * 5 + d)
    P = random_policy(M, rng, zeros=0.3 if M > 4 else 0.0)
    kw = dict(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=1, seed=d + M, trace_rounds=16,
              storage=storage)
    plain = nm.Netmax(fuse_rounds=1, **kw)
    res = nm.Netmax(**kw)
    rounds = 0
    for n in (1, 7, 16, 2, 11):              # single rounds, batches, a full lap of the ring and a wrap
        launches = res.kernel_launches
        plain.round(n)
        res.round(n)
        rounds += n
        if n >= 2:                           # (a single round does not repay bringing the columns on chip)
            assert res.kernel_launches - launches == 3, "the rounds did not run on resident columns"
        else:
            assert res.kernel_launches - launches == 2, "a single round should take the per-round kernel"
    xa, xb = plain.read_replicas(), res.read_replicas()
    assert (xa.view(np.uint32) == xb.view(np.uint32)).all()
    assert (plain.peer_trace(rounds - 16, 16) == res.peer_trace(rounds - 16, 16)).all()
    (ca, la), (cb, lb) = plain.telemetry(rounds - 16, 16), res.telemetry(rounds - 16, 16)
    np.testing.assert_allclose(cb, ca, rtol=2e-5)
    np.testing.assert_allclose(lb, la, rtol=2e-5)
    plain.close()
    res.close()


def test_short_calls_do_not_pay_for_bringing_the_columns_on_chip(nm):
    """Resident columns are loaded and stored once per call; a call takes that shape only from the number of rounds at
    which it was measured to pay (2 up to a million elements, 6 up to four million, then 8 and 16)."""
    for M, d, short, long_ in ((4, 4096, 1, 2), (4096, 1024, 4, 6), (1024, 8192, 7, 8)):
        P = np.full((M, M), 1.0 / (M - 1))
        np.fill_diagonal(P, 0.0)
        kw = dict(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=1, seed=5, trace_rounds=32)
        a, b = nm.Netmax(**kw), nm.Netmax(fuse_rounds=1, **kw)
        for n, resident in ((short, False), (long_, True), (short, False)):
            before = a.kernel_launches
            a.round(n)
            b.round(n)
            launches = a.kernel_launches - before          # sampler + (resident kernel + tile sums | per-round kernels)
            assert (launches == 3) == resident, (M, d, n, launches)
        assert (a.read_replicas().view(np.uint32) == b.read_replicas().view(np.uint32)).all()
        assert (a.peer_trace() == b.peer_trace()).all()
        a.close()
        b.close()


@pytest.mark.parametrize("M,d", [(5048, 146), (5040, 9), (6000, 33)])
def test_more_workers_than_fit_on_chip(nm, M, d):
    """Beyond about 4700 workers the columns do not fit a CTA's shared memory and the per-round kernels run; around
    M = 5040 their table of draws needs just under 48 KB of dynamic shared memory, which with the kernels' static
    part is over the default limit (such a context once failed to plan its launch)."""
    rng = np.random.default_rng(M + d)
    P = random_policy(M, rng, zeros=0.5)
    kw = dict(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=1, seed=M, trace_rounds=8)
    one, many = nm.Netmax(fuse_rounds=1, **kw), nm.Netmax(**kw)
    o = oracle.Sim(M, d, P, full_adj(M), alpha=0.05, rho=one.get_policy()[1], sigma=0.1, objective=1, seed=M)
    o.init(1.0, 1.0)
    o.set_x(one.read_replicas())                       # (the two sides' initial normals differ in the last bit)
    o.set_c(one.read_centres())
    for n in (1, 5):
        one.round(n)
        many.round(n)
        o.round(n)
    xa, xb, xo = one.read_replicas(), many.read_replicas(), o.x().astype(np.float64)
    assert (xa.view(np.uint32) == xb.view(np.uint32)).all()
    assert (one.peer_trace(0, 6) == o.trace(0, 6)).all() and (many.peer_trace(0, 6) == o.trace(0, 6)).all()
    assert (np.abs(xa.astype(np.float64) - xo) <= TOL * (1.0 + np.abs(xo))).all()
    one.close()
    many.close()


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("M,d", [(4, 4096), (6, 4099), (64, 515), (130, 37), (1000, 131)])
def test_resident_columns_match_the_oracle(nm, M, d, objective):
    rng = np.random.default_rng(M + d)
    P = random_policy(M, rng, zeros=0.2)
    g = nm.Netmax(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=objective, seed=9, trace_rounds=64)
    o = oracle.Sim(M, d, P, full_adj(M), alpha=0.05, rho=g.get_policy()[1], sigma=0.1, objective=objective, seed=9)
    o.init(1.0, 1.0)
    x0, c0 = g.read_replicas(), g.read_centres()       # (the two sides' initial normals differ in the last bit)
    o.set_x(x0)
    o.set_c(c0)
    for n in (30, 1, 9):
        g.round(n)
        o.round(n)
    assert (g.peer_trace() == o.trace()).all()
    got, want = g.read_replicas().astype(np.float64), o.x().astype(np.float64)
    assert (np.abs(got - want) <= TOL * (1.0 + np.abs(want))).all()
    gc, gl = g.telemetry()
    oc, ol = o.telemetry()
    np.testing.assert_allclose(gc, oc, rtol=1e-4, atol=1e-9)
    np.testing.assert_allclose(gl, ol, rtol=1e-4, atol=1e-9)
    g.close()


def test_split_calls_change_no_bit_of_replicas_trace_or_telemetry(nm):
    """Every round runs on resident columns whatever the call pattern, so even telemetry is bit-identical."""
    rng = np.random.default_rng(8)
    M, d = 5, 2051
    kw = dict(M=M, d=d, lr=0.05, prob=random_policy(M, rng), sigma=0.1, x0_std=1.0, c_std=1.0, seed=11, trace_rounds=16)
    a, b = nm.Netmax(**kw), nm.Netmax(**kw)
    a.round(37)
    for n in (1, 0, 15, 16, 5):
        b.round(n)
    assert (a.read_replicas() == b.read_replicas()).all()
    ta, tb = a.telemetry(21, 16), b.telemetry(21, 16)
    assert (ta[0] == tb[0]).all() and (ta[1] == tb[1]).all()
    a.close()
    b.close()


# cut tiles (few tiles per CTA, 16 rounds and more): one tile more than CTAs; a last CTA with only the rest of a tile;
# two CTAs per SM; long vectors; instances with 1, 4, 11 and 12 rows per thread, the largest number of workers
@pytest.mark.parametrize("M,d,rounds,storage", [(4096, 149 * 4, 16, "f32"), (4096, 1024, 37, "bf16"), (2100, 1801, 20, "f32"),
                                                (4700, 603, 17, "f32"), (350, 50_002, 16, "f32"), (93, 90_003, 23, "bf16"),
                                                (64, 77_001, 16, "f32"), (1000, 4_001, 40, "f32"), (13, 100_003, 18, "f32")])
def test_cut_tiles_change_no_bit(nm, M, d, rounds, storage):
    rng = np.random.default_rng(M + d)
    P = random_policy(M, rng)
    kw = dict(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=1, seed=d + M, trace_rounds=64, storage=storage)
    plain, res = nm.Netmax(fuse_rounds=1, **kw), nm.Netmax(**kw)
    plain.round(rounds)
    res.round(rounds)
    assert (plain.read_replicas().view(np.uint32) == res.read_replicas().view(np.uint32)).all()
    (ca, la), (cb, lb) = plain.telemetry(), res.telemetry()
    np.testing.assert_allclose(cb, ca, rtol=2e-5)      # fp32 partial sums in another order: M up to 4700 of them, 2e-5 as above
    np.testing.assert_allclose(lb, la, rtol=2e-5)
    plain.close()
    res.close()


# both samplers (thresholds through the caches, rows in shared memory) around the rule's borders: M not a multiple of
# four, of sixteen, of the rows of a CTA; rounds that fill no pass; two rows per CTA; a row whose last entries are zero
@pytest.mark.parametrize("M,rounds", [(127, 1100), (128, 1024), (131, 1001), (1025, 129), (4095, 103), (4096, 70), (5003, 127), (8200, 210)])
def test_peer_draws_equal_the_oracle(nm, M, rounds):
    import torch
    rng = np.random.default_rng(M)
    P = rng.random((M, M)) + 0.05
    P[:, M - 5:] *= rng.random((M, 1)) < 0.5           # in half of the rows the last five workers are never drawn
    P /= P.sum(axis=1, keepdims=True)
    g = nm.Netmax(M=M, d=8, lr=0.05, prob=P, seed=M, trace_rounds=4)
    out = torch.full((rounds, M), -1, dtype=torch.int32, device="cuda")
    g.sample_peers(7, rounds, out.data_ptr())
    assert (out.cpu().numpy() == oracle.peer_draws(P, M, 7, rounds)).all()
    g.close()


@pytest.mark.parametrize("when", ["address taken first", "address taken after the rounds"])
@pytest.mark.parametrize("own_workspace", [False, True])
@pytest.mark.parametrize("rounds", [1, 5])
def test_replicas_changed_on_the_device_are_what_is_read(nm, when, own_workspace, rounds):
    """A program that reads small replicas after every call gets them with the rounds -- but one that has changed them on
    the device in between gets what it wrote, and a read after a read what is there."""
    import torch
    M, d = 4, 1003
    kw = dict(M=M, d=d, lr=0.05, prob=random_policy(M, np.random.default_rng(3)), sigma=0.1, x0_std=1.0, c_std=1.0, seed=5)
    if own_workspace:
        size = nm.Netmax.workspace_size(M, d)
        memory = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        kw.update(workspace=(memory.data_ptr() + 255) // 256 * 256, workspace_bytes=size)
    g, same = nm.Netmax(**kw), nm.Netmax(**{k: v for k, v in kw.items() if not k.startswith("workspace")})

    def row(i):  # row i of the current replicas, as a tensor over the context's memory
        ptr, ld = g.replicas_device()
        iface = {"shape": (d,), "typestr": "<f4", "data": (ptr + 4 * i * ld, False), "version": 3}
        return torch.as_tensor(type("Row", (), {"__cuda_array_interface__": iface})(), device="cuda")

    def step():
        for s in (g, same):
            s.round(rounds)

    step()
    assert (g.read_replicas() == same.read_replicas()).all()   # (from here on reads are expected after every call)
    if when == "address taken first":
        row(0)
    for k in range(3):
        step()
        row(2).fill_(0.25 * (k + 1))
        torch.cuda.synchronize()
        x = g.read_replicas()
        want = same.read_replicas()
        want[2] = 0.25 * (k + 1)
        assert (x.view(np.uint32) == want.view(np.uint32)).all()
        assert (g.read_replicas() == want).all()
        same.set_replicas(want)
    g.close()
    same.close()


@pytest.mark.parametrize("M,d,ring", [(4, 1003, 16), (3, 400_003, 16), (70, 260, 7)])
def test_telemetry_and_peers_do_not_depend_on_when_they_are_looked_at(nm, M, d, ring):
    """Rounds of a call that follows a look leave telemetry and peers in host memory, others on the device: whatever the
    order of looks, every round that is still in the ring reads the same."""
    kw = dict(M=M, d=d, lr=0.05, prob=random_policy(M, np.random.default_rng(M)), sigma=0.1, x0_std=1.0, c_std=1.0, seed=9, trace_rounds=ring)
    never, always, some = nm.Netmax(**kw), nm.Netmax(**kw), nm.Netmax(**kw)
    for k, n in enumerate((2, 1, 5, 3, 2, 1, 4, 2 * ring + 3, 1, 6)):
        for g in (never, always, some):
            g.round(n)
        first = max(0, never.rounds_done - ring)
        if k % 3 == 2:
            some.telemetry(first, 1)
        if k % 4 == 1:
            some.peer_trace(first, 1)
        always.telemetry(first, 1)
        always.peer_trace(first, 1)
    want = never.telemetry(first, ring), never.peer_trace(first, ring)
    for g in (always, some):
        assert (g.peer_trace(first, ring) == want[1]).all()
        for got, ref in zip(g.telemetry(first, ring), want[0]):
            np.testing.assert_allclose(got, ref, rtol=1e-12)
    for g in (never, always, some):
        g.close()
