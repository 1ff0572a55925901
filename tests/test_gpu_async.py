"""GPU parity of the asynchronous timeline (one worker per global step, Eq. 17) and of the
on-demand telemetry, against the CPU oracle: event traces (worker, peer, local iteration,
finish time) bit-exact, replicas within 1e-5 (1 + |x|)."""
import numpy as np
import pytest

from oracle import oracle
from oracle import policy as opolicy
from paper_2009_05766_b200 import workloads

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


def close(got, want, tol=TOL):
    got64, want64 = got.astype(np.float64), want.astype(np.float64)
    excess = np.abs(got64 - want64) - tol * (1.0 + np.abs(want64))
    assert excess.max() <= 0.0, f"max excess {excess.max():.3e}"


def random_policy(M, rng, self_prob=True):
    P = rng.random((M, M)) + 0.05
    if not self_prob:
        np.fill_diagonal(P, 0.0)
    return P / P.sum(axis=1, keepdims=True)


def random_times(M, rng):
    t = rng.uniform(1.0, 4.0, (M, M))
    t = 0.5 * (t + t.T)
    t[np.diag_indices(M)] = 0.2
    return t


@pytest.mark.parametrize("objective", [0, 1])
@pytest.mark.parametrize("M,d", [(2, 5), (3, 1), (5, 67), (8, 4099), (16, 3001), (64, 515), (300, 37)])
def test_async_steps_match_oracle(nm, M, d, objective):
    rng = np.random.default_rng(M * 13 + d)
    P, t = random_policy(M, rng), random_times(M, rng)
    g = nm.Netmax(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=objective, seed=d + 3)
    rho = g.get_policy()[1]
    o = oracle.Sim(M, d, P, full_adj(M), alpha=0.05, rho=rho, sigma=0.1, objective=objective, seed=d + 3)
    o.init(1.0, 1.0)
    g.async_begin(t, beta=0.7)
    o.async_begin(t, beta=0.7)
    steps = 12 * M
    for n in (1, 0, steps // 3, steps - 1 - steps // 3):
        g.async_steps(n)
        o.async_steps(n)
    gw, gp, gn, gt = g.async_trace()
    ow, op, on, ot = o.async_trace()
    assert (gw == ow).all() and (gp == op).all() and (gn == on).all() and (gt == ot).all()
    close(g.read_replicas(), o.x(), tol=2e-5 if objective == 0 else TOL)
    assert g.async_time() == (o.async_now, steps)
    ge, gc = g.async_ema()
    oe, oc = o.async_ema()
    assert (gc == oc).all() and (ge == oe).all()
    # on-demand telemetry against the oracle's definition on its own state
    cons, loss = g.measure()
    ocons, oloss = o.telemetry_now()
    assert cons == pytest.approx(ocons, rel=1e-4) and loss == pytest.approx(oloss, rel=1e-4)
    with pytest.raises(nm.NetmaxError):
        g.round(1)
    g.close()


def test_async_policy_and_time_changes_apply_to_later_iterations(nm):
    rng = np.random.default_rng(5)
    M, d = 6, 500
    P1, P2 = random_policy(M, rng, self_prob=False), random_policy(M, rng)
    t1, t2 = random_times(M, rng), random_times(M, rng)
    g = nm.Netmax(M=M, d=d, lr=0.05, prob=P1, sigma=0.05, x0_std=1.0, c_std=1.0, seed=8)
    o = oracle.Sim(M, d, P1, full_adj(M), alpha=0.05, rho=g.get_policy()[1], sigma=0.05, objective=1, seed=8)
    o.init(1.0, 1.0)
    g.async_begin(t1, 0.5)
    o.async_begin(t1, 0.5)
    g.async_steps(40)
    o.async_steps(40)
    g.set_policy(prob=P2)
    o.set_policy(P2, full_adj(M), g.get_policy()[1])
    g.async_set_times(t2)
    o.async_set_times(t2)
    g.async_steps(60)
    o.async_steps(60)
    for a, b in zip(g.async_trace(), o.async_trace()):
        assert (a == b).all()
    close(g.read_replicas(), o.x())
    for a, b in zip(g.async_ema(), o.async_ema()):
        assert (a == b).all()
    g.close()


def test_iterations_in_flight_keep_their_weight_and_duration(nm):
    """Algorithm 2 reads the policy at the top of an iteration and records the time the iteration
    took: with every first iteration in flight, a new policy that gives the drawn peers probability
    zero and a slower time matrix must leave those iterations' pulls (old alpha rho / (2 p_im)) and
    moving averages (old t_im) untouched.  Closed form, no oracle."""
    M, d, alpha, beta = 3, 1027, 0.1, 0.5
    P1 = np.array([[0, 1.0, 0], [0, 0, 1.0], [1.0, 0, 0]])
    P2 = np.array([[0, 0, 1.0], [1.0, 0, 0], [0, 1.0, 0]])
    rho1, rho2 = 0.8, 2.4
    t1 = np.array([[0.1, 1.0, 1.0], [1.0, 0.1, 1.0], [1.0, 1.0, 0.1]])
    x0 = np.random.default_rng(12).standard_normal((M, d)).astype(np.float32)
    g = nm.Netmax(M=M, d=d, lr=alpha, prob=P1, rho=rho1, objective=0, seed=13)
    g.set_replicas(x0)
    g.async_begin(t1, beta)
    g.set_policy(prob=P2, rho=rho2)
    g.async_set_times(3.0 * t1)
    a32 = float(np.float32(alpha))
    w_old, w_new = float(np.float32(a32 * rho1)), float(np.float32(a32 * rho2))
    g.async_steps(6)
    worker, peer, local_iter, time = g.async_trace()
    x = x0.astype(np.float64)
    for i, m, n, tt in zip(worker, peer, local_iter, time):
        assert m == ((i + 1) % M if n == 0 else (i + 2) % M)
        assert tt == pytest.approx(1.0 if n == 0 else 4.0)
        x[i] = np.float32(x[i] - (w_old if n == 0 else w_new) * (x[i] - x[m]))
    close(g.read_replicas(), x.astype(np.float32))
    ema, count = g.async_ema()
    want = np.zeros((M, M))
    for i in range(M):
        want[i, (i + 1) % M] = (1 - beta) * 1.0
        want[i, (i + 2) % M] = (1 - beta) * 3.0
    np.testing.assert_allclose(ema, want, rtol=1e-12)
    assert (count == (want > 0)).all()
    g.close()


def test_async_needs_begin_and_a_fresh_context(nm):
    M, d = 3, 10
    P = random_policy(M, np.random.default_rng(1))
    g = nm.Netmax(M=M, d=d, lr=0.05, prob=P, x0_std=1.0, c_std=1.0, seed=1)
    with pytest.raises(nm.NetmaxError):
        g.async_steps(1)
    g.round(1)
    with pytest.raises(nm.NetmaxError):
        g.async_begin(None, 0.5)
    h = nm.Netmax(M=M, d=d, lr=0.05, prob=P, x0_std=1.0, c_std=1.0, seed=1, trace_rounds=4)
    with pytest.raises(nm.NetmaxError):
        h.async_begin(None, 1.0)
    h.async_begin(None, 0.5)                      # iteration times from (equal) link speeds
    h.async_steps(2000)
    assert h.async_time()[1] == 2000
    w, p, n, t = h.async_trace(2000 - 1024, 1024)
    assert (np.diff(t) >= 0).all()
    with pytest.raises(nm.NetmaxError) as e:
        h.async_trace(0, 10)
    assert e.value.code == -5
    g.close()
    h.close()


def test_measure_matches_round_telemetry(nm):
    M, d = 7, 12345
    P = random_policy(M, np.random.default_rng(2))
    g = nm.Netmax(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, seed=2)
    g.round(5)
    cons, loss = g.measure()
    before = g.read_replicas()
    g.round(1)
    tc, tl = g.telemetry(5, 1)                   # the round's telemetry is taken on its start state
    assert cons == pytest.approx(tc[0], rel=1e-6) and loss == pytest.approx(tl[0], rel=1e-6)
    h = nm.Netmax(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, seed=2)
    h.round(5)
    assert (h.read_replicas() == before).all()   # measuring changed nothing
    g.close()
    h.close()


def test_async_full_size_resnet18_vectors_on_sampled_columns(nm):
    w = workloads.config(2)
    t, adj = opolicy.iteration_times(w.link_speeds(0), w.d)
    P, rho, _ = opolicy.generate_policy(t, adj, w.lr, 6, 6)
    cols = workloads.sample_columns(w.d, 2000, w.seed)
    g = nm.Netmax(M=w.M, d=w.d, lr=w.lr, link_speed_gbps=w.link_speeds(0), prob=P, rho=rho, sigma=w.sigma,
                  x0_std=w.x0_std, c_std=w.c_std, seed=w.seed)
    o = oracle.Sim(w.M, w.d, P, adj, alpha=w.lr, rho=rho, sigma=w.sigma, objective=1, seed=w.seed, cols=cols)
    o.init(w.x0_std, w.c_std)
    g.async_begin(None, 0.9)                      # the library's own iteration times from the link speeds
    o.async_begin(t, 0.9)
    steps = 40 * w.M
    g.async_steps(steps)
    o.async_steps(steps)
    for a, b in zip(g.async_trace(), o.async_trace()):
        assert (a == b).all()
    close(g.read_columns(cols), o.x())
    g.close()


def test_network_monitor_loop_matches_an_oracle_driven_replay(nm):
    """Algorithm 1 on the simulated clock: workers start with uniform probabilities, the monitor
    installs Algorithm 3's policy from the measured (EMA) iteration times every period, and
    adapts one period after the link speeds change.  The replay drives the oracle step by step
    and computes each policy with the oracle's numpy Algorithm 3."""
    rng = np.random.default_rng(21)
    M, d, lr, beta, K, R = 6, 400, 0.05, 0.8, 6, 6

    def times(seed):
        r = np.random.default_rng(seed)
        s = np.triu(np.exp(r.uniform(np.log(1.0), np.log(40.0), (M, M))), 1)
        return opolicy.iteration_times(s + s.T, 1_000_000)

    t1, adj = times(1)
    t2, _ = times(2)
    P0 = np.full((M, M), 1.0 / M)                       # Algorithm 2: initial probabilities 1/M
    rho0 = 0.5 / (2 * lr * M)
    period = 12 * t1[adj == 1].mean()
    g = nm.Netmax(M=M, d=d, lr=lr, prob=P0, rho=rho0, sigma=0.05, x0_std=1.0, c_std=1.0, seed=4, policy_K=K, policy_R=R)
    o = oracle.Sim(M, d, P0, adj, alpha=lr, rho=rho0, sigma=0.05, objective=1, seed=4)
    o.init(1.0, 1.0)
    g.async_begin(t1, beta)
    o.async_begin(t1, beta)
    g.async_monitor(period)
    state = dict(next=period, t=t1, refreshes=0)

    def replay(n):
        for _ in range(n):
            while o.async_next_time >= state["next"]:
                ema, count = o.async_ema()
                est = np.where(count > 0, ema / (1.0 - beta ** np.maximum(count, 1)), state["t"])
                est = np.where((adj == 1) | np.eye(M, dtype=bool), est, 0.0)
                try:
                    P, rho, _ = opolicy.generate_policy(est, adj, lr, K, R)
                    o.set_policy(P, adj, rho)
                    state["refreshes"] += 1
                except ValueError:
                    pass
                state["next"] += period
            o.async_steps(1)

    g.async_steps(150)
    replay(150)
    g.async_set_times(t2)                                # the network changes
    o.async_set_times(t2)
    state["t"] = t2
    g.async_steps(250)
    replay(250)
    for a, b in zip(g.async_trace(), o.async_trace()):
        assert (a == b).all()
    close(g.read_replicas(), o.x())
    assert g.async_monitor_refreshes == state["refreshes"] >= 3
    Pg, rhog = g.get_policy()
    assert np.abs(Pg - P0).max() > 0.05                  # the monitor moved the policy away from uniform
    g.close()


def test_adaptive_policy_converges_sooner_in_simulated_time(nm):
    """The paper's claim, on its own process: with a heterogeneous network (2 machines x 4
    workers, inter-machine links 10x slower) the adaptive policy of Algorithm 3 (printed rho
    grid, K = 10) reaches a given distance from the optimum mean(c_i) in less simulated time
    than uniform neighbour choice."""
    M, d, lr = 8, 2000, 0.1
    group = np.arange(M) // 4
    s = np.where(group[:, None] == group[None, :], 100.0, 10.0)
    np.fill_diagonal(s, 0.0)
    t, adj = nm.netmax_iteration_times(s, 11_173_962)
    c = workloads.clustered_centres(M, d, 4, spread=1.0, within=0.3, seed=1)
    cbar = c.astype(np.float64).mean(axis=0)
    P_ad, rho_ad, _ = nm.netmax_policy_generate(t, adj, lr, 10, 20, rho_upper=0.5 / lr)
    P_un = (1.0 - np.eye(M)) / (M - 1)
    rho_un = 0.9 / (M - 1) / (2 * lr)
    assert P_ad[0, 1] > 1.3 * P_ad[0, 5]                 # fast links are preferred

    def time_to(P, rho, level):
        g = nm.Netmax(M=M, d=d, lr=lr, link_speed_gbps=s, prob=P, rho=rho, sigma=0.05, x0_std=1.0, seed=5)
        g.set_centres(c)
        g.async_begin(t, 0.9)
        try:
            for _ in range(300):
                g.async_steps(10)
                x = g.read_replicas().astype(np.float64)
                if ((x - cbar) ** 2).sum(axis=1).mean() / d < level:
                    return g.async_time()[0]
            return float("inf")
        finally:
            g.close()

    for level in (0.2, 0.12):
        t_un, t_ad = time_to(P_un, rho_un, level), time_to(P_ad, rho_ad, level)
        assert np.isfinite(t_un) and np.isfinite(t_ad)
        assert t_un / t_ad > 1.15, (level, t_un, t_ad)


# steps of one call on resident columns (launches of at most 160) against the same steps call by call (one launch each):
# lengths around a launch, ragged tails, one column group, narrow and wide CTAs, the last columns of a partial tile
@pytest.mark.parametrize("M,d,steps,storage", [(2, 3, 160, "f32"), (3, 8_191, 161, "f32"), (8, 700_003, 321, "bf16"), (8, 1_200_001, 40, "f32"),
                                               (16, 300_002, 159, "f32"), (40, 50_001, 162, "f32"), (150, 33, 400, "f32"),
                                               (150, 33, 400, "bf16")])
@pytest.mark.parametrize("objective", [0, 1])
def test_steps_on_resident_columns_change_no_bit(nm, M, d, steps, storage, objective):
    rng = np.random.default_rng(M + d)
    P, t = random_policy(M, rng), random_times(M, rng)
    kw = dict(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=objective, seed=d, storage=storage)
    a, b = nm.Netmax(**kw), nm.Netmax(**kw)
    a.async_begin(t, beta=0.7)
    b.async_begin(t, beta=0.7)
    before = a.kernel_launches
    a.async_steps(steps)
    launches = a.kernel_launches - before
    if M >= 100 and storage == "bf16":     # (so many bfloat16 rows cost more to bring in than the steps save)
        assert launches < steps // 4
    else:
        assert launches == -(-steps // 160), "the steps did not run on resident columns"
    for _ in range(steps):
        b.async_steps(1)
    assert (a.read_replicas().view(np.uint32) == b.read_replicas().view(np.uint32)).all()
    for p, q in zip(a.async_trace(), b.async_trace()):
        assert (p == q).all()
    a.close()
    b.close()
