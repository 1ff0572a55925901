"""GPU parity of the launch shape for small problems in which a warp holds all M rows of a few column groups and
others draw its noise and add up its telemetry (asserted per case): replicas and peer traces equal, bit for bit, those of one launch per round
(fuse_rounds = 1), telemetry to fp32 rounding (sums of at most 100 terms in fp32: 2e-5 relative)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# one column; one to eight rows per lane, the last one short or whole; 1 to 32 column groups per tile; tiles that do not
# fill the last CTA; the largest worker count, and sizes next to where the tiles of a whole CTA take over
SHAPES = [(2, 1), (2, 75_773), (3, 9), (4, 4096), (5, 8195), (8, 37_885), (13, 1111), (31, 5), (32, 591), (33, 6), (48, 4735),
          (64, 1181), (65, 130), (100, 67)]
NEXT_TO = [(8, 37_885)]  # these run on tiles


@pytest.fixture(scope="module")
def nm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2009_05766_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("storage,objective", [("f32", 1), ("f32", 0), ("bf16", 1)])
@pytest.mark.parametrize("M,d", SHAPES)
def test_small_problems_change_no_bit(nm, M, d, storage, objective):
    rng = np.random.default_rng(M * 7 + d)
    P = rng.random((M, M)) + 0.05
    P /= P.sum(axis=1, keepdims=True)
    kw = dict(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=objective, seed=d + M, trace_rounds=70,
              storage=storage, first_round=(1 << 32) - 40)  # (the high word of the round number changes on the way)
    plain, small = nm.Netmax(fuse_rounds=1, **kw), nm.Netmax(**kw)
    assert small.launch_shape(8)[0] == ("pipe" if (M, d) not in NEXT_TO else "tiles")
    for n in (4, 9, 33, 70, 8, 65):  # batches cut short, whole ones, more than a lap of the ring
        plain.round(n)
        small.round(n)
        assert (plain.read_replicas().view(np.uint32) == small.read_replicas().view(np.uint32)).all(), n
    first = plain.rounds_done - 70
    assert (plain.peer_trace(first, 70) == small.peer_trace(first, 70)).all()
    (ca, la), (cb, lb) = plain.telemetry(first, 70), small.telemetry(first, 70)
    np.testing.assert_allclose(cb, ca, rtol=2e-5)
    np.testing.assert_allclose(lb, la, rtol=2e-5)
    plain.close()
    small.close()
