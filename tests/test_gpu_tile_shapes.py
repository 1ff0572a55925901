"""Instances of the tile kernel made for one shape (40 to 1,280 workers, 32 to one column groups per tile), whole and short last
rows, a ragged last group: replicas bit for bit those of one launch per round, telemetry to 2e-5."""
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


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("M,d", [(40, 180_003), (39, 400_001), (54, 150_001), (64, 150_002), (57, 380_003), (80, 290_001), (150, 140_003),
                                 (313, 70_001), (637, 33_003), (1275, 16_001)])
def test_shapes_of_their_own_change_no_bit(nm, M, d, storage):
    P = np.full((M, M), 1.0 / M)
    kw = dict(M=M, d=d, lr=0.1, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=1, seed=M, trace_rounds=64, storage=storage)
    plain, tiles = nm.Netmax(fuse_rounds=1, **kw), nm.Netmax(**kw)
    for n in (9, 20):
        plain.round(n)
        tiles.round(n)
        assert (plain.read_replicas().view(np.uint32) == tiles.read_replicas().view(np.uint32)).all(), n
    (ca, la), (cb, lb) = plain.telemetry(0, 29), tiles.telemetry(0, 29)
    np.testing.assert_allclose(cb, ca, rtol=2e-5)
    np.testing.assert_allclose(lb, la, rtol=2e-5)
    plain.close()
    tiles.close()
