"""Instances of the tile kernel made for one shape (39 to 1,280 workers, 32 to one column groups per tile), whole and short last
rows, a ragged last group, across a change of the round number's high word: replicas bit for bit those of one launch per round, telemetry to
2e-5.  Cases with a shape are meant for its instance, and assert it."""
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
@pytest.mark.parametrize("M,d,shape", [(40, 500_003, (32, 10, 4)), (39, 500_001, (32, 10, 4)), (40, 180_003, None), (39, 400_001, None), (54, 150_001, (32, 7, 8)), (56, 150_001, (32, 7, 8)),
                                       (64, 150_002, (32, 8, 8)), (57, 380_003, None), (80, 290_001, (16, 10, 4)), (77, 290_001, (16, 10, 4)),
                                       (150, 140_003, (8, 10, 4)), (313, 70_001, (4, 10, 4)), (637, 33_003, (2, 10, 4)), (1275, 16_001, (1, 10, 4))])
def test_shapes_of_their_own_change_no_bit(nm, M, d, shape, storage):
    P = np.full((M, M), 1.0 / M)
    kw = dict(M=M, d=d, lr=0.1, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=1, seed=M, trace_rounds=64, storage=storage,
              first_round=(1 << 32) - 14)
    plain, tiles = nm.Netmax(fuse_rounds=1, **kw), nm.Netmax(**kw)
    kernel, groups, rows, warps, own = tiles.launch_shape(20)
    assert kernel == "tiles" and (shape is None or (own and (groups, rows, warps) == shape))
    for n in (9, 20):  # (the second call holds the change of the high word)
        plain.round(n)
        tiles.round(n)
        assert (plain.read_replicas().view(np.uint32) == tiles.read_replicas().view(np.uint32)).all(), n
    (ca, la), (cb, lb) = plain.telemetry((1 << 32) - 14, 29), tiles.telemetry((1 << 32) - 14, 29)
    np.testing.assert_allclose(cb, ca, rtol=2e-5)
    np.testing.assert_allclose(lb, la, rtol=2e-5)
    plain.close()
    tiles.close()
