"""Parts of the noise's first products that a launch works out once per column, round or row: fused rounds with and without the
rows' table (17 and 18 workers), across a change of the round number's high word, equal one launch per round bit for bit."""
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
@pytest.mark.parametrize("M,d", [(2, 620_001), (8, 310_003), (17, 303_106), (18, 303_109), (36, 303_111)])
def test_fused_rounds_across_the_high_word_change_no_bit(nm, M, d, storage):
    P = np.full((M, M), 1.0 / M)
    kw = dict(M=M, d=d, lr=0.1, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=1, seed=M, trace_rounds=64, storage=storage,
              first_round=(1 << 32) - 11)
    plain, fused = nm.Netmax(fuse_rounds=1, **kw), nm.Netmax(**kw)
    for n in (2, 5, 9, 20):      # launches of the instances for four, eight and more rounds; the third call holds the change
        before = fused.kernel_launches
        plain.round(n)
        fused.round(n)
        assert fused.kernel_launches - before < n + 1, "the rounds did not run several to a launch"
        assert (plain.read_replicas().view(np.uint32) == fused.read_replicas().view(np.uint32)).all(), n
    (ca, la), (cb, lb) = plain.telemetry((1 << 32) - 11, 36), fused.telemetry((1 << 32) - 11, 36)
    np.testing.assert_allclose(cb, ca, rtol=2e-5)
    np.testing.assert_allclose(lb, la, rtol=2e-5)
    plain.close()
    fused.close()
