"""Telemetry of small problems, run many rounds to a launch, against 64-bit sums of the replicas that it describes.  At most
eight rows of a column are added in fp32: rounding errors of such sums are independent from column to column and from eight rows to the
next, so that hundreds of them average out far below one fp32 rounding, 2^-24, which is what 1/M costs.  (One fp32 chain over all rows is
six times that for 100 workers in bfloat16.)"""
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


@pytest.mark.parametrize("M,d,storage", [(100, 400, "bf16"), (64, 401, "bf16"), (100, 1310, "f32"), (72, 1823, "f32"), (48, 2731, "f32"), (9, 7281, "f32"),
                                         (17, 3333, "bf16")])
def test_sums_of_small_problems_are_as_exact_as_one_rounding(nm, M, d, storage):
    n = 24
    rng = np.random.default_rng(M + d)
    P = rng.random((M, M)) + 0.05
    P /= P.sum(axis=1, keepdims=True)
    kw = dict(M=M, d=d, lr=0.05, prob=P, sigma=0.1, x0_std=1.0, c_std=1.0, objective=1, seed=d + M, trace_rounds=32, storage=storage)
    plain, small = nm.Netmax(fuse_rounds=1, **kw), nm.Netmax(**kw)
    c = plain.read_centres().astype(np.float64)
    want = np.empty((2, n))
    for k in range(n):
        x = plain.read_replicas().astype(np.float64)
        want[:, k] = ((x - x.mean(axis=0)) ** 2).sum() / M, 0.5 * ((x - c) ** 2).sum() / M
        plain.round(1)
    small.round(n)
    error = np.sqrt(((np.array(small.telemetry(0, n)) / want - 1.0) ** 2).mean(axis=1))
    assert (error < 2.0 ** -24).all(), error
    plain.close()
    small.close()
