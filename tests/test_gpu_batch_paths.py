"""Paths of the batch forms that ordinary batches seldom or never take, against
the oracle: one test per way they have gone wrong or could."""
import numpy as np
import pytest

from paper_2211_12265_gb300 import workload as W

pytestmark = pytest.mark.gpu

LEVELS = (2, 3, 5)


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _inputs(orc, level, n, seed, lo=32, hi=32):
    pk, sk = orc.keygen_batch(level, W.seeds(n, seed))
    lens = W.message_lengths(n, seed, "uniform" if hi > lo else "fixed", lo, hi)
    msg, off = W.messages(lens, seed)
    return pk, sk, msg, off.astype(np.uint64)


@pytest.mark.parametrize("level", LEVELS)
def test_hash_whose_input_is_the_hash_before(torch_cuda, orc, level):
    """A pair of threads hashes tr and then H(tr || M), mu and then H(K || mu): each
    thread writes every other word of the first and fetches whole 8-byte units of
    it for the second.  609 tasks are the first batch on Verify's two-thread
    hashes; every mu and rho' is another one, and messages end anywhere in a
    block."""
    from gpu_util import gpu_sign, gpu_verify
    from paper_2211_12265_gb300 import dil
    n = 609
    pk, sk, msg, off = _inputs(orc, level, n, 1000 + level, 0, 400)
    osig, ost, oit = orc.sign_batch(level, sk, msg, off)
    with dil.Context(0) as ctx:
        sig, st, it = gpu_sign(ctx, level, sk, msg, off)
        ok = gpu_verify(ctx, level, pk, msg, off, osig)
    assert np.array_equal(sig, osig) and np.array_equal(st, ost) and np.array_equal(it, oit)
    assert ok.all()
