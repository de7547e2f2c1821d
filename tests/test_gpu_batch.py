"""The batch forms (hashes sixteen to a warp, Sign in rounds) against the
oracle where they can go wrong: task counts around a hashing warp's sixteen,
messages around SHAKE256's 136-byte blocks (the 32-byte prefix included),
buffers at odd addresses, rejected tasks among valid ones, more tasks than
pairs of threads, the repetition cap inside a round, tasks that no round
settles, and a workspace of many small launches.  Every output is bytes or
whole numbers and must be equal."""
import numpy as np
import pytest

from paper_2211_12265_gb300 import workload as W

pytestmark = pytest.mark.gpu

LEVELS = (2, 3, 5)
# 32 + length around one, two and eight blocks, every length mod 4, empty
LENGTHS = [0, 1, 2, 3, 4, 99, 100, 101, 102, 103, 104, 105, 106, 107, 108, 136, 239, 240, 241, 242, 243, 1055, 1056, 1057]


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _at(torch, a, shift):
    """Device copy of a uint8 array whose first byte lies `shift` bytes past an aligned address."""
    buf = torch.zeros(a.size + 32, dtype=torch.uint8, device="cuda")
    out = buf[shift:shift + a.size].view(*a.shape)
    out.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return out


def _tasks(orc, level, n, seed):
    pk, sk = orc.keygen_batch(level, W.seeds(n, seed))
    lens = np.array([LENGTHS[(7 * i + n) % len(LENGTHS)] for i in range(n)], dtype=np.int64)
    msg, off = W.messages(lens, seed)
    return pk, sk, msg, off.astype(np.uint64)


@pytest.mark.parametrize("level", LEVELS)
@pytest.mark.parametrize("n,shift", [(1, 0), (15, 1), (16, 2), (17, 3), (40, 0)])
def test_counts_lengths_and_alignment(torch_cuda, orc, level, n, shift):
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    pk, sk, msg, off = _tasks(orc, level, n, 900 + n)
    osig, ost, oit = orc.sign_batch(level, sk, msg, off)
    bad = osig.copy()
    bad[::3, 5] ^= np.uint8(1)     # a bit of c~
    bad[1::3, 50] ^= np.uint8(4)   # a bit of z
    ook = orc.verify_batch(level, pk, msg, off, bad).astype(np.uint8)
    with dil.Context(0) as ctx:
        d_msg, d_off = _at(torch, msg, (shift + 1) % 4), dev(off)
        gpk, gsk = (_at(torch, np.zeros_like(a), shift) for a in (pk, sk))
        dil.dil_keygen(ctx.handle, level, n, _at(torch, W.seeds(n, 900 + n), shift), gpk, gsk)
        sig = _at(torch, np.full_like(osig, 0x5A), shift)
        st = torch.full((n,), 9, dtype=torch.int32, device="cuda")
        it = torch.zeros(n, dtype=torch.int32, device="cuda")
        dil.dil_sign_ex(ctx.handle, level, n, gsk, d_msg, d_off, sig, st, it)
        ok = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
        dil.dil_verify(ctx.handle, level, n, gpk, d_msg, d_off, _at(torch, bad, shift), ok)
        torch.cuda.synchronize()
        assert np.array_equal(host(gpk), pk) and np.array_equal(host(gsk), sk)
        assert np.array_equal(host(sig), osig) and np.array_equal(host(st), ost) and np.array_equal(host(it), oit)
        assert np.array_equal(host(ok), ook)


@pytest.mark.parametrize("level", LEVELS)
def test_rejected_tasks_among_valid_ones(torch_cuda, orc, level):
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    n, keys = 37, 5
    pk, sk = orc.keygen_batch(level, W.seeds(keys, 940))
    key = (np.arange(n) % keys).astype(np.int32)
    lens = np.full(n, 40, dtype=np.int64)
    msg, off = W.messages(lens, 940)
    off = off.astype(np.uint64)
    good = np.ones(n, dtype=bool)
    unknown = key.copy()
    unknown[[3, 20, 36]] = [-1, keys, 1 << 30]
    good[[3, 20, 36]] = False
    osig, ost, _ = orc.sign_batch(level, sk[key], msg, off)
    swapped = off.copy()   # task 8's offsets decrease, so task 7 takes 80 bytes
    swapped[8], swapped[9] = off[9], off[8]
    with dil.Context(0) as ctx:
        ks = dil.dil_keystore_create(ctx.handle, level, keys, dev(pk), dev(sk))
        sig = torch.full((n, osig.shape[1]), 0x5A, dtype=torch.uint8, device="cuda")
        st = torch.full((n,), 9, dtype=torch.int32, device="cuda")
        dil.dil_sign_keyed(ctx.handle, ks, n, dev(unknown), dev(msg), dev(off), sig, st)
        ok = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
        dil.dil_verify_keyed(ctx.handle, ks, n, dev(unknown), dev(msg), dev(off), dev(osig), ok)
        sig2, st2, it2 = ctx.sign(level, dev(sk[key]), dev(msg), dev(swapped), iterations=True)
        ok2 = ctx.verify(level, dev(pk[key]), dev(msg), dev(swapped), dev(osig))
        torch.cuda.synchronize()
        sig, st, ok, sig2, st2, it2, ok2 = (host(x) for x in (sig, st, ok, sig2, st2, it2, ok2))
        dil.dil_keystore_destroy(ks)
    assert np.array_equal(st, np.where(good, ost, dil.EINVAL)) and np.array_equal(ok, good.astype(np.uint8))
    assert np.array_equal(sig, np.where(good[:, None], osig, 0))
    rest = np.ones(n, dtype=bool)
    rest[[7, 8, 9]] = False
    assert st2[8] == dil.EINVAL and it2[8] == 0 and not sig2[8].any() and ok2[8] == 0
    assert (st2[[7, 9]] == 0).all() and not ok2[[7, 9]].any()
    assert np.array_equal(sig2[rest], osig[rest]) and (st2[rest] == 0).all() and ok2[rest].all()


@pytest.mark.parametrize("level,n", [(2, 9729), (2, 9800), (5, 4865), (3, 610)])
def test_more_tasks_than_a_first_share(torch_cuda, orc, level, n):
    """More tasks than the hashing warps start with (9,728) and than the attempts
    that fill the GPU: 40 distinct tasks, repeated."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    pk, sk, msg, off = _tasks(orc, level, 40, 960)
    osig, ost, oit = orc.sign_batch(level, sk, msg, off)
    pick = np.arange(n) % 40
    lens = (off[1:] - off[:-1])[pick]
    big_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    big_msg = np.concatenate([msg[off[i]:off[i + 1]] for i in pick] + [np.zeros(1, np.uint8)])
    bad = osig[pick]
    bad[::7, 60] ^= np.uint8(8)
    with dil.Context(0) as ctx:
        d_msg, d_off = dev(big_msg), dev(big_off)
        sig, st, it = ctx.sign(level, dev(sk[pick]), d_msg, d_off, iterations=True)
        ok = ctx.verify(level, dev(pk[pick]), d_msg, d_off, dev(bad))
        sig, st, it, ok = host(sig), host(st), host(it), host(ok)
    assert np.array_equal(sig, osig[pick]) and np.array_equal(st, ost[pick]) and np.array_equal(it, oit[pick])
    assert np.array_equal(ok, (np.arange(n) % 7 != 0).astype(np.uint8))


@pytest.mark.parametrize("level", LEVELS)
@pytest.mark.parametrize("cap", [1, 5, 33])
def test_repetition_cap_inside_a_round(torch_cuda, orc, level, cap):
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    n = 30
    _, sk, msg, off = _tasks(orc, level, n, 980)
    osig, ost, oit = orc.sign_batch(level, sk, msg, off, max_iter=cap)
    with dil.Context(0) as ctx:
        ctx.set_max_iter(cap)
        sig, st, it = (host(x) for x in ctx.sign(level, dev(sk), dev(msg), dev(off), iterations=True))
    assert np.array_equal(sig, osig) and np.array_equal(st, ost) and np.array_equal(it, oit)


def test_tasks_no_round_settles(torch_cuda, orc):
    """Tasks that need more repetitions than a lone task's rounds hold (32) end in
    the kernel behind the rounds."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    level, n = 3, 10000
    with dil.Context(0) as ctx:
        _, sk = ctx.keygen(level, dev(W.seeds(n, 990)))
        msg, off = W.messages(np.full(n, 32), 990)
        _, _, it = ctx.sign(level, sk, dev(msg), dev(off.astype(np.uint64)), iterations=True)
        late = np.nonzero(host(it) > 32)[0][:4]
        assert late.size, "10,000 tasks hold about nine such"
        for i in late:
            m = msg[off[i]:off[i + 1]]
            o = np.array([0, m.size], dtype=np.uint64)
            sig, st, it1 = (host(x) for x in ctx.sign(level, sk[int(i):int(i) + 1].contiguous(), dev(m), dev(o),
                                                      iterations=True))
            want = orc.sign_batch(level, host(sk[int(i)])[None], m, o)
            assert np.array_equal(sig, want[0]) and np.array_equal(st, want[1]) and np.array_equal(it1, want[2])


@pytest.mark.parametrize("level", LEVELS)
def test_small_workspaces(torch_cuda, orc, level):
    """Budgets from one fused task's scratch (the fused kernels run) to a few
    tasks of the batch forms a launch."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    n = 23
    pk, sk, msg, off = _tasks(orc, level, n, 995)
    osig, ost, oit = orc.sign_batch(level, sk, msg, off)
    k, l = {2: (4, 4), 3: (6, 5), 5: (8, 7)}[level]
    one = 1024 * (k * l + l + 2 * k + (l + 15) + l + k + l)
    for budget in (one, one + 4096, 2 * one, 5 * one):
        with dil.Context(0, workspace_budget=budget) as ctx:
            sig, st, it = (host(x) for x in ctx.sign(level, dev(sk), dev(msg), dev(off), iterations=True))
            ok = host(ctx.verify(level, dev(pk), dev(msg), dev(off), dev(osig)))
        assert np.array_equal(sig, osig) and np.array_equal(st, ost) and np.array_equal(it, oit), budget
        assert ok.all(), budget
    with dil.Context(0, workspace_budget=one - 1) as ctx:
        with pytest.raises(dil.DilError):
            ctx.sign(level, dev(sk), dev(msg), dev(off))
