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


# (tasks, lengths): the 25-lane hashes alone (up to 608 tasks), both forms (the line
# at 8,192 bytes and around it), and the two-thread form alone
SPLITS = [(3, [8191, 70000, 0]), (608, [40, 8192, 300]), (609, [8191, 8192, 8193, 32]), (1520, [0, 9000, 40, 16384]),
          (1521, [8192, 31]), (1824, [32, 12345]), (1825, [8192, 1])]
# few long messages of sixteen, or too many, around the lines of that rule
FEW, MANY = [9000] + [40] * 15, [8192] * 9 + [40] * 7
SPLITS += [(1217, MANY), (1825, FEW), (2400, MANY), (2433, FEW), (3072, MANY + FEW), (3073, FEW), (6144, FEW), (6145, FEW)]


@pytest.mark.parametrize("level", LEVELS)
@pytest.mark.parametrize("n,lengths", SPLITS)
def test_long_messages_beside_short_ones(torch_cuda, orc, level, n, lengths):
    """Every task is hashed once, by the form that its length and the batch's size
    give it, resident keys and rejected tasks among them."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    keys, m = 4, min(n, 24)   # m distinct tasks, repeated
    pk, sk = orc.keygen_batch(level, W.seeds(keys, 1010))
    lens = np.array([lengths[i % len(lengths)] for i in range(m)], dtype=np.int64)
    msg, off = W.messages(lens, 1010 + n)
    key = (np.arange(m) % keys).astype(np.int32)
    osig, ost, oit = orc.sign_batch(level, sk[key], msg, off.astype(np.uint64))
    pick = np.arange(n) % m
    big = np.concatenate([msg[off[i]:off[i + 1]] for i in pick] + [np.zeros(1, np.uint8)])
    big_off = np.concatenate([[0], np.cumsum(lens[pick])]).astype(np.uint64)
    key = key[pick]
    unknown = np.arange(n) % 11 == 10   # of resident keys
    bad = osig[pick]
    bad[::5, 40] ^= np.uint8(2)
    with dil.Context(0) as ctx:
        d_msg, d_off = dev(big), dev(big_off)
        sig, st, it = (host(x) for x in ctx.sign(level, dev(sk[key]), d_msg, d_off, iterations=True))
        ok = host(ctx.verify(level, dev(pk[key]), d_msg, d_off, dev(bad)))
        ks = dil.dil_keystore_create(ctx.handle, level, keys, dev(pk), dev(sk))
        d_key = dev(np.where(unknown, keys, key).astype(np.int32))
        ksig = torch.full((n, osig.shape[1]), 0x5A, dtype=torch.uint8, device="cuda")
        kst = torch.full((n,), 9, dtype=torch.int32, device="cuda")
        kok = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
        dil.dil_sign_keyed(ctx.handle, ks, n, d_key, d_msg, d_off, ksig, kst)
        dil.dil_verify_keyed(ctx.handle, ks, n, d_key, d_msg, d_off, dev(bad), kok)
        ksig, kst, kok = host(ksig), host(kst), host(kok)
        dil.dil_keystore_destroy(ks)
    want_ok = np.arange(n) % 5 != 0
    assert np.array_equal(sig, osig[pick]) and np.array_equal(st, ost[pick]) and np.array_equal(it, oit[pick])
    assert np.array_equal(ok, want_ok.astype(np.uint8))
    assert np.array_equal(ksig, np.where(unknown[:, None], 0, osig[pick]))
    assert np.array_equal(kst, np.where(unknown, dil.EINVAL, ost[pick]))
    assert np.array_equal(kok, (want_ok & ~unknown).astype(np.uint8))


@pytest.mark.parametrize("n", [1, 400])
def test_long_messages_end_with_the_25_lane_chain(torch_cuda, n):
    """The hash of one long message is what such a call waits for: 24 rounds a
    block at about 224 clocks each for a warp on the 25-lane form, 250 and the
    absorbing for two threads to a state (1.43 times as long, measured).  The
    bound is the fused kernel's time, which hashes that way, and a fifth."""
    import time
    from gpu_util import dev
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    size = 1 << 18
    msg = torch.randint(0, 256, (size + 32 * n,), dtype=torch.uint8, device="cuda")
    off = np.concatenate([[0], size + 32 * np.arange(n, dtype=np.uint64)]).astype(np.uint64)
    took = {}
    for shape in (None, (8, 2)):
        with dil.Context(0) as ctx:
            if shape:
                ctx.set_tuning(1, shape[0], shape[1], 2)
            _, sk = ctx.keygen(2, dev(W.seeds(n, 1030)))
            d_off = dev(off)
            ts = []
            for _ in range(4):
                torch.cuda.synchronize()
                t = time.perf_counter()
                ctx.sign(2, sk, msg, d_off)
                torch.cuda.synchronize()
                ts.append(time.perf_counter() - t)
            took[shape] = min(ts)
    assert took[None] < 1.2 * took[(8, 2)], took


@pytest.mark.parametrize("n", [2048, 2500])
def test_keygen_does_not_slow_down_in_parts(torch_cuda, n):
    """2,047 Dilithium3 keys take 236 us; in two halves beside each other 2,048 and
    2,500 took 411 and 436.  The bound is the ratio of the counts and a quarter."""
    from gpu_util import dev
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda

    def took(m):
        seeds = dev(W.seeds(m, 1040))
        pk, sk = ctx.keygen(3, seeds)
        ts = []
        for _ in range(9):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            for _ in range(4):
                dil.dil_keygen(ctx.handle, 3, m, seeds, pk, sk)
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1) / 4)
        return sorted(ts)[4]

    with dil.Context(0) as ctx:
        fewer, more = took(2047), took(n)
    assert more < 1.25 * n / 2047 * fewer, (fewer, more)


@pytest.mark.parametrize("level,n", [(2, 5001), (3, 9001)])
def test_keygen_in_parts(torch_cuda, level, n):
    """An odd batch on two streams equals its two halves, made one by one."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    seeds = W.seeds(n, 1050)
    with dil.Context(0) as ctx:
        pk, sk = (host(x) for x in ctx.keygen(level, dev(seeds)))
        for part in (slice(0, 2000), slice(2000, 4500), slice(4500, n)):
            for got, want in zip((pk, sk), ctx.keygen(level, dev(seeds[part]))):
                assert np.array_equal(got[part], host(want))


@pytest.mark.parametrize("level", LEVELS)
@pytest.mark.parametrize("n", [5, 608, 609, 1216, 1217])
def test_rows_on_four_warps(torch_cuda, orc, level, n):
    """Signatures spoiled where one warp of a task's four sees it (each z
    polynomial, the hint, c~) or all do, on both sides of the lines between one and
    four warps; plain and with resident keys."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    k, l, zbits = {2: (4, 4, 18), 3: (6, 5, 20), 5: (8, 7, 20)}[level]
    m = l + 4
    pk, sk, msg, off = _inputs(orc, level, m, 1060, 0, 300)
    good, _, _ = orc.sign_batch(level, sk, msg, off)
    bad = good.copy()
    for j in range(l):                              # z_j's last coefficient out of range
        bad[j, 32 + 32 * zbits * (j + 1) - 2:32 + 32 * zbits * (j + 1)] = 0
    bad[l, -1] = 255                                # hint counts
    bad[l + 1, -k - 1] ^= np.uint8(1)               # unused hint byte, or its order
    bad[l + 2, 3] ^= np.uint8(64)                   # c~
    bad[l + 3, 40] ^= np.uint8(1)                   # z within its range
    assert not orc.verify_batch(level, pk, msg, off, bad).any()
    pick = np.arange(n) % m
    spoil = np.arange(n) % 3 != 0
    sig = np.where(spoil[:, None], bad[pick], good[pick])
    big = np.concatenate([msg[off[i]:off[i + 1]] for i in pick] + [np.zeros(1, np.uint8)])
    big_off = np.concatenate([[0], np.cumsum((off[1:] - off[:-1])[pick])]).astype(np.uint64)
    with dil.Context(0) as ctx:
        d_msg, d_off, d_sig = dev(big), dev(big_off), dev(sig)
        ok = host(ctx.verify(level, dev(pk[pick]), d_msg, d_off, d_sig))
        ks = dil.dil_keystore_create(ctx.handle, level, m, dev(pk))
        kok = dev(np.full(n, 7, np.uint8))
        dil.dil_verify_keyed(ctx.handle, ks, n, dev(pick.astype(np.int32)), d_msg, d_off, d_sig, kok)
        kok = host(kok)
        dil.dil_keystore_destroy(ks)
    assert np.array_equal(ok, (~spoil).astype(np.uint8)) and np.array_equal(kok, ok)


def test_keyed_verify_of_short_messages_is_no_slower_than_fused(torch_cuda):
    """A few checks of short messages against resident keys: the fused kernel that
    two warps per task select bounds the call's time, a twentieth to spare."""
    from gpu_util import dev
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    n = 13
    took = {}
    for shape in (None, (8, 2)):
        with dil.Context(0) as ctx:
            if shape:
                ctx.set_tuning(2, shape[0], shape[1], 5)
            pk, sk = ctx.keygen(5, dev(W.seeds(n, 1070)))
            msg, off = W.messages(np.full(n, 32), 1070)
            d_msg, d_off = dev(msg), dev(off.astype(np.uint64))
            sig, _ = ctx.sign(5, sk, d_msg, d_off)
            ks = dil.dil_keystore_create(ctx.handle, 5, n, pk)
            key, ok = dev(np.arange(n, dtype=np.int32)), dev(np.zeros(n, np.uint8))
            ts = []
            for _ in range(9):
                e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                e0.record()
                for _ in range(8):
                    dil.dil_verify_keyed(ctx.handle, ks, n, key, d_msg, d_off, sig, ok)
                e1.record()
                torch.cuda.synchronize()
                ts.append(e0.elapsed_time(e1) / 8)
            took[shape] = sorted(ts)[4]
            dil.dil_keystore_destroy(ks)
    assert took[None] < 1.05 * took[(8, 2)], took


def _stubborn_keys(orc, level, n, seed):
    """Secret keys whose t0 has only the two extreme values: the hint has too many
    ones in all but about one repetition of a thousand (Dilithium2)."""
    pk, sk = orc.keygen_batch(level, W.seeds(n, seed))
    k = {2: 4, 3: 6, 5: 8}[level]
    fields = np.random.default_rng(seed).integers(0, 2, (n, 256 * k, 1), dtype=np.uint8)
    sk[:, -416 * k:] = np.packbits(np.broadcast_to(fields, (n, 256 * k, 13)).reshape(n, -1), axis=1, bitorder="little")
    return sk


def test_many_tasks_that_no_round_settles(torch_cuda, orc):
    """A batch whose keys (damaged ones) almost never accept is signed by the loop
    behind the rounds, on as many warps as the GPU holds: eleven times
    the tasks of a batch that leaves most of it idle take less than four times as
    long (the rounds before it included)."""
    import time
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    m, cap = 8, 400
    sk = _stubborn_keys(orc, 2, m, 1080)
    msg, off = W.messages(np.full(m, 32), 1080)
    osig, ost, oit = orc.sign_batch(2, sk, msg, off.astype(np.uint64), max_iter=cap)
    assert (ost == dil.EITER).sum() > m // 2
    took = {}
    with dil.Context(0) as ctx:
        ctx.set_max_iter(cap)
        for n in (64, 704):
            pick = np.arange(n) % m
            d_sk, d_off = dev(sk[pick]), dev((np.arange(n + 1) * 32).astype(np.uint64))
            d_msg = dev(np.concatenate([msg[off[i]:off[i + 1]] for i in pick]))
            ts = []
            for _ in range(3):
                torch.cuda.synchronize()
                t = time.perf_counter()
                sig, st, it = ctx.sign(2, d_sk, d_msg, d_off, iterations=True)
                torch.cuda.synchronize()
                ts.append(time.perf_counter() - t)
            took[n] = min(ts)
            assert np.array_equal(host(st), ost[pick]) and np.array_equal(host(it), oit[pick])
            assert np.array_equal(host(sig), osig[pick])
    assert took[704] < 4 * took[64], took


@pytest.mark.parametrize("level", LEVELS)
def test_leftover_tasks_of_a_batch(torch_cuda, orc, level):
    """The loop behind the rounds on several tasks at a time, resident keys and a
    workspace of few slots included."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    n, cap = 21, 90
    sk = _stubborn_keys(orc, level, n, 1090)
    pk, _ = orc.keygen_batch(level, W.seeds(n, 1090))
    msg, off = W.messages(np.full(n, 50), 1090)
    off = off.astype(np.uint64)
    osig, ost, oit = orc.sign_batch(level, sk, msg, off, max_iter=cap)
    for budget in (0, 6 << 20):
        with dil.Context(0, workspace_budget=budget) as ctx:
            ctx.set_max_iter(cap)
            sig, st, it = (host(x) for x in ctx.sign(level, dev(sk), dev(msg), dev(off), iterations=True))
            ks = dil.dil_keystore_create(ctx.handle, level, n, dev(pk), dev(sk))
            ksig, kst = torch.zeros_like(dev(osig)), dev(np.full(n, 9, np.int32))
            dil.dil_sign_keyed(ctx.handle, ks, n, dev(np.arange(n, dtype=np.int32)), dev(msg), dev(off), ksig, kst)
            ksig, kst = host(ksig), host(kst)
            dil.dil_keystore_destroy(ks)
        assert np.array_equal(sig, osig) and np.array_equal(st, ost) and np.array_equal(it, oit)
        assert np.array_equal(ksig, osig) and np.array_equal(kst, ost)


def _persistent(torch, dil, ctx, jobs):
    """One persistent launch of (level, sk, msg, off) jobs on the device: per job
    signatures, statuses and repetitions."""
    outs, descs = [], []
    for level, sk, msg, off in jobs:
        n = sk.shape[0]
        o = (torch.full((n, dil.SIZES[level][2]), 0x5A, dtype=torch.uint8, device="cuda"),
             torch.full((n,), 9, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"))
        outs.append(o)
        descs.append(dil.sign_job(level, n, sk, msg, off, *o))
    dil.dil_sign_persistent(ctx.handle, descs)
    assert dil.dil_persistent_status(ctx.handle) == dil.OK
    return [tuple(x.cpu().numpy() for x in o) for o in outs]


def test_persistent_launch_where_memory_is_short(torch_cuda):
    """A device that refuses the rounds' workspace: smaller parts, then the device
    queue, then smaller parts still, and DIL_ENOMEM only where nothing fits; the
    context is usable throughout and outputs are the same."""
    from gpu_util import dev
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    jobs, want = [], []
    with dil.Context(0) as ctx:
        for level, n in ((2, 5000), (5, 3001)):
            _, sk = ctx.keygen(level, dev(W.seeds(n, 1100 + level)))
            msg, off = W.messages(np.full(n, 32), 1100 + level)
            jobs.append((level, sk, dev(msg), dev(off.astype(np.uint64))))
            want.append([x.cpu().numpy() for x in ctx.sign(*jobs[-1], iterations=True)])
    mib = 1 << 20
    # rounds take 388 MiB (both jobs), and 194, 97, 48 ...; the queue in this shape 74
    for limit in (700 * mib, 250 * mib, 100 * mib, 80 * mib, 60 * mib, 10 * mib):
        with dil.Context(0) as ctx:
            dil.dil_set_persistent_tuning(ctx.handle, 4, 1, 1, 1, 4)
            dil.dil_test_set_alloc_limit(ctx.handle, limit)
            for part in (jobs[:1], jobs, jobs[:1]):   # a larger workspace, refused; argument sets in turn
                got = _persistent(torch, dil, ctx, part)
                for g, w in zip(got, want):
                    assert all(np.array_equal(a, b) for a, b in zip(g, w)), limit
    with dil.Context(0) as ctx:
        dil.dil_test_set_alloc_limit(ctx.handle, 1)
        with pytest.raises(dil.DilError) as e:
            _persistent(torch, dil, ctx, jobs)
        assert str(dil.ENOMEM) in str(e.value)
        dil.dil_test_set_alloc_limit(ctx.handle, 0)
        got = _persistent(torch, dil, ctx, jobs)
        for g, w in zip(got, want):
            assert all(np.array_equal(a, b) for a, b in zip(g, w))


def test_cancel_ends_a_launch_in_rounds_soon(torch_cuda):
    """Once the cancel word is written the parts in flight end with their round and
    no later one samples or transforms anything: the launch ends in a quarter of its
    time (a third before it did so).  Every task is either signed as before, with
    the repetition it would have had, or canceled, wherever the word finds it."""
    import time
    from gpu_util import dev
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    n = 600_000   # about 38 parts of 16,384 tasks
    whole, rest, hits = [], [], 0
    with dil.Context(0) as ctx:
        _, sk = ctx.keygen(2, dev(W.seeds(n, 1110)))
        msg, off = W.messages(np.full(n, 32), 1110)
        d_msg, d_off = dev(msg), dev(off.astype(np.uint64))
        sig = torch.zeros((n, dil.SIZES[2][2]), dtype=torch.uint8, device="cuda")
        st = torch.zeros(n, dtype=torch.int32, device="cuda")
        it = torch.zeros(n, dtype=torch.int32, device="cuda")
        job = [dil.sign_job(2, n, sk, d_msg, d_off, sig, st, it)]
        for _ in range(3):
            t = time.perf_counter()
            dil.dil_sign_persistent(ctx.handle, job)
            assert dil.dil_persistent_status(ctx.handle) == dil.OK
            whole.append(time.perf_counter() - t)
        want_sig, want_it = sig.clone(), it.clone()
        dil.dil_persistent_cancel(ctx.handle)   # its stream exists from here on
        for k in range(40):
            sig.fill_(0x5A)
            st.fill_(9)
            it.fill_(7)
            torch.cuda.synchronize()
            dil.dil_sign_persistent(ctx.handle, job)
            time.sleep(0.001 * (3 + k))
            dil.dil_persistent_cancel(ctx.handle)
            t = time.perf_counter()
            status = dil.dil_persistent_status(ctx.handle)
            t = time.perf_counter() - t
            ok, gone = st == dil.OK, st == dil.ECANCELED
            assert bool((ok | gone).all())
            assert status == dil.ECANCELED or not bool(gone.any())
            if bool(gone.any()):   # not where the host came before the launch, or after it
                hits += 1
                if k < 8:
                    rest.append(t)
            assert torch.equal(sig[ok], want_sig[ok]) and torch.equal(it[ok], want_it[ok])
            assert not bool(sig[gone].any()) and not bool(it[gone].any())
    assert hits > 10 and min(rest) < min(whole) / 4, (hits, rest, whole)


# Seeds (a number's four bytes eight times) of Dilithium3 keys with a polynomial
# that ExpandS's first two blocks do not fill: (number, polynomial, coefficients
# they hold)
THIRD_BLOCK = [(327, 0, 251), (46958, 1, 255), (54815, 10, 255), (65704, 10, 252)]


@pytest.mark.parametrize("n", [4, 17, 40, 700])
def test_secret_polynomials_that_need_a_third_block(torch_cuda, orc, n):
    """One key in about ten thousand has such a polynomial; here several of a batch
    have, first, last and in the middle of the sixteen that a warp samples."""
    import hashlib
    from gpu_util import gpu_keygen
    from paper_2211_12265_gb300 import dil
    seeds = W.seeds(n, 1120)
    at = [0, n // 2, n - 2, n - 1]
    for (number, poly, held), i in zip(THIRD_BLOCK, at):
        zeta = number.to_bytes(4, "little") * 8
        blocks = hashlib.shake_256(hashlib.shake_256(zeta).digest(128)[32:96] + bytes([poly, 0])).digest(272)
        assert sum((b & 15) < 9 for b in blocks) + sum(b >> 4 < 9 for b in blocks) == held < 256
        seeds[i] = np.frombuffer(zeta, np.uint8)
    opk, osk = orc.keygen_batch(3, seeds)
    with dil.Context(0) as ctx:
        pk, sk = gpu_keygen(ctx, 3, seeds)
    assert np.array_equal(pk, opk) and np.array_equal(sk, osk)


@pytest.mark.parametrize("level", LEVELS)
@pytest.mark.parametrize("n", [1, 5])
def test_expand_a_samples_unfilled_polynomials_again(torch_cuda, level, n):
    """The five blocks that ExpandA takes of a stream fall short with a probability
    below 1e-30; with four every polynomial does."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    k, l = {2: (4, 4), 3: (6, 5), 5: (8, 7)}[level]
    rho = dev(W.seeds(n, 1130))
    c = np.arange(256)
    word = ((c & 4) << 5) + ((c >> 3) << 2) + (c & 3)   # of coefficient c in lane order
    with dil.Context(0) as ctx:
        want, got, lanes = (torch_cuda.zeros((n, k * l, 256), dtype=torch_cuda.int32, device="cuda") for _ in range(3))
        dil.dil_expand_a(ctx.handle, level, n, rho, 32, want)
        dil.dil_test_expand_a_refill(ctx.handle, level, n, rho, False, got)
        dil.dil_test_expand_a_refill(ctx.handle, level, n, rho, True, lanes)
        want, got, lanes = host(want), host(got), host(lanes)
    assert np.array_equal(got, want) and np.array_equal(lanes[:, :, word], want)


def _jobs(torch, dil, spec):
    """(level, n, lo, hi) jobs on the device and their signatures by dil_sign."""
    from gpu_util import dev
    jobs, want = [], []
    with dil.Context(0) as ctx:
        for level, n, lo, hi in spec:
            _, sk = ctx.keygen(level, dev(W.seeds(max(n, 1), 1140 + level)))
            lens = W.message_lengths(max(n, 1), 1140, "uniform" if hi > lo else "fixed", lo, hi)
            msg, off = W.messages(lens, 1140 + level)
            jobs.append((level, sk[:n], dev(msg), dev(off.astype(np.uint64)[:n + 1])))
            want.append([x.cpu().numpy() for x in ctx.sign(*jobs[-1], iterations=True)] if n else None)
    return jobs, want


@pytest.mark.parametrize("shape", [None, (8, 2, 0, 1, 4), (8, 4, 0, 2, 8), (8, 1, 0, 1, 8)])
def test_mixed_empty_and_changing_jobs_in_either_form(torch_cuda, shape):
    """Persistent launches of three levels, with an empty job among others, and of
    argument sets in turn, in rounds (no shape, or one warp per task) and on the
    device queue."""
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    jobs, want = _jobs(torch, dil, [(2, 300, 0, 1500), (5, 211, 0, 4096), (3, 97, 32, 64), (5, 0, 0, 0)])
    with dil.Context(0) as ctx:
        if shape:
            dil.dil_set_persistent_tuning(ctx.handle, *shape)
        for pick in ([0, 1, 2], [0, 3, 2], [1], [0, 1, 2], [2, 0]):
            for g, i in zip(_persistent(torch, dil, ctx, [jobs[i] for i in pick]), pick):
                if want[i] is not None:
                    assert all(np.array_equal(a, b) for a, b in zip(g, want[i])), (pick, i)


def test_one_warp_queue_on_a_refused_workspace(torch_cuda):
    """The one-warp queue at its full size, speculation included, where the rounds'
    workspace is refused: a limit that the queue's fits exactly."""
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    jobs, want = _jobs(torch, dil, [(5, 12000, 32, 32)])
    with dil.Context(0) as ctx:
        dil.dil_set_persistent_tuning(ctx.handle, 8, 1, 2, 1, 8)
        # rounds: 4 x 3,000 tasks of 79 KiB and more, halved; queue: 152 x 2 x 8 workers of 124 KiB
        dil.dil_test_set_alloc_limit(ctx.handle, 310 << 20)
        (got,) = _persistent(torch, dil, ctx, jobs)
    assert all(np.array_equal(a, b) for a, b in zip(got, want[0]))


def test_cancel_on_the_device_queue(torch_cuda):
    import time
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    n = 200_000
    jobs, want = _jobs(torch, dil, [(2, n, 32, 32)])
    level, sk, msg, off = jobs[0]
    with dil.Context(0) as ctx:
        dil.dil_set_persistent_tuning(ctx.handle, 8, 2, 0, 1, 4)
        sig = torch.full((n, dil.SIZES[2][2]), 0x5A, dtype=torch.uint8, device="cuda")
        st = torch.full((n,), 9, dtype=torch.int32, device="cuda")
        it = torch.full((n,), 7, dtype=torch.int32, device="cuda")
        dil.dil_sign_persistent(ctx.handle, [dil.sign_job(2, n, sk, msg, off, sig, st, it)])
        time.sleep(0.01)
        dil.dil_persistent_cancel(ctx.handle)
        assert dil.dil_persistent_status(ctx.handle) == dil.ECANCELED
        s, g, i = st.cpu().numpy(), sig.cpu().numpy(), it.cpu().numpy()
        ok, gone = s == dil.OK, s == dil.ECANCELED
        assert (ok | gone).all() and ok.any() and gone.any()
        assert not g[gone].any() and not i[gone].any()
        assert np.array_equal(g[ok], want[0][0][ok]) and np.array_equal(i[ok], want[0][2][ok])
        (got,) = _persistent(torch, dil, ctx, jobs)   # the next launch starts with the word cleared
    assert all(np.array_equal(a, b) for a, b in zip(got, want[0]))


# Task counts of one stream and of several, with the hashes on a stream of their own
FORKED = [(2, 40), (2, 5200), (3, 2300), (5, 700)]


def _calls(torch, dil, ctx, level, n):
    """Inputs (their true values, and buffers to fill), outputs and the calls of
    every device form of one batch."""
    from gpu_util import dev
    seeds = dev(W.seeds(n, 1150 + level))
    msg, off = W.messages(W.message_lengths(n, 1150, "uniform", 0, 300), 1150)
    msg, off = dev(msg), dev(off.astype(np.uint64))
    pk, sk = ctx.keygen(level, seeds)
    sig, st = ctx.sign(level, sk, msg, off)
    bad = sig.clone()
    bad[::3, 40] ^= 2
    key = torch.arange(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    true = dict(seeds=seeds, pk=pk, sk=sk, msg=msg, off=off.view(torch.int64), sig=bad, key=key)
    x = {k: torch.zeros_like(v) for k, v in true.items()}
    o = dict(pk=torch.zeros_like(pk), sk=torch.zeros_like(sk), sig=torch.zeros_like(sig), st=torch.full_like(st, 9),
             ok=torch.full((n,), 7, dtype=torch.uint8, device="cuda"), ksig=torch.zeros_like(sig),
             kst=torch.full_like(st, 9), kok=torch.full((n,), 7, dtype=torch.uint8, device="cuda"))
    ks = dil.dil_keystore_create(ctx.handle, level, n, pk, sk)
    want_ok = torch.ones(n, dtype=torch.uint8, device="cuda")
    want_ok[::3] = 0
    want = dict(pk=pk, sk=sk, sig=sig, st=st, ok=want_ok, ksig=sig, kst=st, kok=want_ok)

    def run(stream):
        h = ctx.handle
        dil.dil_keygen(h, level, n, x["seeds"], o["pk"], o["sk"], stream)
        dil.dil_sign(h, level, n, x["sk"], x["msg"], x["off"], o["sig"], o["st"], stream)
        dil.dil_verify(h, level, n, x["pk"], x["msg"], x["off"], x["sig"], o["ok"], stream)
        dil.dil_sign_keyed(h, ks, n, x["key"], x["msg"], x["off"], o["ksig"], o["kst"], stream)
        dil.dil_verify_keyed(h, ks, n, x["key"], x["msg"], x["off"], x["sig"], o["kok"], stream)
    return true, x, o, want, run, ks


@pytest.mark.parametrize("level,n", FORKED)
def test_forked_forms_keep_a_callers_stream_in_order(torch_cuda, level, n):
    """Inputs that the caller's own stream fills in late, outputs that it copies
    and overwrites at once: the context's other streams start and end within the
    caller's."""
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    with dil.Context(0) as ctx:
        true, x, o, want, run, ks = _calls(torch, dil, ctx, level, n)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(3):
                for k in x:
                    x[k].zero_()
                torch.cuda._sleep(2_000_000)   # about a millisecond
                for k in x:
                    x[k].copy_(true[k])
                run(s)
                copies = {k: v.clone() for k, v in o.items()}
                for k in x:
                    x[k].fill_(1)
                for v in o.values():
                    v.fill_(3)
        s.synchronize()
        dil.dil_keystore_destroy(ks)
    for k, v in copies.items():
        assert torch.equal(v, want[k]), k
    assert all(bool((v == 3).all()) for v in o.values())


@pytest.mark.parametrize("level,n", FORKED)
def test_forked_forms_under_the_callers_capture(torch_cuda, level, n):
    """Every device form in a graph of the caller's, replayed on other inputs, with
    direct calls in between."""
    from paper_2211_12265_gb300 import dil
    torch = torch_cuda
    with dil.Context(0) as ctx:
        true, x, o, want, run, ks = _calls(torch, dil, ctx, level, n)
        for k in x:
            x[k].copy_(true[k])
        run(torch.cuda.current_stream())   # the workspace is there before the capture
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run(torch.cuda.current_stream())
        for k in x:
            x[k].zero_()
        for _ in range(2):
            for v in o.values():
                v.fill_(3)
            for k in x:
                x[k].copy_(true[k])
            graph.replay()
            torch.cuda.synchronize()
            for k, v in o.items():
                assert torch.equal(v, want[k]), k
            run(torch.cuda.current_stream())
        torch.cuda.synchronize()
        for k, v in o.items():
            assert torch.equal(v, want[k]), k
        del graph
        dil.dil_keystore_destroy(ks)


@pytest.mark.parametrize("level", LEVELS)
def test_keygen_and_verify_in_small_workspaces(torch_cuda, orc, level):
    """Budgets of one task's scratch and a few tasks' a launch; below one task's
    the call is refused, whatever the shape."""
    from gpu_util import dev, host
    from paper_2211_12265_gb300 import dil
    k, l = {2: (4, 4), 3: (6, 5), 5: (8, 7)}[level]
    n = 23
    pk, sk, msg, off = _inputs(orc, level, n, 1160, 0, 300)
    sig, _, _ = orc.sign_batch(level, sk, msg, off)
    gen, ver = 1024 * (l + k * l + l + k), 1024 * (1 + k * l) + 384
    for budget in (gen, gen + 500, 5 * gen):
        with dil.Context(0, workspace_budget=budget) as ctx:
            gpk, gsk = ctx.keygen(level, dev(W.seeds(n, 1160)))
            assert np.array_equal(host(gpk), pk) and np.array_equal(host(gsk), sk)
    for budget in (ver, ver + 500, 5 * ver):
        with dil.Context(0, workspace_budget=budget) as ctx:
            assert host(ctx.verify(level, dev(pk), dev(msg), dev(off), dev(sig))).all()
    for shape in (None, (8, 1), (8, 2), (4, 4)):
        with dil.Context(0, workspace_budget=gen - 1) as c0, dil.Context(0, workspace_budget=ver - 1) as c2:
            for ctx, op in ((c0, 0), (c2, 2)):
                if shape:
                    ctx.set_tuning(op, shape[0], shape[1], level)
            with pytest.raises(dil.DilError):
                c0.keygen(level, dev(W.seeds(n, 1160)))
            with pytest.raises(dil.DilError):
                c2.verify(level, dev(pk), dev(msg), dev(off), dev(sig))
