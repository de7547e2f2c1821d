"""Workloads of the batched Dilithium engine, each one call a user makes.

The sizes are those of the benchmark (`bench.py`: 10,000 tasks per batch,
32-byte or 32 B - 4 KB messages, a mixed-level persistent launch, the served
mix), of the tests (single calls, a few hundred tasks) and odd counts between
them.  ``tuned`` contexts install the committed launch shapes
(``Context.apply_tuning``, as the benchmark does); the others are created the
way the README shows, with no tuning call.

Every output is bytes or whole numbers (keys, signatures, statuses, accept
bits), so there is no rounding to compare: ``exact`` has no values.
"""
import math

import numpy as np
import torch

from paper_2211_12265_gb300 import dil, serving
from paper_2211_12265_gb300 import work as WK

PARAMS = {2: (4, 4), 3: (6, 5), 5: (8, 7)}


def listed():
    return [
        # one signature per call, or the few checks of one document: a service
        # that answers as requests come in; latency and launch cost are all
        # there is
        dict(name="sign2_one", kind="sign", level=2, n=1, lo=32, hi=32, dist="fixed", tuned=False),
        dict(name="verify3_13", kind="verify", level=3, n=13, lo=1000, hi=1000, dist="fixed", tuned=False),
        # a batch too small to fill the GPU, ragged messages, no tuning call
        dict(name="sign5_150", kind="sign", level=5, n=150, lo=32, hi=4096, dist="uniform", tuned=False),
        # key provisioning
        dict(name="keygen2_10k", kind="keygen", level=2, n=10000, tuned=True),
        # the headline batch: 10,000 Dilithium2 tasks on 32-byte messages
        dict(name="sign2_10k", kind="sign", level=2, n=10000, lo=32, hi=32, dist="fixed", tuned=True),
        dict(name="verify2_10k", kind="verify", level=2, n=10000, lo=32, hi=32, dist="fixed", tuned=True),
        # the higher levels on messages of 32 B - 4 KB
        dict(name="sign3_10k", kind="sign", level=3, n=10000, lo=32, hi=4096, dist="uniform", tuned=True),
        dict(name="verify5_10k", kind="verify", level=5, n=10000, lo=32, hi=4096, dist="uniform", tuned=True),
        # two levels in one persistent launch
        dict(name="persist25_40k", kind="persistent", levels="25", n=40000, lo=32, hi=32, dist="fixed", tuned=True),
        # checks against resident keys, an odd count, long-tailed messages
        dict(name="keyed_verify3_8191", kind="keyed_verify", level=3, n=8191, keys=1024, lo=32, hi=16384,
             dist="loguniform", tuned=True),
        # batch in host memory, copies inside the call
        dict(name="host_sign2_10k", kind="host_sign", level=2, n=10000, lo=32, hi=32, dist="fixed", tuned=True),
        # a burst of the served mix (60% verify, all levels) through the server
        dict(name="serve_20k", kind="serve", n=20000, keys=1024, lo=32, hi=16384),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["sign", "sign", "sign", "verify", "verify", "verify", "keygen", "persistent",
                       "keyed_verify", "keyed_sign", "host_sign", "host_verify", "serve"])
    if kind == "serve":
        return dict(kind=kind, n=_log_int(rng, 200, 20000), keys=rng.choice([64, 1024]), lo=32, hi=16384)
    low = 8 if kind.endswith("verify") else 1
    case = dict(kind=kind, level=rng.choice([2, 3, 5]), n=_log_int(rng, low, 20000), tuned=rng.random() < 0.6)
    if kind == "keygen":
        return case
    lo, hi, dist = rng.choice([(32, 32, "fixed"), (0, 0, "fixed"), (1001, 1001, "fixed"), (32, 4096, "uniform"),
                               (0, 300, "uniform"), (32, 16384, "loguniform")])
    case.update(lo=lo, hi=hi, dist=dist)
    if kind == "persistent":
        del case["level"]
        case["levels"] = rng.choice(["2", "3", "5", "25", "35", "235"])
    elif kind.startswith("keyed"):
        case["keys"] = _log_int(rng, 1, 4096)
    elif kind.startswith("host"):
        case["n"] = min(case["n"], 12000)
    return case


# ------------------------------------------------------------------ inputs
def _context(case):
    ctx = dil.Context(0)
    if case["tuned"]:
        ctx.apply_tuning()
    return ctx


def _seeds(n, rng):
    return torch.from_numpy(rng.integers(0, 256, size=(n, 32), dtype=np.uint8)).cuda()


def _messages(case, n, rng):
    lo, hi = case["lo"], case["hi"]
    if case["dist"] == "loguniform":
        lens = np.exp(rng.uniform(np.log(lo), np.log(hi), size=n)).astype(np.int64).clip(lo, hi)
    else:
        lens = rng.integers(lo, hi + 1, size=n, dtype=np.int64)
    off = np.zeros(n + 1, dtype=np.uint64)
    np.cumsum(lens, out=off[1:])
    return rng.integers(0, 256, size=max(int(off[-1]), 1), dtype=np.uint8), off


def _keys(level, n, rng):
    """n key pairs, made by a context of their own (as a user's key store would)."""
    with dil.Context(0) as ctx:
        ctx.apply_tuning()
        pk, sk = ctx.keygen(level, _seeds(n, rng))
        torch.cuda.synchronize()
    return pk, sk


def _signatures(level, sk, msg, off, rng):
    """Valid signatures with one in sixteen (of several, at least one) spoiled
    by a flipped bit."""
    with dil.Context(0) as ctx:
        ctx.apply_tuning()
        sig, _ = ctx.sign(level, sk, msg, off)
        torch.cuda.synchronize()
    n, size = sig.shape
    spoil = rng.random(n) < 1 / 16
    spoil[rng.integers(0, n)] |= n > 1
    bad = np.nonzero(spoil)[0]
    if bad.size:
        at = torch.from_numpy(rng.integers(0, size, size=bad.size)).cuda()
        sig[torch.from_numpy(bad).cuda(), at] ^= 4
    return sig


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind, n = case["kind"], case["n"]
    if kind == "serve":
        return _prepare_serve(case, seed, rng)
    s = {"kind": kind, "ctx": _context(case), "level": case.get("level")}
    level = s["level"]
    if kind == "keygen":
        s["seeds"] = _seeds(n, rng)
    elif kind == "persistent":
        s["jobs"], s["out"], s["keep"] = [], [], []
        for c in case["levels"]:
            lv = int(c)
            msg, off = _messages(case, n, rng)
            msg, off = torch.from_numpy(msg).cuda(), torch.from_numpy(off).cuda()
            _, sk = _keys(lv, n, rng)
            sig = torch.empty((n, dil.SIZES[lv][2]), dtype=torch.uint8, device="cuda")
            status = torch.empty(n, dtype=torch.int32, device="cuda")
            s["keep"].append((sk, msg, off))
            s["out"].append((sig, status))
            s["jobs"].append(dil.sign_job(lv, n, sk, msg, off, sig, status))
    elif kind in ("keyed_sign", "keyed_verify"):
        pk, sk = _keys(level, case["keys"], rng)
        s["store"] = _Store(s["ctx"], level, pk, sk)
        key = rng.integers(0, case["keys"], size=n).astype(np.int32)
        s["key"] = torch.from_numpy(key).cuda()
        msg, off = _messages(case, n, rng)
        s["msg"], s["off"] = torch.from_numpy(msg).cuda(), torch.from_numpy(off).cuda()
        if kind == "keyed_verify":
            s["sig"] = _signatures(level, sk[s["key"].long()].contiguous(), s["msg"], s["off"], rng)
    else:
        pk, sk = _keys(level, n, rng)
        msg, off = _messages(case, n, rng)
        s["pk"], s["sk"] = pk, sk
        s["msg"], s["off"] = torch.from_numpy(msg).cuda(), torch.from_numpy(off).cuda()
        if kind in ("verify", "host_verify"):
            s["sig"] = _signatures(level, sk, s["msg"], s["off"], rng)
        if kind.startswith("host"):   # the batch and its results in pinned host memory
            size = dil.SIZES[level][2]
            for k in ("pk", "sk", "msg", "off", "sig"):
                if k in s:
                    s[k] = s[k].cpu().pin_memory()
            s["h_sig"] = torch.zeros((n, size), dtype=torch.uint8).pin_memory()
            s["h_status"] = torch.zeros(n, dtype=torch.int32).pin_memory()
            s["h_ok"] = torch.zeros(n, dtype=torch.uint8).pin_memory()
    torch.cuda.synchronize()
    return s


class _Store:
    """A resident key store, freed with the state that holds it."""

    def __init__(self, ctx, level, pk, sk):
        self.ctx, self.pk, self.sk = ctx, pk, sk
        self.handle = dil.dil_keystore_create(ctx.handle, level, pk.shape[0], pk, sk)

    def __del__(self):
        dil.dil_keystore_destroy(self.handle)


def _prepare_serve(case, seed, rng):
    keys = {}
    srv = serving.Server(0, memory_budget=1 << 30, streams=2, max_batch=1024)
    for lv in (2, 3, 5):
        pk, sk = _keys(lv, case["keys"], rng)
        keys[lv] = (pk.cpu().numpy(), sk.cpu().numpy())
        srv.add_keys(lv, *keys[lv])
    req = serving.serving_workload(keys, case["n"], rate=1e9, seed=seed, lo=case["lo"], hi=case["hi"])
    return {"kind": "serve", "server": srv, "req": req}


# ------------------------------------------------------------------ one pass
def run(s):
    kind, level = s["kind"], s.get("level")
    if kind == "sign":
        return s["ctx"].sign(level, s["sk"], s["msg"], s["off"])
    if kind == "verify":
        return s["ctx"].verify(level, s["pk"], s["msg"], s["off"], s["sig"])
    if kind == "keygen":
        return s["ctx"].keygen(level, s["seeds"])
    if kind == "persistent":
        dil.dil_sign_persistent(s["ctx"].handle, s["jobs"])
        return s["out"]
    if kind == "serve":
        out = s["server"].replay(s["req"])
        return out["sig"], out["status"], out["ok"]
    h = s["ctx"].handle
    if kind == "host_sign":
        dil.dil_sign_host(h, level, s["sk"].shape[0], s["sk"], s["msg"], s["off"], s["h_sig"], s["h_status"])
        return s["h_sig"], s["h_status"]
    if kind == "host_verify":
        dil.dil_verify_host(h, level, s["pk"].shape[0], s["pk"], s["msg"], s["off"], s["sig"], s["h_ok"])
        return s["h_ok"]
    n = s["key"].shape[0]
    if kind == "keyed_sign":
        sig = torch.empty((n, dil.SIZES[level][2]), dtype=torch.uint8, device="cuda")
        status = torch.empty(n, dtype=torch.int32, device="cuda")
        dil.dil_sign_keyed(h, s["store"].handle, n, s["key"], s["msg"], s["off"], sig, status)
        return sig, status
    ok = torch.empty(n, dtype=torch.uint8, device="cuda")
    dil.dil_verify_keyed(h, s["store"].handle, n, s["key"], s["msg"], s["off"], s["sig"], ok)
    return ok


# ------------------------------------------------------------------ work
def _mean_length(case):
    lo, hi = case["lo"], case["hi"]
    if case.get("dist", "loguniform") == "loguniform" and hi > lo:
        return (hi - lo) / math.log(hi / lo)
    return (lo + hi) / 2


def _expand_s_perms(level):
    """SHAKE256 blocks ExpandS reads per polynomial (expected; 272 candidates a block)."""
    return {2: 1, 3: 2, 5: 1}[level]


def _ops(op, level, n, length, keyed=False):
    """32-bit integer operations of n tasks (the counts of the work model,
    with the expected repetitions of Sign)."""
    k, l = PARAMS[level]
    length = int(length)
    if op == "keygen":
        perms = 1 + 5 * k * l + _expand_s_perms(level) * (k + l) + WK.LEVELS[level]["pk"] // 136 + 1
        return n * (perms * WK.OPS_PER_PERMUTATION + 1024 * (k + l) * WK.OPS_PER_BUTTERFLY
                    + 256 * k * l * WK.OPS_PER_POINTWISE + 256 * (k * l + 3 * k + 2 * l) * WK.OPS_PER_COEFFICIENT)
    reps = WK.expected_iterations(level)
    one = WK.sign_work(level, [1], [length]) if op == "sign" else WK.verify_work(level, [length])
    total = float(WK.int_ops(one))
    if op == "sign":
        total += (reps - 1) * (WK.int_ops(WK.sign_work(level, [2], [length])) - WK.int_ops(one))
    if keyed:   # A^ and the transforms of the key are resident
        transforms = l + 2 * k if op == "sign" else k
        total -= (5 * k * l * WK.OPS_PER_PERMUTATION + 256 * k * l * WK.OPS_PER_COEFFICIENT
                  + 1024 * transforms * WK.OPS_PER_BUTTERFLY)
        if op == "verify":
            total -= (WK.LEVELS[level]["pk"] // 136 + 1) * WK.OPS_PER_PERMUTATION
    return n * total


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "serve":
        m, b, f = _mean_length(case), 0.0, 0.0
        for lv in (2, 3, 5):
            pk, sk, sig = dil.SIZES[lv]
            b += n / 3 * (m + 16 + sig)
            f += _ops("sign", lv, 0.4 * n / 3, m, keyed=True) + _ops("verify", lv, 0.6 * n / 3, m, keyed=True)
        return {"bytes": b, "flops": f}
    if kind == "keygen":
        pk, sk, _ = dil.SIZES[case["level"]]
        return {"bytes": n * (32.0 + pk + sk), "flops": float(_ops("keygen", case["level"], n, 0))}
    m = _mean_length(case)
    op = "verify" if kind.endswith("verify") else "sign"
    levels = [int(c) for c in case["levels"]] if kind == "persistent" else [case["level"]]
    b = f = 0.0
    for lv in levels:
        pk, sk, sig = dil.SIZES[lv]
        k, l = PARAMS[lv]
        if kind.startswith("keyed"):
            polys = k * l + (l + 2 * k if op == "sign" else k)
            key = min(n, case["keys"]) * polys * 1024.0 + 4 * n
        else:
            key = n * float(pk if op == "verify" else sk)
        b += key + n * (m + 8 + sig + (1 if op == "verify" else 4))
        f += _ops(op, lv, n, m, keyed=kind.startswith("keyed"))
    return {"bytes": b, "flops": f}


def exact(case, seed):
    """No output is a rounded number: all are bytes, statuses or accept bits."""
    return None
