"""The work a user of this package has it do, as cases that can be timed.

Every case goes through the public entry points: the ``Verifier`` methods, or
the ``binding`` wrappers of the C ABI where a program keeps its own result
buffers.  Sizes are those of ``paper_2411_01964_gb300.inputs`` (the single
ranges C1, C2 and C3, the 4096-range batch C4, the serving mix C5), of the
tests, or lie between them.  One resident prime table covers every request
(``TABLE_MAX_HI``), as in the benchmark and the server.

All outputs are whole numbers: histograms, first occurrences, lists, per-n
values, bitmap words.  Lists come back in buffers of a size that the case
fixes, zero past their length.

A case is a dict of plain values; ``kind`` says which call it makes:

  points         Verifier.min_k(points): host array in, host array out
  points_device  Verifier.min_k_device: device arrays
  range          Verifier.verify_range (``per_n``: with the per-n output)
  range_buffers  binding.sv_verify_range into the caller's own buffers
                 (``pinned``: page-locked ones)
  range_device   Verifier.launch_range with a device per-n buffer, fetch_range
  bitmap         Verifier.sieve_bitmap (Algorithm 1 alone)
  batch          binding.sv_verify_batch
  serve          binding.sv_submit_many, then sv_poll of every ticket
"""
from __future__ import annotations

import ctypes
import functools
import math

import numpy as np
import torch

from paper_2411_01964_gb300 import Verifier, odd_count
from paper_2411_01964_gb300 import binding as B
from paper_2411_01964_gb300.inputs import TABLE_MAX_HI, SplitMix64, random_points

# 1 - c_(k-1) of Table 2: the share of the odd n with mink >= k
TAIL = (1.0, 1.0, 1.8943e-1, 2.4129e-2, 2.1482e-3, 1.3902e-4, 6.8527e-6)


def listed():
    return [
        # one n asked for by hand or by a request handler: latency alone
        dict(name="point_1", kind="points", count=1, log2_hi=50),
        # the largest point query of the serving mix
        dict(name="points_1024", kind="points", count=1024, log2_hi=50),
        # a program that holds its candidates on the GPU, e.g. filtered from
        # elsewhere: throughput of the exact test
        dict(name="points_device_65536", kind="points_device", count=65536, log2_hi=50),
        # the short range that 70% of the serving mix asks for, by itself
        dict(name="range_short", kind="range_buffers", log2_base=46, length=23457, pinned=False),
        # C1's size from near the bottom, with mink of every n (the plain
        # method's full output)
        dict(name="range_16m_per_n", kind="range", log2_base=0, length=1 << 24, per_n=True),
        # one ordinary range: the longest of the batch requests
        dict(name="range_268m", kind="range", log2_base=47, length=1 << 28, per_n=False),
        # C2: the high range, histogram and list
        dict(name="range_17g", kind="range_buffers", log2_base=40, length=1 << 34, pinned=True),
        # C3's size next to the paper's bound: a chunk of the full sweep
        dict(name="range_69g", kind="range_buffers", log2_base=49.9, length=1 << 36, pinned=True),
        # mink of every n kept on the GPU for further work there
        dict(name="range_device_per_n_2g", kind="range_device", log2_base=44, length=(1 << 31) + 12346),
        # the squarefree flags alone, for other uses of the sieve
        dict(name="bitmap_4g", kind="bitmap", log2_base=45, length=(1 << 32) + 778),
        # C4: uneven ranges as one launch
        dict(name="batch_4096", kind="batch", count=4096, log2_len_lo=10, log2_len_hi=28),
        # C5: a burst of the serving mix, as it stands in the queue of a busy server
        dict(name="serve_256", kind="serve", count=256, log2_long_hi=30),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("points", "points_device", "range", "range", "range_buffers", "range_buffers", "range_device",
                       "bitmap", "batch", "serve"))
    if kind == "points":
        return dict(kind=kind, count=_log_uniform(rng, 1, 4096), log2_hi=rng.randint(30, 50))
    if kind == "points_device":
        return dict(kind=kind, count=_log_uniform(rng, 1, 65536), log2_hi=rng.randint(30, 50))
    if kind == "range":
        per_n = rng.random() < 0.5
        return dict(kind=kind, log2_base=rng.uniform(0, 49.5), length=_log_uniform(rng, 1 << 10, 1 << (24 if per_n else 34)),
                    per_n=per_n)
    if kind == "range_buffers":
        return dict(kind=kind, log2_base=rng.uniform(30, 49.5), length=_log_uniform(rng, 1 << 10, 1 << 36),
                    pinned=rng.random() < 0.5)
    if kind == "range_device":
        return dict(kind=kind, log2_base=rng.uniform(0, 49.5), length=_log_uniform(rng, 1 << 14, 1 << 31))
    if kind == "bitmap":
        return dict(kind=kind, log2_base=rng.uniform(0, 49.5), length=_log_uniform(rng, 1 << 10, 1 << 32))
    if kind == "batch":
        a = rng.randint(8, 20)
        return dict(kind=kind, count=_log_uniform(rng, 8, 4096), log2_len_lo=a, log2_len_hi=rng.randint(a + 2, 28))
    return dict(kind=kind, count=_log_uniform(rng, 8, 256), log2_long_hi=rng.randint(26, 30))


# ---- inputs -------------------------------------------------------------------

_kept = {}  # kind -> Verifier: a program keeps one context (and its prime table) from call to call


def _verifier(kind):
    if kind not in _kept:
        _kept.clear()  # the states of the previous kind hold theirs as long as they need it
        _kept[kind] = Verifier(max_hi=TABLE_MAX_HI)
    return _kept[kind]


def _range_of(case, seed):
    """[lo, lo + length): lo odd, near 2^log2_base and moved by the seed (by at most a sixteenth of it, in whole 64s,
    so that the odd numbers and bitmap words of a case are equally many for every seed)."""
    rng = SplitMix64(seed)
    base, length = max(int(2.0 ** case["log2_base"]), 1 << 10), case["length"]
    base = min(base, (1 << 50) - length - (1 << 20))
    lo = (base & ~63) + 64 * rng.below(max(base >> 10, 2)) + (length % 64 | 1)
    if lo + length > 1 << 50:
        lo = ((1 << 50) - length - 64 * (1 + rng.below(1 << 14)) & ~63) + (length % 64 | 1)
    return lo, lo + length


def _requests(case, seed):
    """Uneven ranges with odd starts uniform in [2^30, 2^50); lengths: octave uniform, then uniform inside it."""
    rng = SplitMix64(seed)
    out = []
    for _ in range(case["count"]):
        lo = (1 << 30) + 1 + 2 * rng.below(((1 << 50) - (1 << 30)) // 2)
        e = case["log2_len_lo"] + rng.below(case["log2_len_hi"] - case["log2_len_lo"])
        out.append((lo, lo + (((1 << e) + rng.below(1 << e)) & ~1)))
    return out


def _mix(case, seed):
    """The serving mix in random order: 70% short ranges, 20% long ones, 10% point queries."""
    rng = SplitMix64(seed)
    n = case["count"]
    n_long, n_points = n // 5, n // 10
    order = [0] * (n - n_long - n_points) + [1] * n_long + [2] * n_points
    for i in range(n - 1, 0, -1):
        j = rng.below(i + 1)
        order[i], order[j] = order[j], order[i]
    out = []
    for c in order:
        if c == 2:
            out.append([3 + 2 * rng.below(1 << 49) for _ in range(1 + rng.below(MAX_POINTS))])
            continue
        lo = (1 << 30) + 1 + 2 * rng.below(((1 << 50) - (1 << 30)) // 2)
        a, b = (12, 16) if c == 0 else (24, case["log2_long_hi"])
        e = a + rng.below(b - a)
        out.append((lo, lo + (((1 << e) + rng.below(1 << e)) & ~1)))
    return out


MAX_POINTS = 1024  # of one point query


def _list_cap(length):
    """Room for every listed n (mink >= 6) of a range, with plenty to spare."""
    return int(TAIL[6] * length) + 64


class _Results:
    """Result structures of several ranges with one arena for their lists, all owned by the caller."""

    FAILS = 8

    def __init__(self, ranges, longest, pinned=False):
        n = len(ranges)
        caps = [_list_cap(hi - lo) for lo, hi in ranges]
        total = max(n, 1) * _list_cap(longest)  # the lists lie one behind the other at its start
        if pinned:
            self._keep = (torch.zeros(total, dtype=torch.int64, pin_memory=True),
                          torch.zeros(total, dtype=torch.uint8, pin_memory=True))
            self.list_n, self.list_k = (t.numpy() for t in self._keep)
        else:
            self.list_n, self.list_k = np.zeros(total, dtype=np.int64), np.zeros(total, dtype=np.uint8)
        self.failures = np.zeros((max(n, 1), self.FAILS), dtype=np.int64)
        self.arr = (B.sv_range_result * max(n, 1))()
        off = 0
        for i, cap in enumerate(caps):
            r = self.arr[i]
            r.list = ctypes.cast(self.list_n.ctypes.data + 8 * off, B.P(B.u64))
            r.list_k = ctypes.cast(self.list_k.ctypes.data + off, B.P(B.u8))
            r.list_cap = cap
            r.failures = ctypes.cast(self.failures.ctypes.data + 8 * self.FAILS * i, B.P(B.u64))
            r.fail_cap = self.FAILS
            off += cap
        # the structures as rows of 64-bit words (every field has eight bytes)
        self.words = np.frombuffer(self.arr, dtype=np.int64).reshape(max(n, 1), -1)[:n]

    def columns(self, name):
        f = getattr(B.sv_range_result, name)
        return self.words[:, f.offset // 8: (f.offset + f.size) // 8]

    def outputs(self):
        out = {k: self.columns(k) for k in ("n_odd", "hist", "first_n", "ksum", "kmax", "list_len", "fail_len",
                                            "list_overflow")}
        out.update(list_n=self.list_n, list_k=self.list_k, failures=self.failures)
        return out

    def one(self):
        """The outputs of a single range (the library leaves the entries past the list's length unspecified)."""
        m = int(self.arr[0].list_len)
        self.list_n[m:] = 0
        self.list_k[m:] = 0
        return self.outputs()


def prepare(case, seed):
    kind = case["kind"]
    v = _verifier(kind)
    s = {"kind": kind, "v": v}
    if kind == "points":
        s["points"] = np.array(random_points(seed, case["count"], 2, 1 << case["log2_hi"]), dtype=np.uint64)
    elif kind == "points_device":
        # splitmix64 outputs, drawn side by side
        with np.errstate(over="ignore"):
            z = np.uint64(seed) + np.arange(1, case["count"] + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z ^= z >> np.uint64(31)
        pts = (z >> np.uint64(64 - case["log2_hi"])) | np.uint64(3)
        s["points"] = torch.from_numpy(pts.view(np.int64)).cuda()
        s["out"] = torch.empty(case["count"], dtype=torch.uint8, device="cuda")
    elif kind in ("batch", "serve"):
        reqs = _requests(case, seed) if kind == "batch" else _mix(case, seed)
        ranges = [r for r in reqs if isinstance(r, tuple)]
        s["res"] = res = _Results(ranges, 1 << case["log2_len_hi" if kind == "batch" else "log2_long_hi"])
        if kind == "batch":
            s["lo"] = np.array([a for a, _ in ranges], dtype=np.uint64)
            s["hi"] = np.array([b for _, b in ranges], dtype=np.uint64)
            return s
        queries = max(sum(isinstance(r, list) for r in reqs), 1)
        s["points"] = np.zeros((queries, MAX_POINTS), dtype=np.uint64)
        s["out_k"] = np.zeros((queries, MAX_POINTS), dtype=np.uint8)
        s["reqs"] = (B.sv_request * len(reqs))()
        s["tickets"], s["status"] = np.zeros(len(reqs), dtype=np.uint64), np.zeros(len(reqs), dtype=np.int32)
        i_range = i_point = 0
        for q, r in zip(s["reqs"], reqs):
            if isinstance(r, tuple):
                q.kind, q.lo, q.hi = B.SV_REQ_RANGE, *r
                q.result = ctypes.pointer(res.arr[i_range])
                i_range += 1
            else:
                q.kind, q.n_points = B.SV_REQ_POINTS, len(r)
                s["points"][i_point, :len(r)] = r
                q.points = s["points"][i_point].ctypes.data_as(B.P(B.u64))
                q.out_k = s["out_k"][i_point].ctypes.data_as(B.P(B.u8))
                i_point += 1
    else:
        s["lo"], s["hi"] = lo, hi = _range_of(case, seed)
        if kind == "range":
            s["per_n"] = case["per_n"]
            s["list_cap"] = _list_cap(case["length"])
        elif kind == "range_buffers":
            s["res"] = _Results([(lo, hi)], case["length"], pinned=case["pinned"])
        elif kind == "range_device":
            s["per_n"] = torch.empty(odd_count(lo, hi), dtype=torch.uint8, device="cuda")
            s["list_cap"] = _list_cap(case["length"])
    return s


# ---- one pass -------------------------------------------------------------------

def _padded(x, n):
    out = np.zeros(n, dtype=x.dtype)
    out[:len(x)] = x
    return out


def _of_result(r, list_cap):
    out = dict(n_odd=r.n_odd, ksum=r.ksum, kmax=r.kmax, list_len=r.list_len, fail_len=r.fail_len,
               hist=np.array(r.hist, dtype=np.uint64).view(np.int64),
               first_n=np.array(r.first_n, dtype=np.uint64).view(np.int64),
               list_n=_padded(r.list_n.view(np.int64), list_cap), list_k=_padded(r.list_k, list_cap))
    if r.per_n_k is not None:
        out["per_n_k"] = r.per_n_k
    return out


def run(s):
    kind, v = s["kind"], s["v"]
    if kind == "points":
        return {"n": s["points"].view(np.int64), "mink": v.min_k(s["points"])}
    if kind == "points_device":
        v.min_k_device(s["points"], s["out"])
        return {"n": s["points"], "mink": s["out"]}
    if kind == "range":
        r = v.verify_range(s["lo"], s["hi"], list_cap=s["list_cap"], per_n=s["per_n"])
        return _of_result(r, s["list_cap"])
    if kind == "range_buffers":
        B.check(B.sv_verify_range(v.ctx, s["lo"], s["hi"], s["res"].arr[0]), "sv_verify_range")
        return s["res"].one()
    if kind == "range_device":
        v.launch_range(s["lo"], s["hi"], s["per_n"])
        out = _of_result(v.fetch_range(list_cap=s["list_cap"]), s["list_cap"])
        out["per_n_k"] = s["per_n"]
        return out
    if kind == "bitmap":
        return v.sieve_bitmap(s["lo"], s["hi"])
    if kind == "batch":
        B.check(B.sv_verify_batch(v.ctx, s["lo"], s["hi"], s["res"].arr), "sv_verify_batch")
        return s["res"].outputs()
    B.check(B.sv_submit_many(v.ctx, s["reqs"], s["tickets"], s["status"]), "sv_submit_many")
    for t in s["tickets"]:
        B.check(B.sv_poll(v.ctx, int(t), -1), "sv_poll")
    return {**s["res"].outputs(), "out_k": s["out_k"]}


# ---- what a pass cannot do without ------------------------------------------------

def _ops_per_odd(hi):
    """Integer operations per odd n in words of 32: two per strike of every p^2 (p >= 3), and a shift, an update and a
    count for every step of the search that a word needs (k until none of its 32 n is left)."""
    strikes = 0.2022 - 1.0 / (math.sqrt(hi) * math.log(math.sqrt(hi)))  # sum of 1 / p^2 over the odd p below sqrt(hi)
    steps = 1.0 + sum(1.0 - (1.0 - t) ** 32 for t in TAIL[2:])
    return 2 * strikes + 3 * steps / 32


def _point_ops(n_hi):
    """The exact test of n - 2^k by the primes up to its cube root, three operations each, 1.22 probes per n."""
    c = n_hi ** (1 / 3)
    return 3 * 1.22 * c / max(math.log(c), 1.0)


RESULT_BYTES = 8 * 142


def work(case):
    kind = case["kind"]
    if kind in ("points", "points_device"):
        return {"bytes": 9 * case["count"], "flops": case["count"] * _point_ops(2.0 ** case["log2_hi"])}
    if kind in ("batch", "serve"):
        if kind == "batch":
            ranges, pts = _requests(case, 1), []
        else:
            mix = _mix(case, 1)
            ranges, pts = [r for r in mix if isinstance(r, tuple)], [n for r in mix if isinstance(r, list) for n in r]
        n = sum(odd_count(a, b) for a, b in ranges)
        return {"bytes": (16 + RESULT_BYTES) * len(ranges) + 9 * TAIL[6] * n + 9 * len(pts),
                "flops": n * _ops_per_odd(2.0 ** 50) + len(pts) * _point_ops(2.0 ** 50)}
    lo, hi = _range_of(case, 1)
    n = odd_count(lo, hi)
    if kind == "bitmap":
        return {"bytes": 16 + n / 8, "flops": n * 2 * 0.2022}
    per_n = n if kind == "range_device" or case.get("per_n") else 0
    return {"bytes": 16 + RESULT_BYTES + 9 * TAIL[6] * n + per_n, "flops": n * _ops_per_odd(hi)}


# ---- the same by numpy -------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _primes(limit):
    flags = np.ones(limit + 1, dtype=bool)
    flags[:2] = False
    flags[4::2] = False
    for p in range(3, math.isqrt(limit) + 1, 2):
        if flags[p]:
            flags[p * p::2 * p] = False
    return np.flatnonzero(flags)[1:].astype(np.int64)  # the odd ones


def _squarefree_odd(lo, hi):
    """Flags of the odd integers lo, lo + 2, ... below hi (lo odd)."""
    n = (hi - lo + 1) // 2
    flags = np.ones(n, dtype=bool)
    p = _primes(1 << max(math.isqrt(hi - 1), 3).bit_length())
    q = p * p
    first = (-lo) % q                       # lo + first is the next multiple
    first = np.where(first % 2 == 0, first, first + q) // 2
    near = first < n
    for f, step in zip(first[near].tolist(), q[near].tolist()):
        flags[f::step] = False
    return flags


def _mink(lo, hi):
    """mink of the odd n in [max(lo, 3), hi)."""
    lo = max(lo, 3) | 1
    n = np.arange(lo, hi, 2, dtype=np.int64)
    out = np.full(len(n), 255, dtype=np.uint8)
    left = np.arange(len(n))
    k = 1
    while len(left) and (1 << k) < hi:
        if len(left) > 64:                  # dense: a shifted sieve
            a = max(lo - (1 << k), 1)
            flags = _squarefree_odd(a, hi - (1 << k)) if hi - (1 << k) > a else np.zeros(0, dtype=bool)
            at = (n[left] - (1 << k) - a) // 2
            ok = (at >= 0) & (n[left] > (1 << k))
            ok[ok] = flags[at[ok]]
        else:
            ok = np.array([int(x) > (1 << k) and bool(_squarefree_odd(int(x) - (1 << k), int(x) - (1 << k) + 1)[0])
                           for x in n[left]])
        out[left[ok]] = k
        left = left[~ok]
        k += 1
    return out


def exact(case, seed):
    """What run() returns for the small single ranges, by numpy; the other cases take too long that way."""
    if case["kind"] not in ("range", "range_buffers") or case["length"] > 1 << 22:
        return None
    lo, hi = _range_of(case, seed)
    k = _mink(lo, hi)
    n = np.arange(max(lo, 3) | 1, hi, 2, dtype=np.int64)
    hist = np.bincount(k[k < 64], minlength=64).astype(np.int64)
    first = np.full(64, -1, dtype=np.int64)
    for j in np.flatnonzero(hist):
        first[j] = n[np.argmax(k == j)]
    listed_n = (k >= 6) & (k < 255)
    got = dict(n_odd=len(n), ksum=int((hist * np.arange(64)).sum()), kmax=int(np.flatnonzero(hist).max(initial=0)),
               list_len=int(listed_n.sum()), fail_len=int((k == 255).sum()), hist=hist, first_n=first,
               list_n=_padded(n[listed_n], _list_cap(case["length"])),
               list_k=_padded(k[listed_n], _list_cap(case["length"])))
    if case["kind"] == "range_buffers":
        cell = lambda x: np.array([[x]], dtype=np.int64)  # noqa: E731
        got = {m: cell(x) if isinstance(x, int) else x for m, x in got.items()}
        got.update(hist=hist[None], first_n=first[None], list_overflow=cell(0),
                   failures=_padded(n[k == 255], _Results.FAILS)[None])
    elif case["per_n"]:
        got["per_n_k"] = k
    return got
