"""What this library is timed on: sorts as its users call them, from one small
request to the largest arrays, through the public binding.

A pass copies fresh, unsorted input over the working buffers (the sorts are in
place, and a second sort of sorted data would be another workload) and sorts
them.  Keys and values share one buffer, so that the copy is one launch.
Inputs are made on the device from the seed alone; payloads are the original
index, so that the outputs also show stability.
"""
import math

import numpy as np
import torch

from paper_2607_05302_gb300 import radsort as R
from paper_2607_05302_gb300 import workloads as W

DEV = "cuda"


def listed():
    return [
        # one short request sorted on its own, the call without a workspace:
        # launches and latency are all there is
        sort_case("sort_u32_1000", 1000, workspace=False),
        # a short array that the automatic plan sorts out of place in scratch
        sort_case("sort_u32_100003", 100_003),
        # one million keys, the smallest size the package is configured for
        sort_case("sort_u32_2p20", 1 << 20),
        # keys alone, ragged size
        sort_case("sort_u32_keys_16777259", 16_777_259, values=False),
        # uniform keys with their index, the size every distribution is run at
        sort_case("sort_u32_2p28", 1 << 28),
        # skewed keys at that size (Zipf over 2^16 values), as identifiers and
        # words in logs and columns are
        sort_case("sort_u32_zipf_2p28", 1 << 28, dist="zipf"),
        # float32 keys N(0,1): scores sorted with their index, ragged size
        sort_case("sort_f32_67108901", 67_108_901, dist="float"),
        # the benchmark's headline array
        sort_case("sort_u32_2p30", 1 << 30),
        # 64-bit keys, the largest request of the serving configuration
        sort_case("sort_u64_2p29", 1 << 29, key_bytes=8),
        # 64-bit keys with the wide digits
        sort_case("sort_u64_d11_2p27", 1 << 27, key_bytes=8, digit_bits=11),
        # 20,000 arrays of lognormal lengths in one call, replayed as a graph
        seg_case("segmented_u32_20000_graph", 20_000, 4096.0, 2.0, 1 << 22, graph=True),
        # the permuted representation: sorted, read in order without
        # Finalize, cut to a prefix, finalized
        perm_case("perm_u32_30000001", 30_000_001, 0.25),
    ]


def sort_case(name, n, *, dist="uniform", key_bytes=4, values=True, digit_bits=8, workspace=True):
    c = {"name": name, "kind": "sort", "n": n, "dist": dist, "key_bytes": key_bytes, "values": values,
         "digit_bits": digit_bits, "workspace": workspace}
    return c if name else {k: v for k, v in c.items() if k != "name"}


def seg_case(name, num, median, sigma, longest, *, key_bytes=4, digit_bits=8, graph=False, lengths_seed=7):
    c = {"name": name, "kind": "segmented", "num": num, "median": median, "sigma": sigma, "longest": longest,
         "key_bytes": key_bytes, "digit_bits": digit_bits, "graph": graph, "lengths_seed": lengths_seed}
    return c if name else {k: v for k, v in c.items() if k != "name"}


def perm_case(name, n, keep, *, key_bytes=4, digit_bits=8):
    c = {"name": name, "kind": "perm", "n": n, "keep": keep, "key_bytes": key_bytes, "digit_bits": digit_bits}
    return c if name else {k: v for k, v in c.items() if k != "name"}


def _spread(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi], odd ones among them."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["sort", "segmented", "perm"], [8, 2, 1])[0]
    if kind == "perm":
        return perm_case(None, _spread(rng, 1 << 19, 1 << 27), rng.choice([0.01, 0.1, 0.5, 1.0]),
                         key_bytes=rng.choice([4, 4, 8]))
    if kind == "segmented":
        # batches of requests: few longer ones up to many short ones
        num = _spread(rng, 16, 20_000)
        median = float(_spread(rng, 256, max(300, min(65_536, (1 << 25) // num))))
        return seg_case(None, num, median, rng.choice([0.5, 1.0, 2.0]), 1 << 22, key_bytes=rng.choice([4, 4, 8]),
                        digit_bits=rng.choice([8, 8, 8, 11]), graph=rng.random() < 0.5,
                        lengths_seed=rng.randrange(1 << 20))
    kb = rng.choice([4, 4, 4, 8])
    db = rng.choice([8, 8, 8, 8, 8, 11])
    dist = rng.choice(["uniform"] * 4 + ["sorted", "low_bits"] + (["zipf", "float"] if kb == 4 else []))
    top = (1 << 29 if kb == 4 else 1 << 28) if db == 8 else 1 << 26
    if dist in ("zipf", "sorted"):
        top = min(top, 1 << 27)
    return sort_case(None, _spread(rng, 500, top), dist=dist, key_bytes=kb, values=rng.random() < 0.75,
                     digit_bits=db, workspace=rng.random() < 0.7)


# ---------------------------------------------------------------- inputs
_STEP = 1 << 26  # elements made at a time


def _lsr(x, k):
    return (x >> k) & ((1 << (64 - k)) - 1)


def _fmix32(h):
    """MurmurHash3's 32-bit finaliser on int64 holding 32-bit values (the
    mapping of workloads.fmix32_np)."""
    m = 0xFFFFFFFF
    h = h ^ (h >> 16)
    h = (h * 0x85EBCA6B) & m
    h = h ^ (h >> 13)
    h = (h * 0xC2B2AE35) & m
    return h ^ (h >> 16)


def _fill_keys(out, dist, seed):
    """Keys of a distribution into the int32 / float32 / int64 tensor `out`."""
    n = out.numel()
    if dist == "zipf":
        w = np.arange(1, (1 << 16) + 1, dtype=np.float64) ** -1.1
        cdf = np.cumsum(w)
        cdf = torch.from_numpy(cdf / cdf[-1]).to(DEV)
    for s in range(0, n, _STEP):
        c = min(_STEP, n - s)
        o = out[s:s + c]
        if dist == "float":
            r = W.splitmix64_torch(seed, 2 * s, 2 * c, device=DEV)
            u = _lsr(r, 11).to(torch.float64) * 2.0 ** -53
            o.copy_(torch.sqrt(-2.0 * torch.log(u[0::2] + 2.0 ** -53)) * torch.cos(2.0 * math.pi * u[1::2]))
            continue
        r = W.splitmix64_torch(seed, s, c, device=DEV)
        if dist == "zipf":
            u = _lsr(r, 11).to(torch.float64) * 2.0 ** -53
            rank = torch.searchsorted(cdf, u, right=True).clamp_(max=(1 << 16) - 1)
            o.copy_(_fmix32(rank ^ (W.SEEDS["zipf"] & 0xFFFFFFFF)))
        elif dist == "low_bits":  # identifiers far below the key type's range: the top digits are constant
            o.copy_(_lsr(r, 40))
        else:
            o.copy_(_lsr(r, 32) if out.element_size() == 4 else r)
    if dist == "sorted":
        out.copy_(torch.sort(out).values)


def _al(x):
    return (x + 255) // 256 * 256


class _Arrays:
    """Input and working buffers, [keys | values] in one allocation each."""

    def __init__(self, n, key_bytes, values, dist, seed):
        kbytes = _al(n * key_bytes)
        total = kbytes + (_al(n * 4) if values else 0)
        kt = torch.int64 if key_bytes == 8 else torch.float32 if dist == "float" else torch.int32
        self.fresh = torch.zeros(total, dtype=torch.uint8, device=DEV)
        self.work = torch.empty_like(self.fresh)

        def split(buf):
            return (buf[:n * key_bytes].view(kt),
                    buf[kbytes:kbytes + n * 4].view(torch.int32) if values else None)

        k, v = split(self.fresh)
        _fill_keys(k, dist, seed)
        if values:
            torch.arange(n, dtype=torch.int32, device=DEV, out=v)
        self.keys, self.vals = split(self.work)

    def refresh(self):
        self.work.copy_(self.fresh)


def _seg_offsets(case):
    lens = W.lognormal_lengths(case["num"], median=case["median"], sigma_ln=case["sigma"], hi=case["longest"],
                               seed=0xC0FFEE07 + case["lengths_seed"])
    off = np.zeros(case["num"] + 1, np.uint64)
    np.cumsum(lens.astype(np.uint64), out=off[1:])
    return off


def _seed(seed):
    return (0x5EED + 0x9E3779B1 * int(seed)) & 0x7FFFFFFFFFFFFFFF


def prepare(case, seed):
    seed, kb, db = _seed(seed), case["key_bytes"], case["digit_bits"]
    if case["kind"] == "segmented":
        off = _seg_offsets(case)
        n = int(off[-1])
        a = _Arrays(n, kb, True, "uniform", seed)
        st = {"case": case, "a": a, "off": off, "off_dev": torch.from_numpy(off.view(np.int64)).to(DEV),
              "ws": torch.empty(max(1, R.segmented_workspace_size(off, kb, 4, db)), dtype=torch.uint8, device=DEV)}
        if case["graph"]:
            _segmented(st)  # the library's streams exist before the capture
            torch.cuda.synchronize()
            st["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(st["graph"]):
                _segmented(st)
        return st
    n = case["n"]
    if case["kind"] == "perm":
        return {"case": case, "a": _Arrays(n, kb, True, "uniform", seed),
                "ws": torch.empty(R.perm_workspace_size(n, kb, 4, db), dtype=torch.uint8, device=DEV),
                "out": (torch.empty(n, dtype=torch.int64 if kb == 8 else torch.int32, device=DEV),
                        torch.empty(n, dtype=torch.int32, device=DEV))}
    st = {"case": case, "a": _Arrays(n, kb, case["values"], case["dist"], seed), "ws": None}
    if case["workspace"]:
        need = R.radsort_workspace_size(n, kb, 4 if case["values"] else 0, db)
        st["ws"] = torch.empty(max(1, need), dtype=torch.uint8, device=DEV)
    return st


# ---------------------------------------------------------------- one pass
def _segmented(st):
    a = st["a"]
    R.sort_segmented_tensors(a.keys, a.vals, st["off_dev"], st["off"], digit_bits=st["case"]["digit_bits"],
                             workspace=st["ws"])


def run(st):
    case, a = st["case"], st["a"]
    a.refresh()
    if case["kind"] == "segmented":
        if case["graph"]:
            st["graph"].replay()
        else:
            _segmented(st)
        return [a.keys, a.vals]
    if case["kind"] == "perm":
        n, db = case["n"], case["digit_bits"]
        m = max(1, int(n * case["keep"]))
        p = R.Perm(a.keys, a.vals, digit_bits=db, workspace=st["ws"])
        p.rounds(0, -(-8 * case["key_bytes"] // db))
        p.gather(*st["out"])
        p.truncate(m)
        p.finalize()
        p.close()
        return [*st["out"], a.keys[:m], a.vals[:m]]
    R.sort_tensors(a.keys, a.vals, digit_bits=case["digit_bits"], float_keys=case["dist"] == "float",
                   workspace=st["ws"])
    return [a.keys] if a.vals is None else [a.keys, a.vals]


def work(case):
    """Every element read once and written once (the permuted case writes the
    gathered sequence and the finalized prefix); no arithmetic to speak of."""
    n = int(_seg_offsets(case)[-1]) if case["kind"] == "segmented" else case["n"]
    e = case["key_bytes"] + (4 if case.get("values", True) else 0)
    out = n + max(1, int(n * case["keep"])) if case["kind"] == "perm" else n
    return {"bytes": float(n * e + out * e), "flops": 0.0}


def exact(case, seed):
    """Float keys in ascending order (whole numbers are compared as they are)."""
    if case["kind"] != "sort" or case["dist"] != "float":
        return None
    keys = torch.empty(case["n"], dtype=torch.float32, device=DEV)
    _fill_keys(keys, "float", _seed(seed))
    k64 = torch.sort(keys.to(torch.float64)).values
    return [k64, None] if case["values"] else [k64]
