"""Finalize's plan at the edges of its forms (one CTA, a thread-block cluster,
launches between the steps) and on maps of different kinds: random keys (few
long cycles), constant and sorted keys (nothing or one chain moves), reversed
runs (many short cycles) and a truncated permuted representation (paths that
end in the array).  Blocks of 64, so that n_pi = n/64 + 1025 positions are
reached with short arrays; the oracle is numpy's stable argsort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2607_05302_gb300 import radsort as R  # noqa: E402

pytestmark = pytest.mark.gpu


def make(kind, n):
    rng = np.random.default_rng(n)
    if kind == "random":
        return rng.integers(0, 2 ** 32, n, dtype=np.uint64).astype(np.uint32)
    if kind == "constant":
        return np.full(n, 0x01020304, dtype=np.uint32)
    if kind == "sorted":
        return np.arange(n, dtype=np.uint32)
    return (np.arange(n, dtype=np.uint32) // 977) ^ np.uint32(0xA5)


def check(kt, vt, keys, order):
    R.radsort_device_status()
    assert np.array_equal(kt.cpu().numpy().view(np.uint32), keys[order])
    assert np.array_equal(vt.cpu().numpy(), order.astype(np.int32))


@pytest.mark.parametrize("kind", ["random", "constant", "sorted", "runs"])
@pytest.mark.parametrize("npi", [1026, 4096, 4097, 30000, 65534, 65535])
@pytest.mark.parametrize("extra", [0, 17])
def test_edges(kind, npi, extra):
    n = (npi - 1025) * 64 + extra
    keys = make(kind, n)
    kt = torch.from_numpy(keys.view(np.int32)).cuda()
    vt = torch.arange(n, dtype=torch.int32, device="cuda")
    R.sort_tensors(kt, vt, layout="grid", block_size=64)
    check(kt, vt, keys, np.argsort(keys, kind="stable"))


@pytest.mark.parametrize("npi", [4096, 4097, 65534, 65535])
@pytest.mark.parametrize("share", [0.25, 0.9])
def test_truncated(npi, share):
    n = (npi - 1025) * 64 + 5
    keys = make("random", n)
    kt = torch.from_numpy(keys.view(np.int32)).cuda()
    vt = torch.arange(n, dtype=torch.int32, device="cuda")
    p = R.Perm(kt, vt, block_size=64)
    p.rounds(0, 4)
    m = int(n * share)
    p.truncate(m)
    p.finalize()
    check(kt[:m], vt[:m], keys, np.argsort(keys, kind="stable")[:m])


@pytest.mark.parametrize("chunks", [2, 7])
def test_chunk_layout(chunks):
    n = 3_000_017
    keys = make("random", n)
    kt = torch.from_numpy(keys.view(np.int32)).cuda()
    vt = torch.arange(n, dtype=torch.int32, device="cuda")
    R.sort_tensors(kt, vt, layout="chunks", block_size=256, num_chunks=chunks)
    check(kt, vt, keys, np.argsort(keys, kind="stable"))
