"""The allocation-free colouring of graphs whose neighbours lie anywhere (sparse ones take the kernel per
level), and of the same graphs in order, against the oracle, on both sides of the sizes and degrees at
which the kernel changes."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


def _csr(n, i, j):
    key = np.unique(np.concatenate([i * n + j, j * n + i]))
    a, b = key // n, key % n
    a, b = a[a != b], b[a != b]
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(a, minlength=n))
    return rp, b.astype(np.uint32)


def _edges(kind, n, rng):
    if kind == "path":
        i = np.arange(n - 1)
        return n, i, i + 1
    if kind == "grid":
        w = int(n ** 0.5)
        n = w * w
        v = np.arange(n)
        r = v[v % w < w - 1]
        return n, np.concatenate([r, v[:n - w]]), np.concatenate([r + 1, v[:n - w] + w])
    if kind == "matching":
        p = rng.permutation(n)
        return n, p[0:n // 2 * 2:2], p[1::2]
    m = int(n * float(kind) / 2)
    return n, rng.integers(n, size=m), rng.integers(n, size=m)


@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("kind,n", [("path", 16383), ("path", 16384), ("path", 40001), ("grid", 120409), ("grid", 132496),
                                    ("matching", 16385), ("matching", 150000), ("1.0", 180000), ("1.0", 200000),
                                    ("4.0", 150000), ("0.0", 20000)])
def test_static_matches_oracle(kind, n, shuffle):
    import torch

    rng = np.random.default_rng(5)
    n, i, j = _edges(kind, n, rng)
    if shuffle:
        p = rng.permutation(n)
        i, j = p[i], p[j]
    rp, col = _csr(n, i.astype(np.int64), j.astype(np.int64))
    ref, rounds, delta = O.kw_colour_graph(rp, col, 0)
    d_rp = torch.from_numpy(rp.astype(np.int32)).cuda()
    d_col = torch.from_numpy(col.view(np.int32).copy() if col.size else np.zeros(1, np.int32)).cuda()
    out = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        out.fill_(-1)
        got = sco.kw_colour_static(d_rp.data_ptr(), d_col.data_ptr(), n, out.data_ptr(),
                                   stream=torch.cuda.current_stream().cuda_stream)
        assert got == (delta, rounds)
        assert np.array_equal(out.cpu().numpy(), ref)
