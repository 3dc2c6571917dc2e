"""The largest problems the image engine takes: two warps' states fill a CTA's shared memory.

A state of a byte per decision, syndrome bit and parity beside the messages bounds what fits. The steps' decision
words stand in the bytes' place; on a graph of long chains they may be longer, and must then not push out a problem
that fits with the bytes.
"""
import numpy as np
import pytest

import oracle
from paper_2508_15743_gb300 import dem as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SMEM = 227 * 1024


def a16(x):
    return (x + 15) // 16 * 16


def chain_problem(m, n, chain):
    """Columns 0..chain-1 each share a check with the one before: as many steps in natural order. The rest
    have one check each, spread so that no row has more than 8 entries (two FP32 chunks)."""
    cols = [sorted({i % m, (i + 1) % m}) for i in range(chain)]
    deg = np.zeros(m, int)
    for c in cols:
        deg[c] += 1
    for _ in range(n - chain):
        c = int(deg.argmin())
        cols.append([c])
        deg[c] += 1
    assert 5 <= deg.max() <= 8
    rows = [[] for _ in range(m)]
    for j, c in enumerate(cols):
        for r in c:
            rows[r].append(j)
    return D.DEM(D.CSR.from_rows(rows, n), D.CSR.from_rows([list(range(0, n, 5))], n),
                 np.random.default_rng(3).uniform(0.0005, 0.01, n))


@pytest.mark.parametrize("chain", [4400, 4550, 4700])
def test_long_chains_fit_where_bytes_do(chain):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_15743_gb300 import build
    build.build_library()
    from paper_2508_15743_gb300 import vibe as V
    m, n = 3000, 12608
    messages, candidate = a16(m * 8 * 4), a16((n + 31) // 32 * 4)
    with_bytes = messages + a16(n) + 2 * a16(m) + candidate
    assert SMEM - 64 < 2 * with_bytes <= SMEM        # the largest of its kind
    dm = chain_problem(m, n, chain)
    perms = np.arange(n, dtype=np.uint32)[None]
    syn, _ = D.sample(dm, 20, 5)
    dec = V.Decoder(dm, 1, perms, T=3, M=1, engine=V.ENGINE_IMAGE)
    out = dec.decode(torch.from_numpy(syn.view(np.int32)).cuda(), want_soft=True)
    torch.cuda.synchronize()
    r = oracle.decode(dm, perms, syn, 3, 0.625, 1, nthreads=8)
    assert np.array_equal(out["corrections"].cpu().numpy().view(np.uint32), r["corrections"])
    st = V.stats_to_numpy(out["stats"])
    for f in r["stats"].dtype.names:
        assert np.array_equal(st[f], r["stats"][f]), f
    assert np.array_equal(out["soft"].cpu().numpy().view(np.uint32), r["soft"].astype(np.float32).view(np.uint32))
    dec.close()
