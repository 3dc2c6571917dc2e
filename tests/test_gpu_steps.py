"""GPU parity of the packed steps (32 edges of columns that share no check) at their edges.

A sweep runs a member's columns in steps: every lane takes one edge, the lanes of a column pass each
other its check-to-variable messages. The problems here sit where that packing can go wrong: columns
without checks, columns that fill half a step or leave lanes over, chains where every step holds one
column, rows of one entry and of the most entries, steps at the ends of the blocks the kernels work in,
hard constraints. Results must equal the oracle's bit for bit (corrections, logical
flips, records, posteriors) on both engines and in shot and pair mode.
"""
import numpy as np
import pytest

import oracle
from paper_2508_15743_gb300 import dem as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_15743_gb300 import build
    build.build_library()
    from paper_2508_15743_gb300 import vibe
    return vibe


def make_dem(cols, m, seed):
    """A DEM whose column j touches the checks cols[j]; one logical over every third column."""
    n = len(cols)
    H = np.zeros((m, n), np.uint8)
    for j, c in enumerate(cols):
        H[list(c), j] = 1
    L = np.zeros((1, n), np.uint8)
    L[0, ::3] = 1
    rng = np.random.default_rng(seed)
    return D.DEM(D.CSR.from_dense(H), D.CSR.from_dense(L), rng.uniform(0.005, 0.2, n))


def random_cols(rng, n, m, degs):
    return [sorted(rng.choice(m, int(d), replace=False)) for d in rng.choice(degs, n)]


def problem(name):
    rng = np.random.default_rng(7)
    if name == "one_by_one":
        return make_dem([[0]], 1, 1)
    if name == "no_checks":   # columns without checks between the others
        cols = random_cols(rng, 90, 12, [0, 0, 1, 3])
        return make_dem(cols + [[c] for c in range(12)], 12, 2)
    if name == "chain":   # consecutive columns share a check: a step per column in natural order
        return make_dem([[c, c + 1] for c in range(69)] + [[0]], 70, 3)
    if name == "wide":   # many disjoint columns: full steps, none left over, then a remainder
        return make_dem([[2 * j, 2 * j + 1] for j in range(163)] + [[4 * j] for j in range(50)], 326, 4)
    if name == "degree16":   # columns of up to 16 checks: two fill a step
        cols = random_cols(rng, 70, 40, [1, 5, 15, 16])
        return make_dem(cols + [[c] for c in range(40)], 40, 5)
    if name == "row255":   # one row of 255 entries, rows of one entry
        return make_dem([[0] if j < 100 else [0, 1 + j % 30] for j in range(255)] + [[31]], 32, 6)
    if name == "hard":   # two rows of one entry on the same column: hard constraints, infinite messages
        return make_dem([[0, 1, 2], [2, 3], [3, 4], [4], [2, 4]], 5, 7)
    raise KeyError(name)


@pytest.mark.parametrize("fp16", [False, True])
@pytest.mark.parametrize("name", ["one_by_one", "no_checks", "chain", "wide", "degree16", "row255", "hard"])
def test_steps_match_oracle(V, name, fp16):
    dm = problem(name)
    K, T, M, B = 3, 7, 2, 150
    perms = np.stack([np.arange(dm.n, dtype=np.uint32), *D.schedules(dm.n, K - 1, 3)])
    syn, _ = D.sample(dm, B, 9)
    r = oracle.decode(dm, perms, syn, T, 0.625, M, mode=oracle.FP16MSG if fp16 else oracle.FP32, nthreads=4)
    syn_t = torch.from_numpy(syn.view(np.int32)).cuda()
    for engine in (V.ENGINE_IMAGE, V.ENGINE_SUMMARY):
        for pair in (False, True):
            dec = V.Decoder(dm, K, perms, T=T, alpha=0.625, M=M, msg_fp16=fp16, engine=engine, pair_mode=pair)
            out = dec.decode(syn_t, want_soft=True)
            torch.cuda.synchronize()
            what = f"{name} fp16={fp16} engine={engine} pair={pair}"
            assert np.array_equal(out["corrections"].cpu().numpy().view(np.uint32), r["corrections"]), what
            assert np.array_equal(out["logical"].cpu().numpy().view(np.uint32), r["logical"]), what
            st = V.stats_to_numpy(out["stats"])
            for f in r["stats"].dtype.names:
                assert np.array_equal(st[f], r["stats"][f]), f"{what}: stats.{f}"
            a, b = out["soft"].cpu().numpy(), r["soft"].astype(np.float32)
            assert np.array_equal(a.view(np.uint32), b.view(np.uint32)), what
            dec.close()
