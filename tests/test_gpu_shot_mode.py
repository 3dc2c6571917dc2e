"""One warp or team per shot, and shot mode's small batches as pairs, each held to the oracle bit for bit.

Shot mode runs a small batch as (shot, member) pairs unless its records may take no memory (vibe_set_pairs),
so the driver that large batches use is asked for here and checked to be the one that ran. Flooding and layered
members, mixed scaling factors, the order-lambda search, hard constraints, columns of more than 16 checks,
columns without checks, graphs wide enough for a team of eight warps, mixed batches; both engines, both
precisions, with and without soft output.
"""
import numpy as np
import pytest

import oracle
from paper_2508_15743_gb300 import circuit as C
from paper_2508_15743_gb300 import dem as D
from test_gpu_steps import make_dem, problem as step_problem, random_cols

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


def degree32():
    """Columns of up to 32 checks, which only the image engine takes: one fills a step."""
    rng = np.random.default_rng(17)
    return make_dem(random_cols(rng, 60, 40, [1, 7, 16, 17, 31, 32]) + [[c] for c in range(40)], 40, 18)


def team():
    """Sparse and wide: units of 8 x 32 edges keep their lanes at work, and the image fits no CTA."""
    rng = np.random.default_rng(19)
    m, n = 2000, 16000
    cols = [sorted(rng.choice(m, int(d), replace=False)) for d in rng.choice([2, 3, 3, 4], n)]
    cols += [[c, (c + 1) % m] for c in range(0, m, 2)]   # no row is empty
    rows = [[] for _ in range(m)]
    for j, c in enumerate(cols):
        for r in c:
            rows[r].append(j)
    H = D.CSR.from_rows([sorted(r) for r in rows], len(cols))
    L = D.CSR.from_rows([list(range(0, len(cols), 7))], len(cols))
    return D.DEM(H, L, rng.uniform(0.001, 0.006, len(cols)))


IMAGE, SUMMARY = 1, 2
MIX = np.array([0.5, 0.625, 0.75, 1.0, 0.875, 0.5625], np.float32)
CASES = {
    # name: (DEM builder, K, M, T, shots, engine, decoder options)
    "pheno_d9": (lambda: D.build_workload("cc666_d9_pheno"), 8, 3, 20, 400, IMAGE, {}),
    "pheno_d7_order3": (lambda: D.phenomenological_dem(7, 7, 0.015, 0.015), 6, 2, 12, 400, IMAGE, dict(lsd_order=3)),
    "mixed_schedules": (lambda: D.phenomenological_dem(5, 5, 0.02, 0.02), 6, 2, 12, 500, IMAGE,
                        dict(n_flood=2, n_layered=2, member_alpha=MIX)),
    "pheno488_d7": (lambda: D.phenomenological_dem(7, 7, 0.012, 0.012, "488"), 6, 3, 15, 400, IMAGE,
                    dict(member_alpha=MIX)),
    "degree32": (degree32, 3, 2, 7, 150, IMAGE, dict(lsd_order=2)),
    "degree16": (lambda: step_problem("degree16"), 3, 2, 7, 150, SUMMARY, dict(lsd_order=2)),
    "hard_image": (lambda: step_problem("hard"), 3, 2, 7, 150, IMAGE, {}),
    "hard_summary": (lambda: step_problem("hard"), 3, 2, 7, 150, SUMMARY, {}),
    "no_checks": (lambda: step_problem("no_checks"), 3, 2, 7, 150, SUMMARY, {}),
    "row255": (lambda: step_problem("row255"), 3, 2, 7, 150, SUMMARY, {}),
    "circuit_d5": (lambda: C.circuit_dem(5, 5, 0.003, noise="si1000", basis="X"), 6, 2, 12, 250, SUMMARY,
                   dict(lsd_order=3, member_alpha=MIX)),
    "team": (team, 3, 2, 5, 40, SUMMARY, dict(lsd_order=1)),
    "team_full": (team, 3, 2, 5, 700, SUMMARY, {}),   # a batch that fills the GPU: single warps
}


def check(V, out, r, what):
    assert np.array_equal(out["corrections"].cpu().numpy().view(np.uint32), r["corrections"]), what
    assert np.array_equal(out["logical"].cpu().numpy().view(np.uint32), r["logical"]), what
    st = V.stats_to_numpy(out["stats"])
    for f in r["stats"].dtype.names:
        assert np.array_equal(st[f], r["stats"][f]), f"{what}: stats.{f}"
    if out["soft"] is not None:
        assert np.array_equal(out["soft"].cpu().numpy().view(np.uint32),
                              r["soft"].astype(np.float32).view(np.uint32)), f"{what}: soft"


@pytest.mark.parametrize("fp16", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_both_drivers_match_oracle(V, name, fp16):
    build, K, M, T, B, engine, opt = CASES[name]
    dm = build()
    perms = D.schedules(dm.n, K, 23)
    syn, obs = D.sample(dm, B, 29)
    ref = {k: v for k, v in opt.items() if k in ("lsd_order", "n_flood", "n_layered", "member_alpha")}
    r = oracle.decode(dm, perms, syn, T, 0.625, M, mode=oracle.FP16MSG if fp16 else oracle.FP32, nthreads=8, **ref)
    syn_t = torch.from_numpy(syn.view(np.int32)).cuda()
    obs_t = torch.from_numpy(obs.view(np.int32)).cuda()
    dec = V.Decoder(dm, K, perms, T=T, M=M, msg_fp16=fp16, engine=engine, **opt)
    fails = int((r["logical"] != obs).any(axis=1).sum())
    for record_bytes, as_pairs in ((0, 0), (-1, 1)):
        dec.set_pairs(record_bytes)
        for soft in (True, False):
            cnt = torch.zeros(8, dtype=torch.int64, device="cuda")
            out = dec.decode(syn_t, observables=obs_t, want_soft=soft, counters=cnt)
            torch.cuda.synchronize()
            what = f"{name} fp16={fp16} pairs={as_pairs} soft={soft}"
            assert dec.pairs()["last"] == as_pairs, what
            assert dec.pairs()["team"] == (8 if name == "team" else 1), what
            check(V, out, r, what)
            cnt = cnt.tolist()
            assert cnt[V.CNT_SHOTS] == B and cnt[V.CNT_FAILURES] == fails, what
            assert cnt[V.CNT_LSD] == int(r["stats"]["lsd_invoked"].sum()), what
    dec.close()


@pytest.mark.parametrize("B,largest_team", [(90, 8), (2400, 1)])
def test_mixed_batch_drivers_match_oracle(V, B, largest_team):
    """An image-engine problem, a single-warp and a wide problem in one batch, shots out of order; the wide one
    runs with a team of eight warps unless its share of the batch fills the GPU."""
    probs = [(D.phenomenological_dem(5, 5, 0.02, 0.02), 5, 2, 10), (CASES["circuit_d5"][0](), 4, 2, 8),
             (team(), 3, 1, 4)]
    rng = np.random.default_rng(31)
    pid = (np.arange(B) % 3).astype(np.int32)
    rng.shuffle(pid)
    pid[7] = 5   # no such problem
    mw = max(D.words(p[0].m) for p in probs)
    syn = np.zeros((B, mw), np.uint32)
    refs = []
    for i, (dm, K, M, T) in enumerate(probs):
        rows = np.nonzero(pid == i)[0]
        s, _ = D.sample(dm, len(rows), 37 + i)
        syn[rows, :s.shape[1]] = s
        refs.append((rows, oracle.decode(dm, D.schedules(dm.n, K, 41 + i), s, T, 0.625, M, nthreads=8, want_soft=False)))
    decs = [V.Decoder(dm, K, D.schedules(dm.n, K, 41 + i), T=T, M=M, engine=IMAGE if i == 0 else SUMMARY)
            for i, (dm, K, M, T) in enumerate(probs)]
    mb = V.MixedBatch(decs)
    for record_bytes, as_pairs in ((0, 0), (-1, 1)):
        mb.set_pairs(record_bytes)
        out = mb.decode(torch.from_numpy(pid).cuda(), torch.from_numpy(syn.view(np.int32)).cuda())
        torch.cuda.synchronize()
        assert mb.pairs()["last"] == as_pairs and mb.pairs()["team"] == largest_team
        corr, st = out["corrections"].cpu().numpy().view(np.uint32), V.stats_to_numpy(out["stats"])
        for (rows, r), (dm, *_rest) in zip(refs, probs):
            assert np.array_equal(corr[rows][:, :D.words(dm.n)], r["corrections"])
            for f in r["stats"].dtype.names:
                assert np.array_equal(st[f][rows], r["stats"][f]), f
        assert st["status"][7] == V.VIBE_STATUS_BAD_PROBLEM and not corr[7].any()
    mb.close()
    for d in decs:
        d.close()


@pytest.mark.parametrize("sample", [8, 600])
def test_launch_search_of_a_wide_problem_keeps_the_bits(V, sample):
    """The search times the packing that a batch like its sample runs; small and large batches stay as they were."""
    dm = team()
    K = 3
    dec = V.Decoder(dm, K, D.schedules(dm.n, K, 23), T=4, M=2)
    syn, _ = D.sample(dm, 700, 43)
    syn = torch.from_numpy(syn.view(np.int32)).cuda()
    want = {B: dec.decode(syn[:B]) for B in (40, 700)}
    dec.autotune(syn[:sample])
    for B, largest in ((40, 8), (700, 1)):
        out = dec.decode(syn[:B])
        torch.cuda.synchronize()
        assert dec.pairs()["team"] == largest
        for k in ("corrections", "logical", "stats"):
            assert torch.equal(out[k], want[B][k]), (B, k)
    dec.close()


def test_pairs_wants_exactly_one_object(V):
    import ctypes
    out = V.vibe_pairs()
    assert V._lib.vibe_get_pairs(None, None, ctypes.byref(out)) == V.VIBE_ERR_INVALID
    assert V._lib.vibe_set_pairs(None, None, 0) == V.VIBE_ERR_INVALID
