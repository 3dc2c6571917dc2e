"""The launch search times pair mode against one warp per shot, also on samples that shot mode runs as pairs.

Two samples below that line, one where a few shots hold K x T sweeps each (pairs win by far) and one of
empty shots (a pair of each member has to be taken, 1.5 million in all; one warp per shot wins by far), and what is
kept must be what then runs.
"""
import numpy as np
import pytest

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


SAMPLES = {
    # name: (distance, noise, K, M, T, shots, mode that must win)
    "hard_and_few": (5, 0.02, 16, 5, 30, 16, 1),
    "empty": (3, 0.01, 64, 1, 20, 24_000, 0),
}


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("name", sorted(SAMPLES))
def test_tuner_compares_the_modes_on_small_samples(V, name, mixed):
    d, p, K, M, T, B, mode = SAMPLES[name]
    dm = D.phenomenological_dem(d, d, p, p)
    syn = np.zeros((B, D.words(dm.m)), np.uint32) if name == "empty" else D.sample(dm, B, 11)[0]
    syn_t = torch.from_numpy(syn.view(np.int32)).cuda()
    pid = torch.zeros(B, dtype=torch.int32, device="cuda")
    dec = V.Decoder(dm, K, D.schedules(dm.n, K, 12), T=T, M=M)
    assert B <= dec.pairs()["shots"]
    obj = V.MixedBatch([dec]) if mixed else dec
    run = (lambda: obj.decode(pid, syn_t)) if mixed else (lambda: obj.decode(syn_t))
    want = run()
    assert obj.pairs()["last"] == 1   # shot mode runs it as pairs before the search
    if mixed:
        obj.autotune(pid, syn_t)
    else:
        obj.autotune(syn_t)
    assert obj.launch()["pair_mode"] == mode
    got = run()
    torch.cuda.synchronize()
    assert obj.pairs()["last"] == mode
    for k in ("corrections", "logical", "stats"):
        assert torch.equal(got[k], want[k]), k
    if mode == 0:
        assert obj.pairs()["held_bytes"] == 0   # the search's records are gone
    if mixed:
        obj.close()
    dec.close()


def test_large_sample_leaves_small_batches_as_pairs(V):
    dm = D.phenomenological_dem(3, 3, 0.0003, 0.0003)
    K, B = 64, 60_000
    syn_t = torch.zeros((B, D.words(dm.m)), dtype=torch.int32, device="cuda")
    dec = V.Decoder(dm, K, D.schedules(dm.n, K, 14), T=20, M=1)
    limit = dec.pairs()["shots"]
    assert limit < B
    dec.autotune(syn_t)
    assert dec.launch()["pair_mode"] == 0 and dec.pairs()["held_bytes"] == 0
    dec.decode(syn_t[:200])
    assert dec.pairs()["last"] == 1
    dec.close()
