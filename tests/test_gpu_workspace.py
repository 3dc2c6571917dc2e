"""The workspace promise: a batch no larger than an earlier one allocates nothing, whatever came between.

Batch sizes and calls with and without soft output are mixed on one handle; free device memory must stay as it
is, and a graph captured after the warm-up must replay to the same bits. The buffers at stake are far above the
allocator's granularity (140 KB of members' records per shot here).
"""
import numpy as np
import pytest

from paper_2508_15743_gb300 import circuit as C
from paper_2508_15743_gb300 import dem as D

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

IMAGE, SUMMARY = 1, 2


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_15743_gb300 import build
    build.build_library()
    from paper_2508_15743_gb300 import vibe
    return vibe


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


class Calls:
    """Decodes of the first B shots of one batch into buffers made beforehand."""

    def __init__(self, V, dm, K, shots, **kw):
        self.dec = V.Decoder(dm, K, D.schedules(dm.n, K, 3), T=8, M=2, **kw)
        syn, _ = D.sample(dm, shots, 5)
        self.syn = torch.from_numpy(syn.view(np.int32)).cuda()
        self.out = {s: dict(corrections=torch.zeros((shots, self.dec.nw), dtype=torch.int32, device="cuda"),
                            logical=torch.zeros((shots, self.dec.kw), dtype=torch.int32, device="cuda"),
                            stats=torch.zeros((shots, 12), dtype=torch.uint8, device="cuda"),
                            soft=torch.zeros((shots, dm.n), device="cuda") if s else None) for s in (False, True)}

    def __call__(self, B, soft=False):
        out = {k: v if v is None else v[:B] for k, v in self.out[soft].items()}
        self.dec.decode(self.syn[:B], out=out)
        return out


PROBLEMS = {
    "summary": (lambda: C.circuit_dem(5, 5, 0.003, noise="si1000", basis="X"), SUMMARY),
    "image": (lambda: D.phenomenological_dem(9, 9, 0.01, 0.01), IMAGE),
}


@pytest.mark.parametrize("pair", [False, True])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_smaller_batches_between_allocate_nothing(V, name, pair):
    build, engine = PROBLEMS[name]
    run = Calls(V, build(), 16, 1000, engine=engine, pair_mode=pair)
    run(1000)
    run(10, soft=True)     # a first soft output may grow the scratch
    before = free_bytes()
    for B, soft in ((1000, False), (10, True), (1, False), (1000, False), (7, True), (999, False)):
        run(B, soft)
    assert free_bytes() == before
    run.dec.close()


def test_capture_after_mixed_warm_up_replays_the_same_bits(V):
    build, engine = PROBLEMS["summary"]
    run = Calls(V, build(), 16, 1000, engine=engine)
    want = {k: v.clone() for k, v in run(1000).items() if v is not None}
    run(10, soft=True)
    run(1000)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = run(1000)
    run(10, soft=True)
    run(500)
    for v in out.values():
        if v is not None:
            v.zero_()
    g.replay()
    torch.cuda.synchronize()
    for k, v in want.items():
        assert torch.equal(out[k], v), k
    run.dec.close()


def test_records_are_held_only_for_batches_that_run_as_pairs(V):
    build, engine = PROBLEMS["image"]
    run = Calls(V, build(), 4, 60_000, engine=engine)
    limit = run.dec.pairs()["shots"]
    assert 0 < limit < 60_000
    run(60_000)                       # one warp per shot: no records
    p = run.dec.pairs()
    assert p["last"] == 0 and p["held_bytes"] == 0
    before = free_bytes()
    run(100)                          # no larger than an earlier one: nothing may be allocated for it
    assert run.dec.pairs()["last"] == 0 and free_bytes() == before
    run.dec.close()
    run = Calls(V, build(), 4, 60_000, engine=engine)
    run(100)
    held = run.dec.pairs()["held_bytes"]
    assert run.dec.pairs()["last"] == 1 and held > 0
    run(limit)
    assert run.dec.pairs()["last"] == 1 and run.dec.pairs()["held_bytes"] > held
    run(60_000)
    assert run.dec.pairs()["last"] == 0
    before = free_bytes()
    for B in (100, limit):            # the records stayed
        run(B)
        assert run.dec.pairs()["last"] == 1
    assert free_bytes() == before
    run.dec.close()


def test_first_small_batch_under_capture_allocates_nothing(V):
    build, engine = PROBLEMS["image"]
    run = Calls(V, build(), 4, 60_000, engine=engine)
    run(60_000)
    want = {k: v.clone() for k, v in run(300).items() if v is not None}
    run.dec.set_pairs(-1)             # the next small batch outside a capture would get records
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = run(300)
    assert run.dec.pairs()["last"] == 0 and run.dec.pairs()["held_bytes"] == 0
    for v in out.values():
        if v is not None:
            v.zero_()
    g.replay()
    torch.cuda.synchronize()
    for k, v in want.items():
        assert torch.equal(out[k], v), k
    run.dec.close()


@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_first_soft_output_of_a_small_batch_runs_as_pairs(V, name):
    build, engine = PROBLEMS[name]
    run = Calls(V, build(), 16, 1000, engine=engine)
    run(1000)
    run(50, soft=True)
    assert run.dec.pairs()["last"] == 1
    before = free_bytes()
    for B, soft in ((1000, True), (1000, False), (3, True)):   # the posteriors' records are there for all of them
        run(B, soft)
        assert run.dec.pairs()["last"] == 1
    assert free_bytes() == before
    run.dec.close()


@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_posteriors_count_in_the_bound(V, name):
    build, engine = PROBLEMS[name]
    run = Calls(V, build(), 16, 1000, engine=engine)
    run(500)
    per_shot = run.dec.pairs()["held_bytes"] / 500
    bound = int(per_shot * 800)
    run.dec.set_pairs(bound)
    p = run.dec.pairs()
    assert p["shots"] == 800 and p["shots_soft"] < 500   # a posterior is as long as the term kept without it
    for B, soft, as_pairs in ((800, False, 1), (1000, False, 0), (p["shots_soft"], True, 1), (500, True, 0)):
        run(B, soft)
        q = run.dec.pairs()
        assert q["last"] == as_pairs, (B, soft)
        assert q["held_bytes"] <= bound, (B, soft)
    run.dec.close()


def test_mixed_scratch_is_sized_by_team(V):
    """A batch of a narrow and a wide problem: the many one-warp teams don't get the wide problem's scratch."""
    from test_gpu_shot_mode import team

    def used(call):
        before = free_bytes()
        call()
        return before - free_bytes()

    decs, alone = [], 0
    for dm in (PROBLEMS["summary"][0](), team()):
        run = Calls(V, dm, 4, 1, engine=SUMMARY)
        run.dec.set_pairs(0)
        run(1)                # kernels are loaded now
        run.dec.close()
        run = Calls(V, dm, 4, 1, engine=SUMMARY)
        run.dec.set_pairs(0)
        alone += used(lambda: run(1))
        decs.append(run.dec)
    first = V.MixedBatch(decs)
    syn = torch.zeros((2, first.mw), dtype=torch.int32, device="cuda")
    pid = torch.arange(2, dtype=torch.int32, device="cuda")
    first.decode(pid, syn)
    first.close()
    mb = V.MixedBatch(decs)
    out = dict(corrections=torch.zeros((2, mb.nw), dtype=torch.int32, device="cuda"),
               logical=torch.zeros((2, mb.kw), dtype=torch.int32, device="cuda"),
               stats=torch.zeros((2, 12), dtype=torch.uint8, device="cuda"))
    assert used(lambda: mb.decode(pid, syn, out=out)) <= alone + (64 << 20)   # its buffers are rounded up, too
    mb.close()
    for d in decs:
        d.close()
