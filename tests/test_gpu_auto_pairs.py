"""Shot mode runs small batches as (shot, member) pairs and large ones with a warp per shot: the same bits.

A batch of more shots than the pair limit (eight per resident warp) is decoded at once and again in
small slices; both must agree bit for bit, and a sample of them with the oracle.
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


@pytest.mark.parametrize("fp16", [False, True])
@pytest.mark.parametrize("engine", [1, 2])
def test_large_batch_equals_small_ones(V, engine, fp16):
    dm = D.phenomenological_dem(3, 3, 0.03, 0.03)
    K, T, M, B, part = 5, 12, 2, 100_000, 7_001
    perms = D.schedules(dm.n, K, 2)
    syn, _ = D.sample(dm, B, 4)
    syn_t = torch.from_numpy(syn.view(np.int32)).cuda()
    dec = V.Decoder(dm, K, perms, T=T, M=M, msg_fp16=fp16, engine=engine)
    limit = 8 * 64 * dec.launch()["num_sms"]   # at most 64 warps are resident on an SM
    assert part < B and limit < B
    whole = dec.decode(syn_t, want_soft=True)
    for lo in (0, part, B - 33):
        hi = min(B, lo + part)
        few = dec.decode(syn_t[lo:hi].contiguous(), want_soft=True)
        for k in ("corrections", "logical", "stats"):
            assert torch.equal(few[k], whole[k][lo:hi]), k
        assert torch.equal(few["soft"].view(torch.int32), whole["soft"][lo:hi].view(torch.int32))
    r = oracle.decode(dm, perms, syn[:500], T, 0.625, M, mode=oracle.FP16MSG if fp16 else oracle.FP32, nthreads=4)
    assert np.array_equal(whole["corrections"][:500].cpu().numpy().view(np.uint32), r["corrections"])
    st = V.stats_to_numpy(whole["stats"][:500])
    for f in r["stats"].dtype.names:
        assert np.array_equal(st[f], r["stats"][f]), f
    dec.close()
