"""The service's device-memory budget with the members' records that shot mode's small batches use."""
import gc

import numpy as np
import pytest

from paper_2508_15743_gb300 import service as S


@pytest.mark.parametrize("room", [0, 99, 100, 12_345, 1 << 33])
@pytest.mark.parametrize("pipelines", [1, 2, 3])
def test_split_stays_within_the_room_and_records_take_an_eighth_of_it(room, pipelines):
    mb, records = S.split_budget(room, pipelines, 50, 4096)
    assert records >= 0 and pipelines * (50 * mb + records) <= room
    assert mb == 4096 or records < room // pipelines // 8 + 50


def test_split_of_no_room():
    assert S.split_budget(-5, 2, 50, 10) == (0, 0)


@pytest.mark.gpu
@pytest.mark.parametrize("max_batch", [2048, 1 << 22])
def test_service_stays_within_its_budget(max_batch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_15743_gb300 import build
    build.build_library()
    from paper_2508_15743_gb300 import vibe as V
    gc.collect()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    svc, backend, decs, dems = S.build_service(["pheno_d9"], 1 << 30, fp16=False, max_batch=max_batch, seed=3)
    b = svc.budget
    assert b["used_bytes"] <= b["budget_bytes"]
    assert b["max_batch"] == 2048 or max_batch > 2048
    if max_batch == 2048:   # room is left: small batches run as pairs after the warm-up
        backend.launch(0, np.zeros(16, np.int32), np.zeros((16, backend.mw), np.uint32))
        torch.cuda.synchronize()
        assert V.vibe_get_pairs(b=backend.handles[0])["last"] == 1
    free = torch.cuda.mem_get_info()[0]
    for i, n in enumerate((1, 300, b["max_batch"])):   # serving allocates nothing
        backend.launch(i % 2, np.zeros(n, np.int32), np.zeros((n, backend.mw), np.uint32))
        torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    backend.close()
    for d in decs:
        d.close()
