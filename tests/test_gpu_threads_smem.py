"""Host threads whose launches of one kernel need different amounts of shared
memory: the limit is a process-wide attribute, and no launch may find it
lowered by another thread."""
import threading

import numpy as np
import pytest

import iesh_inputs as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["float64", "float32"])
def test_two_sizes_from_two_threads(dtype):
    import torch
    from paper_2212_00518_gb300 import eocc as E
    # 54 to 133 KB (FP64) of shared memory per block
    sizes = (1600, 4000) if dtype == "float64" else (3600, 4000)
    Ne = 40 if dtype == "float64" else 700
    work = []
    for M in sizes:
        wl = W.eocc_workload(M=M, B=2, Ne=Ne)
        work.append((E.EOccModel(wl), torch.tensor(wl["x"], dtype=getattr(torch, dtype), device="cuda"),
                     torch.tensor(wl["theta"], dtype=getattr(torch, dtype), device="cuda")))
    errors, out = [], [None, None]
    start = threading.Barrier(2)

    def loop(i):
        try:
            model, x, th = work[i]
            start.wait(30)
            for _ in range(400):
                out[i] = model.forward(x, th)[0]
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for (model, x, th), e in zip(work, out):
        assert np.array_equal(model.forward(x, th)[0].cpu().numpy(), e.cpu().numpy())
        model.close()
