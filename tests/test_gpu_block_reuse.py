"""Workspace blocks that pass from one context to the next: labels stay those
of a context of its own, over sizes that do and do not fit the blocks left, on
several threads and streams at once, and the memory kept stays bounded.
"""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_contexts_of_changing_sizes(ms_lib, precision):
    import torch
    frames = [synth.make_frame(i, 1, n, 16, n, min(3, n), n / min(3, n), 0.2, 60.0, 200.0, 0.0)
              for i, n in enumerate((5000, 700, 2600, 4999, 1, 5000))]
    embs = [torch.from_numpy(f.emb).cuda() for f in frames]
    first = [ms_lib.cluster(e, precision=precision).labels.cpu().numpy() for e in embs]
    for order in ((5, 1, 0, 4, 2, 3), (3, 2, 1, 0, 5, 4)):
        held = ms_lib.ms_create(ms_lib.ms_config_default(precision=precision), embs[0], None)  # keeps its block
        for i in order:
            assert np.array_equal(ms_lib.cluster(embs[i], precision=precision).labels.cpu().numpy(), first[i])
        lab = torch.empty(5000, dtype=torch.int32, device="cuda")
        ms_lib.ms_run(held, lab)
        held.close()
        assert np.array_equal(lab.cpu().numpy(), first[0])


def test_threads_with_their_own_streams(ms_lib):
    import torch
    frames = [synth.make_frame(20 + i, 1, 3000 + 400 * i, 16, 3000 + 400 * i, 4, 800.0, 0.2, 60.0, 200.0, 0.0)
              for i in range(4)]
    embs = [torch.from_numpy(f.emb).cuda() for f in frames]
    first = [ms_lib.cluster(e).labels.cpu().numpy() for e in embs]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(6):
                if not np.array_equal(ms_lib.cluster(embs[i]).labels.cpu().numpy(), first[i]):
                    bad.append(i)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert bad == []


def test_kept_memory_is_bounded(ms_lib):
    import torch
    e = torch.nn.functional.normalize(torch.randn(600000, 16, device="cuda", generator=torch.Generator("cuda").manual_seed(1)))
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    for n in (600000, 150000, 300000, 40000, 75000, 20000, 9000, 600000, 4000, 2000, 1000, 500):
        ms_lib.ms_create(ms_lib.ms_config_default(), e[:n], None).close()
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    assert free0 - free1 <= (512 << 20) + (64 << 20)  # 64 MB for the driver's rounding
