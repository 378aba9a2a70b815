"""A context's whole life on its own stream while another stream of the process is
being captured (relaxed mode): the capture stays valid and its graph replays, the
labels are those of a run without it.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_contexts_during_a_capture(ms_lib, precision):
    import torch
    f = synth.make_frame(6, 1, 5000, 16, 5000, 5, 1000.0, 0.2, 60.0, 200.0, 0.0)
    e = torch.from_numpy(f.emb).cuda()
    ref = ms_lib.cluster(e, precision=precision).labels.cpu().numpy()
    cfg = ms_lib.ms_config_default(precision=precision)
    labels = torch.zeros(5000, dtype=torch.int32, device="cuda")
    x = torch.zeros(1000, device="cuda")
    own = torch.cuda.Stream()
    held = ms_lib.ms_create(cfg, e, None, own)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode="relaxed"):
        x.add_(1.0)
        held.close()
        ctx = ms_lib.ms_create(cfg, e, None, own)
        ms_lib.ms_run(ctx, labels)
        ctx.close()
        x.add_(1.0)
    assert np.array_equal(labels.cpu().numpy(), ref)
    g.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 2000.0
