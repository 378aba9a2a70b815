"""Batches around the 32 frames that a pass of the work lists' warp covers:
every frame's labels and seed-iterations are those of a run of its own.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 32, 33, 65])
def test_batch_sizes_around_a_warp(ms_lib, B):
    import torch
    frames = [synth.make_frame(300 + i, 1, 200 + 37 * (i % 7), 16, 200 + 37 * (i % 7), 2, 100.0, 0.2, 60.0, 200.0, 0.0)
              for i in range(B)]
    embs = [torch.from_numpy(f.emb).cuda() for f in frames]
    b = ms_lib.ms_batch_create(ms_lib.ms_config_default(n_initial=16), embs, [None] * B)
    try:
        ms_lib.ms_batch_run(b)
        for i in range(B):
            r = ms_lib.cluster(embs[i], n_initial=16, frame_id=i)
            assert np.array_equal(b.labels[i].cpu().numpy(), r.labels.cpu().numpy())
            assert ms_lib.ms_batch_stats(b, i)["seed_iters"] == r.stats["seed_iters"]
    finally:
        b.close()
