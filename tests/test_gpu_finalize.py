"""The end of a shift iteration at the sizes where its splits end: 32 seeds to
a block, a tile of 128 masks (4096 seeds) to a pass of the list's writer, and
steps that FP32 settles (far from tol), leaves to FP64 (tol below 1e-15) or
that never converge by the early stop (gamma = 1). Seeds, their iteration
count and the windows they end on equal the oracle's.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _run(ms_lib, f, batch, **kw):
    import torch
    e = torch.from_numpy(f.emb).cuda()
    if not batch:
        r = ms_lib.cluster(e, **kw)
        return r.stats["seed_iters"], r.stats["support"], r.labels.cpu().numpy()
    b = ms_lib.ms_batch_create(ms_lib.ms_config_default(dim=f.emb.shape[1], **kw), [e], [None])
    try:
        ms_lib.ms_batch_run(b)
        return ms_lib.ms_batch_stats(b, 0)["seed_iters"], None, b.labels[0].cpu().numpy()
    finally:
        b.close()


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("d", [16, 20])
@pytest.mark.parametrize("n_initial", [1, 31, 32, 33, 129])
def test_seed_counts_around_a_block(ms_lib, n_initial, d, batch):
    f = synth.make_frame(n_initial + d, 1, 600, d, 600, 3, 200.0, 0.1, 100.0, 300.0, 0.0)
    it, sup, lab = _run(ms_lib, f, batch, n_initial=n_initial)
    ref = oracle.run(f.emb, n_initial=n_initial)
    assert np.array_equal(lab, ref.labels)
    assert it == ref.stats["seed_iters"]
    assert sup is None or np.array_equal(sup, ref.support)


@pytest.mark.parametrize("n", [4095, 4097, 8200])
def test_lists_longer_than_one_tile_of_masks(ms_lib, n):
    f = synth.make_frame(n, 1, n, 16, n, 4, n / 4.0, 0.1, 100.0, 300.0, 0.0)
    it, sup, lab = _run(ms_lib, f, False, all_seeds=1)
    ref = oracle.run(f.emb, all_seeds=1)
    assert it == ref.stats["seed_iters"] and np.array_equal(sup, ref.support) and np.array_equal(lab, ref.labels)


@pytest.mark.parametrize("tol", [1e-16, 1e-6, 1e-3, 10.0])
def test_step_tolerances(ms_lib, tol):
    f = synth.make_frame(9, 1, 900, 16, 900, 4, 225.0, 0.1, 100.0, 300.0, 0.0)
    it, sup, lab = _run(ms_lib, f, False, tol=tol, gamma=1.0, max_iter=40)
    ref = oracle.run(f.emb, tol=tol, gamma=1.0, max_iter=40)
    assert it == ref.stats["seed_iters"] and np.array_equal(sup, ref.support) and np.array_equal(lab, ref.labels)
