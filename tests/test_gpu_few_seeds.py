"""Selection of a few seeds by one CTA, which ranks them among themselves, at the
sizes where it starts (above 4096 pixels), takes a second seed per thread (1024)
and ends (2048 seeds), and on frames so covered that it passes many positions or
leaves the selection to the passes over all pixels. Seeds, draw order, rounds,
iterations and supports equal the oracle's.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _check(ms_lib, emb, precision, **kw):
    import torch
    e = torch.from_numpy(emb).cuda()
    r = ms_lib.cluster(e, precision=precision, **kw)
    ref = oracle.run(emb, **kw)
    assert np.array_equal(r.stats["seed_log"], ref.seed_log)
    assert np.array_equal(r.stats["round_log"], ref.round_log)
    assert np.array_equal(r.stats["support"], ref.support)
    assert r.stats["seed_iters"] == ref.stats["seed_iters"]
    b = ms_lib.ms_batch_create(ms_lib.ms_config_default(dim=emb.shape[1], precision=precision, **kw), [e], [None])
    try:
        ms_lib.ms_batch_run(b)
        assert ms_lib.ms_batch_stats(b, 0)["seed_iters"] == ref.stats["seed_iters"]
        assert np.array_equal(ms_lib.ms_batch_modes(b, 0), r.modes.cpu().numpy())
    finally:
        b.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_initial", [1, 3, 1023, 1024, 1025, 2047, 2048, 2049])
def test_seed_counts_around_its_limits(ms_lib, n_initial, precision):
    f = synth.make_frame(n_initial, 1, 4500, 16, 4500, 9, 500.0, 0.1, 2000.0, 3000.0, 0.0)
    _check(ms_lib, f.emb, precision, n_initial=n_initial, max_rounds=3)


@pytest.mark.parametrize("n_initial", [1500, 2048])
def test_two_seeds_a_thread_on_a_large_frame(ms_lib, n_initial):
    f = synth.make_frame(5, 1, 230000, 16, 230000, 20, 11500.0, 0.1, 2000.0, 3000.0, 0.0)
    for precision in (0, 1):
        _check(ms_lib, f.emb, precision, n_initial=n_initial, max_rounds=1)


@pytest.mark.parametrize("precision", [0, 1])
def test_scattered_uncovered_pixels(ms_lib, precision):
    """One cluster covers all but 60 of 20,000 pixels: later rounds look for them over the whole frame."""
    rng = np.random.default_rng(11)
    emb = synth.sample_vmf(rng, np.eye(16)[0], 5000.0, 20000)
    emb[rng.choice(20000, 60, replace=False)] = synth.uniform_sphere(rng, 60, 16)
    _check(ms_lib, emb.astype(np.float32), precision, n_initial=4)
