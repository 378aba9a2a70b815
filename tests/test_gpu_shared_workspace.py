"""Arrays of a context that share memory, at the sizes where their uses come
closest: every pixel a seed, a candidate and a mode (the candidates fill what the
modes leave), modes of earlier rounds and conflict lists in the rows of pixels that
coverage and the next round read again, labels between rounds. Results equal the
oracle's; batches of such frames equal single frames.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _spread(n, d, seed):
    """n directions with no two within 0.9 of one another, then near copies of every third."""
    rng = np.random.default_rng(seed)
    P = synth.uniform_sphere(rng, n, d)
    P[1::3] = P[0::3][: len(P[1::3])] + 0.02 * rng.standard_normal((len(P[1::3]), d)) / np.sqrt(d)
    return np.ascontiguousarray(P.astype(np.float32))


def _equal(r, ref):
    assert np.array_equal(r.stats["support"], ref.support)
    assert np.array_equal(r.stats["seed_log"], ref.seed_log)
    assert np.array_equal(r.stats["round_log"], ref.round_log)
    assert np.array_equal(r.labels.cpu().numpy(), ref.labels)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d", [16, 32])
@pytest.mark.parametrize("n", [1, 128, 129, 1000])
@pytest.mark.parametrize("kw", [dict(all_seeds=1), dict(n_initial=100), dict(n_initial=7)])
def test_every_pixel_a_mode(ms_lib, kw, n, d, precision):
    import torch
    emb = _spread(n, d, n + d)
    _equal(ms_lib.cluster(torch.from_numpy(emb).cuda(), precision=precision, **kw), oracle.run(emb, **kw))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d", [16, 24])
def test_labels_between_rounds(ms_lib, d, precision):
    import torch
    f = synth.make_frame(3, 40, 50, d, 1500, 12, 125.0, 0.3, 60.0, 200.0, 0.02)
    e, m = torch.from_numpy(f.emb).cuda(), torch.from_numpy(f.mask).cuda()
    ref = ms_lib.cluster(e, m, precision=precision)
    ctx = ms_lib.ms_create(ms_lib.ms_config_default(dim=d, precision=precision), e, m)
    labels = torch.empty(len(f.emb), dtype=torch.int32, device="cuda")
    while ms_lib.ms_seed_batch(ctx) > 0:
        ms_lib.ms_iterate(ctx)
        k, _ = ms_lib.ms_merge_modes(ctx)
        modes = torch.empty((k, d), dtype=torch.float32, device="cuda")
        ms_lib.ms_label(ctx, labels, modes)
        got = (e @ modes.T / e.norm(dim=1, keepdim=True)).double().cpu().numpy()
        fg = f.mask != 0
        assert (got[fg, labels.cpu().numpy()[fg]] >= got[fg].max(1) - 1e-5).all()
    assert torch.equal(labels, ref.labels) and torch.equal(modes, ref.modes)
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d", [16, 32])
@pytest.mark.parametrize("kw", [dict(all_seeds=1), dict(n_initial=60)])
def test_batches_of_such_frames(ms_lib, kw, d, precision):
    import torch
    embs = [torch.from_numpy(_spread(n, d, 7 * n)).cuda() for n in (1, 300, 129, 1000, 128, 2, 640)]
    embs.append(torch.from_numpy(synth.make_frame(4, 1, 900, d, 900, 3, 300.0, 0.1, 500.0, 900.0, 0.0).emb).cuda())
    b = ms_lib.ms_batch_create(ms_lib.ms_config_default(dim=d, precision=precision, **kw), embs, [None] * len(embs))
    try:
        for _ in range(2):  # the second run finds what the first left
            ms_lib.ms_batch_run(b)
            for f, e in enumerate(embs):
                r = ms_lib.cluster(e, precision=precision, frame_id=f, **kw)
                assert torch.equal(b.labels[f], r.labels)
                assert np.array_equal(ms_lib.ms_batch_modes(b, f), r.modes.cpu().numpy())
                assert ms_lib.ms_batch_stats(b, f)["seed_iters"] == r.stats["seed_iters"]
    finally:
        b.close()


@pytest.mark.parametrize("n_pix", [1, 30, 127])
def test_selftest_of_few_pixels(ms_lib, n_pix):
    import torch
    rng = np.random.default_rng(n_pix)
    P = synth.uniform_sphere(rng, n_pix, 16).astype(np.float32)
    X = synth.uniform_sphere(rng, 128, 16).astype(np.float32)
    S, acc = ms_lib.ms_tc_selftest(torch.from_numpy(X).cuda(), torch.from_numpy(P).cuda(), 0.3)
    cos = X.astype(np.float64) @ P.astype(np.float64).T
    clear = (np.abs(cos - 0.3) > 1e-5).all(1)
    assert np.array_equal(acc[clear, 16], (cos >= 0.3).sum(1)[clear])
