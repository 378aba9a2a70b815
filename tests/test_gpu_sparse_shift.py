"""The shift over the pieces of the score matrix that hold windows, and the
seed selection in pixel order, at the sizes where their splits end.

* Selection: the seeds and their draw order are the oracle's at the borders of
  its one-CTA form (4096 pixels), of a block of 1024 and of a single pixel.
* Batches with many short work items per CTA (one pixel tile each, every
  iteration) equal single-frame runs bit for bit, in every warp arrangement: a
  CTA's roles pass from item to item at their own pace.
* Windows from a single pixel to the whole frame, so that no piece, some and
  all of them hold pairs: the BF16 form's supports are the exact window sizes.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _cuda(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n", [1, 2, 1023, 1025, 4096, 4097, 5121])
@pytest.mark.parametrize("precision", [0, 1])
def test_selection_in_draw_order(ms_lib, n, precision):
    f = synth.make_frame(n + 3, 1, n, 16, n, max(1, n // 700), max(1.0, n / max(1, n // 700)), 0.2, 60.0, 200.0, 0.0)
    r = ms_lib.cluster(_cuda(f.emb), precision=precision, n_initial=37)
    ref = oracle.run(f.emb, n_initial=37)
    assert np.array_equal(r.stats["seed_log"], ref.seed_log)
    assert np.array_equal(r.stats["round_log"], ref.round_log)
    assert np.array_equal(r.stats["support"], ref.support)


@pytest.mark.parametrize("shape", range(8))
def test_batch_of_short_items_equals_single_frames(ms_lib, shape):
    # five frames of 130..215 pixel tiles: the first rounds give every CTA four
    # or five items of one tile, from different frames
    frames = [synth.make_frame(40 + i, 260, 260, 16, n, 12, n / 12.0, 0.3, 30.0, 200.0, 0.02)
              for i, n in enumerate((27602, 16906, 22001, 17003, 25000))]
    embs, masks = [_cuda(f.emb) for f in frames], [_cuda(f.mask) for f in frames]
    b = ms_lib.ms_batch_create(ms_lib.ms_config_default(precision=ms_lib.MS_BF16, tc_shape=shape), embs, masks)
    ms_lib.ms_batch_run(b)
    for i in range(len(frames)):
        r = ms_lib.cluster(embs[i], masks[i], precision=ms_lib.MS_BF16, frame_id=i)
        assert np.array_equal(b.labels[i].cpu().numpy(), r.labels.cpu().numpy())
        assert np.array_equal(ms_lib.ms_batch_modes(b, i), r.modes.cpu().numpy())
        assert ms_lib.ms_batch_stats(b, i)["seed_iters"] == r.stats["seed_iters"]
    b.close()


@pytest.mark.parametrize("n", [1, 127, 128, 129, 700])
@pytest.mark.parametrize("c", [-0.2, 0.0, 0.5, 0.9, 0.999])
@pytest.mark.parametrize("d", [16, 24])
def test_windows_of_every_density(ms_lib, n, c, d):
    rng = np.random.default_rng(1000 * n + d)
    centre = synth.uniform_sphere(rng, 3, d)
    P = np.concatenate([synth.sample_vmf(rng, centre[i % 3], 40.0, 1) for i in range(n)]).astype(np.float32)
    kw = dict(bandwidth_cos=c, merge_cos=max(c, 0.5))
    f = ms_lib.cluster(_cuda(P), **kw)
    b = ms_lib.cluster(_cuda(P), precision=ms_lib.MS_BF16, **kw)
    assert np.array_equal(f.stats["seed_log"], b.stats["seed_log"])
    if c > 0:  # at c <= 0 the padding rows of the last tile count
        assert np.array_equal(f.stats["support"], b.stats["support"])
        assert np.array_equal(f.labels.cpu().numpy(), b.labels.cpu().numpy())
