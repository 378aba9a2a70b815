"""Labels and coverage where the tensor-core score leaves the decision open.

Pixels lie at the same cosine (to FP32 rounding) of two or of three cluster
centres and otherwise apart, or at the bandwidth from a centre to within 1e-4:
two-mode ties take the reader's own exact test, three-mode ties the queue (a
few take a block each, thousands the tiled form), doubtful coverage the
reader's test. The reference is the FP64 cosine of the raw embeddings with the
modes that the run kept; the pixels' FP32 rounding leaves gaps of 1e-9 and more
there, seven digits above FP64's.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _frame(rng, n_tie, ways, d, cos_sum):
    """Three tight clusters at the first axes, then n_tie pixels at equal cosines to the first `ways`."""
    n_blob = max(60, n_tie)  # every centre is drawn
    eye = np.eye(d)
    blob = np.concatenate([synth.sample_vmf(rng, eye[k], 5000.0, n_blob) for k in range(3)])
    w = rng.standard_normal((n_tie, d))
    w[:, :3] = 0.0
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    centre = np.stack([blob[n_blob * k:n_blob * (k + 1)].sum(0) for k in range(3)])
    centre /= np.linalg.norm(centre, axis=1, keepdims=True)
    # the vector in the centres' span with the same cosine to each of them
    dual = np.linalg.pinv(centre[:ways]) @ np.ones(ways)
    p = cos_sum * dual + np.sqrt(1.0 - cos_sum**2 * (dual @ dual)) * (w - w @ np.linalg.pinv(centre) @ centre)
    return np.ascontiguousarray(np.concatenate([blob, p]).astype(np.float32))


def _cos(emb, modes):
    e, m = emb.astype(np.float64), modes.astype(np.float64)
    return (e / np.linalg.norm(e, axis=1, keepdims=True)) @ (m / np.linalg.norm(m, axis=1, keepdims=True)).T


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d", [16, 24])
@pytest.mark.parametrize("ways", [2, 3])
@pytest.mark.parametrize("n_tie", [40, 3000])
@pytest.mark.parametrize("batch", [False, True])
def test_ties_of_two_and_three_modes(ms_lib, n_tie, ways, d, precision, batch):
    import torch
    rng = np.random.default_rng(100 * d + 10 * ways + n_tie)
    emb = _frame(rng, n_tie, ways, d, 0.4)
    e = torch.from_numpy(emb).cuda()
    # merge_cos below the ties' cosine: a tie pixel drawn as a seed joins a centre's mode
    kw = dict(precision=precision, n_initial=100, max_rounds=1, merge_cos=0.3)
    if batch:
        b = ms_lib.ms_batch_create(ms_lib.ms_config_default(dim=d, **kw), [e], [None])
        ms_lib.ms_batch_run(b)
        labels, modes = b.labels[0].cpu().numpy(), np.array(ms_lib.ms_batch_modes(b, 0))
        b.close()
    else:
        r = ms_lib.cluster(e, **kw)
        labels, modes = r.labels.cpu().numpy(), r.modes.cpu().numpy()
    cos = _cos(emb, modes)
    top = np.sort(cos, axis=1)
    near = top[:, -1] - top[:, -ways] < 2e-5
    assert modes.shape[0] == 3 and near.sum() == n_tie  # the ties are there
    assert np.array_equal(labels, np.argmax(cos, axis=1))


def _band_frame(d):
    """One tight cluster and 200 pixels at 0.9 of its centre, few enough to hardly move it."""
    rng = np.random.default_rng(7 + d)
    blob = synth.sample_vmf(rng, np.eye(d)[0], 5000.0, 20000)
    centre = blob.sum(0) / np.linalg.norm(blob.sum(0))
    w = rng.standard_normal((200, d))
    w -= np.outer(w @ centre, centre)
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    return np.concatenate([blob, 0.9 * centre + np.sqrt(1 - 0.9**2) * w]).astype(np.float32)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d", [16, 24])
def test_coverage_at_the_bandwidth(ms_lib, d, precision):
    import torch
    emb, c = _band_frame(d), 0.9
    r = ms_lib.cluster(torch.from_numpy(emb).cuda(), precision=precision, n_initial=64, max_rounds=1,
                       bandwidth_cos=c, merge_cos=c)
    best = _cos(emb, r.modes.cpu().numpy()).max(axis=1)
    assert (np.abs(best - c) < 6e-5).sum() > 40
    drawn = np.zeros(len(emb), bool)
    drawn[r.stats["seed_log"]] = True
    assert r.stats["round_log"][0][3] == np.count_nonzero(~drawn & (best < c))
