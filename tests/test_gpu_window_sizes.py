"""Window sizes, seeds and labels of both forms against the FP64 oracle, from
windows of one pixel to windows of the whole frame and for bandwidths on both
sides of zero, at sizes around a 128-pixel tile: the rows that pad a frame's
last tile belong to no window, whatever the bandwidth.

Every input is the first of its seeds whose decisions (windows, coverage,
merge, labels) the oracle finds at least 1e-5 from their thresholds. FP32 dot
products of unit vectors are within 4e-6 of those of the oracle (at most 33
roundings of 2^-24 each, and the rounding of both vectors), so all counts are
compared for equality.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

MARGIN = 1e-5


def _case(n, c, d):
    for seed in range(400):
        rng = np.random.default_rng((seed, n, d, int(1000 * c) + 1000))
        centre = synth.uniform_sphere(rng, 3, d)
        P = np.concatenate([synth.sample_vmf(rng, centre[i % 3], 40.0, 1) for i in range(n)]).astype(np.float32)
        ref = oracle.run(P, bandwidth_cos=c, merge_cos=max(c, 0.5))
        st = ref.stats
        if min(st["min_window_margin"], st["min_cover_margin"], st["min_merge_margin"],
               np.nanmin(ref.label_margin)) > MARGIN:
            return P, ref
    raise AssertionError("no input with clear decisions")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d", [16, 24])
@pytest.mark.parametrize("c", [-0.5, -0.2, -0.01, 0.0, 0.5, 0.999])
@pytest.mark.parametrize("n", [1, 65, 127, 128, 129, 300])
def test_counts_equal_the_oracle(ms_lib, n, c, d, precision):
    import torch
    P, ref = _case(n, c, d)
    e = torch.from_numpy(P).cuda()
    kw = dict(bandwidth_cos=c, merge_cos=max(c, 0.5), precision=precision)
    r = ms_lib.cluster(e, **kw)
    assert np.array_equal(r.stats["support"], ref.support)
    assert np.array_equal(r.stats["seed_log"], ref.seed_log)
    assert np.array_equal(r.stats["round_log"], ref.round_log)
    assert r.stats["seed_iters"] == ref.stats["seed_iters"]
    assert np.array_equal(r.labels.cpu().numpy(), ref.labels)
    b = ms_lib.ms_batch_create(ms_lib.ms_config_default(dim=d, **kw), [e, e[: (n + 1) // 2].clone()], [None, None])
    try:
        ms_lib.ms_batch_run(b)
        assert np.array_equal(b.labels[0].cpu().numpy(), ref.labels)
        assert ms_lib.ms_batch_stats(b, 0)["seed_iters"] == ref.stats["seed_iters"]
        assert np.array_equal(ms_lib.ms_batch_modes(b, 0), r.modes.cpu().numpy())
    finally:
        b.close()
