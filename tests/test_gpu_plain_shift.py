"""Window sums of the FP32 form against a kernel that shares nothing with it but
the split into chunks: ms_window_sums_static scans all pairs with FP32 dot products
(k_shift_fp32), while the form finds windows with tensor-core scores and skips
pieces of the score matrix.

A kept mode is the normalised sum over the window of a seed within tol = 1e-6 of
it, which is its own window unless a pixel lies that close to the window's edge:
modes with a pixel within 4e-6 of it (tol, and FP32's error in the scores) are left
out. For the others the scan's sums at the modes, normalised as the update does,
give the modes back bit for bit, and its counts are their supports. At most 256
seeds keep both to one seed tile and so to the same chunks, in which FP32 sums round
alike. The BF16 form is held to the scan's counts, and its modes to the worst case
of both sums: n additions of relative error 2^-24 in the scan, n / 16 of 2^-23 in the
tensor cores' accumulation.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _frame(n, seed):
    rng = np.random.default_rng(seed)
    centre = synth.uniform_sphere(rng, 6, 16)
    return np.concatenate([synth.sample_vmf(rng, centre[i * 6 // n], 60.0, 1) for i in range(n)]).astype(np.float32)


def _scan(ms_lib, modes, emb, c):
    import torch
    out = torch.empty((modes.shape[0], 17), dtype=torch.int64, device="cuda")
    ms_lib.ms_window_sums_static(modes, emb, out, c)
    torch.cuda.synchronize()
    acc = out.cpu().numpy()
    y = acc[:, :16].astype(np.float64)
    cos = modes.double() @ torch.nn.functional.normalize(emb.double(), dim=1).T
    clear = ((cos - c).abs() > 4e-6).all(1).cpu().numpy()
    assert clear.mean() > 0.5
    return (y / np.sqrt((y * y).sum(1))[:, None]).astype(np.float32), acc[:, 16], clear


@pytest.mark.parametrize("c", [-0.2, 0.3, 0.7, 0.9, 0.98])
@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 1000, 4097, 12001])
def test_modes_are_the_scan_of_their_windows(ms_lib, n, c):
    import torch
    emb = torch.from_numpy(_frame(n, n)).cuda()
    kw = dict(bandwidth_cos=c, merge_cos=max(c, 0.3), n_initial=200, max_rounds=1)
    r = ms_lib.cluster(emb, **kw)
    modes, count, clear = _scan(ms_lib, r.modes.contiguous(), emb, c)
    assert np.array_equal(count[clear], r.stats["support"][clear])
    assert np.array_equal(modes[clear], r.modes.cpu().numpy()[clear])
    r = ms_lib.cluster(emb, precision=ms_lib.MS_BF16, **kw)
    modes, count, clear = _scan(ms_lib, r.modes.contiguous(), emb, c)
    assert np.array_equal(count[clear], r.stats["support"][clear])
    tol = (n / 16 + 2) * 2.0 ** -23 + n * 2.0 ** -24
    assert np.abs(modes - r.modes.cpu().numpy())[clear].max() <= tol
