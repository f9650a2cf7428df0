"""Subband spectra of candidates whose windows leave the beam at either end, lie
inside it by one sample, or miss it, for bins of one to 64 samples (read a sample or
a word at a time), and of subbands with more channels than share offsets: whole
numbers, compared exactly."""
import numpy as np
import pytest
import torch

import paper_2606_27262_gb300 as sp
import synth
from paper_2606_27262_gb300 import build as spbuild

pytestmark = pytest.mark.gpu

WIDTHS = [1, 8, 12, 16, 28, 32, 36, 64, 100, 256]  # bins of 1, 2, 3, 4, 7, 8, 9, 16, 25, 64 samples


@pytest.mark.parametrize("nchan,n_in,t_in,cases", [(512, 2003, 30, 60), (256, 9001, 513, 30), (76800, 901, 7, 12)])
def test_windows_at_the_ends_of_the_beam(nchan, n_in, t_in, cases):
    spbuild.build()
    rng = np.random.default_rng(nchan + t_in)
    plan = sp.Plan(synth.band_freqs(nchan), synth.TSAMP, [0.0, 9.0, 30.0], shape=1)
    delays = plan.delays()
    x = rng.integers(0, 256, size=(n_in, nchan), dtype=np.uint8)
    staged = sp.staged_buffer(nchan, n_in)
    sp.stage_input(torch.from_numpy(x).cuda(), staged)
    c = np.zeros((cases, 4), np.int32)
    for i in range(cases):
        w = WIDTHS[i % len(WIDTHS)]
        dec, dm, s = max(1, w // 4), int(rng.integers(0, 3)), int(rng.integers(0, 256))
        d = delays[dm, s * (nchan // 256)]
        first = (-d, -d - int(rng.integers(1, 9)), n_in - d - t_in * dec, n_in - d - t_in * dec + int(rng.integers(1, 9)),
                 -d - t_in * dec + int(rng.integers(0, 9)), int(rng.integers(-50, n_in)))[int(rng.integers(0, 6))]
        c[i] = dm, first + (t_in // 2) * dec - w // 2, i % len(WIDTHS), 0
    got = sp.cnn_extract(plan, staged, n_in, torch.from_numpy(c).cuda(), WIDTHS, t_in=t_in).cpu().numpy()
    sums = np.zeros((n_in + 1, nchan), np.int64)
    np.cumsum(x, axis=0, out=sums[1:])
    for i, (dm, t, k, _) in enumerate(c):
        dec = max(1, WIDTHS[k] // 4)
        first = t + WIDTHS[k] // 2 - (t_in // 2) * dec + delays[dm].astype(np.int64)
        lo = np.clip(first[:, None] + dec * np.arange(t_in), 0, n_in)
        hi = np.clip(first[:, None] + dec * np.arange(1, t_in + 1), 0, n_in)
        ch = np.arange(nchan)[:, None]
        want = (sums[hi, ch] - sums[lo, ch]).reshape(256, nchan // 256, t_in).sum(axis=1)
        assert np.array_equal(got[i], want.astype(np.float32)), (i, dm, t, k)
