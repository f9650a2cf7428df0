"""The DM-time image kernel at the edges of its paths: batch sizes on both
sides of each rows-per-warp choice, spectra of any length and alignment (4- and
16-byte copies), shifts from none to far outside the spectrum, windows too wide
for a stage, and a candidate's images that do not depend on its batch."""
import numpy as np
import pytest
import torch

import oracle.cnn as ocnn
import paper_2606_27262_gb300 as sp
from paper_2606_27262_gb300 import build as spbuild

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    spbuild.build()
    assert torch.cuda.is_available()


def _images(sub, shift):
    b = sub.shape[0]
    img = [torch.empty((b, 256, 256), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    sp.cnn_features(sub, torch.from_numpy(shift.astype(np.int32)).cuda(), img[0], img[1])
    torch.cuda.synchronize()
    return [x.float().cpu().numpy() for x in img]


@pytest.mark.parametrize("t_in,kind", [(256, "sweep"), (257, "sweep"), (400, "sweep"), (512, "random"),
                                       (1030, "wide"), (4096, "wide"), (4096, "random")])
def test_matches_the_oracle(t_in, kind):
    rng = np.random.default_rng(t_in)
    if kind == "random":  # neighbouring rows share nothing; some bins lie outside the spectrum
        shift = rng.integers(-t_in, t_in + 1, size=(256, 256))
    else:
        sweep = (t_in - 256) // 2 if kind == "sweep" else t_in
        shift = ocnn.dmt_shifts(500.0 - np.arange(4096) * (200.0 / 4096), 256, max(sweep, 1))
    sub = rng.standard_normal((2, 256, t_in)).astype(np.float32)
    sub[1] *= 100.0
    # a view whose rows are not 16-byte aligned takes the same values through the 4-byte copies
    flat = torch.empty(sub.size + 1, dtype=torch.float32, device="cuda")
    got = []
    for off in (0, 1):
        view = flat[off:off + sub.size].view(sub.shape)
        view.copy_(torch.from_numpy(sub))
        got.append(_images(view, shift))
    want = ocnn.features(sub.astype(np.float64), shift)
    for g, w in zip(got[0], want):
        # bf16 rounding (2^-9 of the value) plus float32 sums of 256 terms (256 * 2^-24 of their rms, 16)
        assert np.all(np.abs(g - w) <= 2.0 ** -8 * np.abs(w) + 2.0 ** -11)
    assert all(np.array_equal(a, b) for a, b in zip(got[0], got[1]))


def test_images_do_not_depend_on_the_batch():
    rng = np.random.default_rng(7)
    shift = ocnn.dmt_shifts(500.0 - np.arange(4096) * (200.0 / 4096), 256, 128)
    sub = torch.from_numpy(rng.standard_normal((64, 256, 512)).astype(np.float32)).cuda()
    alone = _images(sub[3:4].contiguous(), shift)
    for n in (15, 16, 47, 48, 64):
        many = _images(sub[:n].contiguous(), shift)
        assert all(np.array_equal(a[0], m[3]) for a, m in zip(alone, many))


@pytest.mark.parametrize("odd", [0, 1])
def test_extracted_spectra_are_exact(odd):
    """Bins of 1, 3, 4, 16 and 64 samples that start anywhere, windows over both
    ends of the beam and outside it, rows read four bytes at a time and (a
    beam at an odd address) one at a time: integers, so equal."""
    rng = np.random.default_rng(11)
    freqs, n_in, t_in, widths = 500.0 - np.arange(512) * (200.0 / 512), 3001, 300, [1, 15, 16, 64, 256]
    plan = sp.Plan(freqs, 0.00131072, np.array([0.0, 100.0, 333.0]))
    dl = plan.delays()
    data = rng.integers(0, 256, size=(512, n_in), dtype=np.uint8)
    pitch = sp.staged_pitch(n_in)
    staged = torch.zeros(512 * pitch + odd, dtype=torch.uint8, device="cuda")[odd:].view(512, pitch)
    staged[:, :n_in] = torch.from_numpy(data).cuda()
    cands = [(d, t, w) for d in range(3) for w in range(5) for t in (-40000, 0, 5, 1234, n_in - 2, 2 ** 30)]
    rec = np.array([(d, t, w, 0) for d, t, w in cands], dtype=np.int32)
    sub = sp.cnn_extract(plan, staged, n_in, torch.from_numpy(rec).cuda(), widths, t_in=t_in).cpu().numpy()
    total = np.concatenate([np.zeros((512, 1), np.int64), np.cumsum(data, axis=1, dtype=np.int64)], axis=1)
    for q, (d, t, w) in enumerate(cands):
        dec = max(1, widths[w] // 4)
        start = t + widths[w] // 2 + (np.arange(t_in) - t_in // 2) * dec + dl[d][:, None].astype(np.int64)
        at = lambda x: np.take_along_axis(total, np.clip(x, 0, n_in), axis=1)
        want = (at(start + dec) - at(start)).reshape(256, 2, t_in).sum(axis=1)
        assert np.array_equal(sub[q], want.astype(np.float32)), (d, t, w)
