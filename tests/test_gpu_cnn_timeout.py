"""The bounded waits of the classifier's tensor-core kernels run out on purpose,
with every access in bounds (the hook of sp_debug_staging_fault: the first stage
of every CTA expects 16 bytes that nothing brings, waits give up after 20000 SM
cycles).  The passes report it, no later pass is touched, and the same calls then
give the same results as before, bit for bit."""
import numpy as np
import pytest
import torch

import paper_2606_27262_gb300 as sp
import synth
from paper_2606_27262_gb300 import build as spbuild

pytestmark = pytest.mark.gpu

DEFAULT_LIMIT = 1 << 31


@pytest.fixture(scope="module", autouse=True)
def _built():
    spbuild.build()
    assert torch.cuda.is_available()
    yield
    sp.debug_staging_fault(0, DEFAULT_LIMIT)


@pytest.mark.parametrize("batch", [1, 3, 40])
def test_timeout_is_reported_and_the_next_passes_are_right(batch):
    g = torch.Generator(device="cuda").manual_seed(batch)
    ft, dmt = (torch.randn((batch, 256, 256), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    labels = (torch.arange(batch, device="cuda") % 2).float()
    clf = sp.Classifier(max_batch=batch, seed=7)

    def forward():
        prob = torch.empty(batch, device="cuda")
        clf.forward(ft, dmt, prob)
        torch.cuda.synchronize()
        return prob.cpu().numpy()

    want = forward()
    clf.backward(ft, dmt, labels)
    want_grads, params = clf.grads(), clf.params()
    assert clf.status() == 0
    sp.debug_staging_fault(16, 20000)
    try:
        forward()
        assert clf.status() == clf.status(clear=True) == sp.SP_STATUS_STAGING_TIMEOUT
        assert clf.status() == 0
        with pytest.raises(sp.SpotlightError) as e:
            clf.backward(ft, dmt, labels)
        assert e.value.code == sp.SP_ETIMEOUT
    finally:
        sp.debug_staging_fault(0, DEFAULT_LIMIT)
    with pytest.raises(sp.SpotlightError) as e:  # void gradients are not handed out
        clf.grads()
    assert e.value.code == sp.SP_EINVAL
    assert clf.status() == 0
    assert np.array_equal(forward(), want)
    clf.backward(ft, dmt, labels)
    assert np.array_equal(clf.grads(), want_grads)
    assert np.array_equal(clf.params(), params)
    clf.close()


def test_timeout_in_a_stream_voids_the_scores_of_its_job():
    """The search of a gulp is over when the hook is set, its classification is
    not started: the gulp keeps its candidates and peaks, without scores; the next
    gulp is scored."""
    nchan, gulp, widths = 256, 1500, [1, 2, 4, 8]
    f, dms = synth.band_freqs(nchan), np.arange(0, 120.0, 1.0)
    plan = sp.Plan(f, synth.TSAMP, dms)
    bursts = [synth.Burst(t0=700 + k * gulp, dm=60.0, fwhm=3.0, snr=30.0) for k in range(2)]
    x = synth.make_beam(9, nchan, plan.max_delay + 2 * gulp, f, bursts, widths=widths)
    hist = torch.from_numpy(x[:plan.max_delay].copy()).pin_memory()
    gulps = [torch.from_numpy(x[plan.max_delay + k * gulp:][:gulp].copy()).pin_memory() for k in range(2)]
    clf = sp.Classifier(max_batch=4, seed=3)
    s = sp.Stream(plan, 1, gulp, widths, 6.0, 0, 4096, 1 << 30, max_batch=1)
    s.attach(clf, t_in=256, kept_cap=8, min_points=2, snr_min=8.0)
    s.history(0, hist)
    s.push(0, gulps[0])
    torch.cuda.synchronize()
    sp.debug_staging_fault(16, 20000)
    try:
        (r, _, kept, prob), = s.drain(sifted=True)
    finally:
        sp.debug_staging_fault(0, DEFAULT_LIMIT)
    assert r.status == sp.SP_ETIMEOUT and r.count > 0 and r.kept == kept.size > 0
    assert (prob == -1.0).all() and r.accepted == 0
    s.push(0, gulps[1])
    (r, _, kept, prob), = s.drain(sifted=True)
    assert r.status == sp.SP_OK and kept.size > 0 and (prob >= 0.0).all()
    assert clf.status() == 0 and plan.status() == 0
    s.close()
    clf.close()
