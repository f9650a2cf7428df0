"""The shared-sum dedispersion kernel (dedisp_sums.cu) against the direct one
and the oracle, bit for bit, on DM lists whose trials share most of their
sums (0.1 to 1.0 pc cm^-3 apart over 1000 or more channels, so that its rule
takes them by a factor of two or more): edges of its tiles (64 trials, 1024
samples), of a 16-bit sum (256 channels), of channel groups (16), unsorted and
repeated trials, saturated input, a batch, and the bounded waits running out."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_27262_gb300 as sp
import synth
from paper_2606_27262_gb300 import build as spbuild
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    spbuild.build()
    assert torch.cuda.is_available()
    yield
    sp.debug_staging_fault(0, 1 << 31)


def _dms(kind, n):
    if kind == "fine":
        return 0.1 * np.arange(n)
    if kind == "coarse":
        return 900.0 + 1.0 * np.arange(n)
    if kind == "down":
        return (300.0 + 0.2 * np.arange(n))[::-1].copy()
    base = 100.0 + 0.1 * np.arange(n)  # mixed: neighbours swapped, some trials repeated
    return base[np.clip(np.arange(n) + np.tile([1, -1, 0, 2], n)[:n], 0, n - 1)]


@pytest.mark.parametrize("nchan,kind,ndm,n_out", [
    (1024, "fine", 64, 1024), (1024, "fine", 65, 1025), (1000, "fine", 63, 1023), (1024, "fine", 130, 1),
    (4096, "fine", 9, 513), (2049, "coarse", 70, 2047), (4096, "coarse", 129, 700), (1024, "down", 128, 1500),
    (1025, "mixed", 100, 3001), (513, "fine", 200, 4099), (257, "fine", 128, 1100), (256, "fine", 128, 1100),
])
def test_equals_the_direct_kernel_and_the_oracle(nchan, kind, ndm, n_out):
    rng = np.random.default_rng(nchan * 7 + ndm)
    f, dms = synth.band_freqs(nchan), _dms(kind, ndm)
    plan = sp.Plan(f, synth.TSAMP, dms)
    direct = sp.Plan(f, synth.TSAMP, dms, shape=1)
    x = rng.integers(0, 256, size=(n_out + plan.max_delay, nchan), dtype=np.uint8)
    got = gu.dev_dedisperse(plan, x).cpu().numpy()
    assert np.array_equal(got, gu.dev_dedisperse(direct, x).cpu().numpy())
    rows = np.unique(np.linspace(0, ndm - 1, 12).astype(int))
    want = oracle.dedisperse(x, oracle.delays(f, synth.TSAMP, dms[rows]), n_out)
    assert np.array_equal(got[rows], want)
    assert plan.status() == 0


@pytest.mark.parametrize("nchan", [1024, 4096])
def test_saturated_input(nchan):
    """All samples 255: every 16-bit partial sum at its largest."""
    f, dms, n_out = synth.band_freqs(nchan), _dms("fine", 100), 1300
    plan = sp.Plan(f, synth.TSAMP, dms)
    x = np.full((n_out + plan.max_delay, nchan), 255, np.uint8)
    assert (gu.dev_dedisperse(plan, x).cpu().numpy() == 255 * nchan).all()


def test_batch_of_two_plans():
    f = synth.band_freqs(1024)
    plans = [sp.Plan(f, synth.TSAMP, _dms("fine", 100)), sp.Plan(f, synth.TSAMP, _dms("coarse", 70))]
    rng = np.random.default_rng(3)
    beams, want = [], []
    for plan, n_out in zip(plans, (2500, 1023)):
        x = rng.integers(0, 256, size=(n_out + plan.max_delay, 1024), dtype=np.uint8)
        st = sp.staged_buffer(1024, x.shape[0])
        sp.stage_input(torch.from_numpy(x).cuda(), st)
        beams.append((plan, st, x.shape[0], torch.full((plan.ndm, n_out), -1, dtype=torch.int32, device="cuda")))
        want.append(gu.dev_dedisperse(sp.Plan(f, synth.TSAMP, plan.dms, shape=1), x))
    work = torch.empty(sp.dedisperse_batch_workspace_bytes(2), dtype=torch.uint8, device="cuda")
    sp.dedisperse_batch(beams, work)
    torch.cuda.synchronize()
    for (_, _, _, out), w in zip(beams, want):
        assert torch.equal(out, w)


def test_timeout_is_flagged_and_device_recovers():
    """As for the direct kernel: the first staging wait of every CTA runs out
    with all accesses in bounds; the status bit is set and the context stays
    usable."""
    rng = np.random.default_rng(11)
    f, dms, n_out = synth.band_freqs(1024), _dms("fine", 70), 1500
    plan = sp.Plan(f, synth.TSAMP, dms)
    x = rng.integers(0, 256, size=(n_out + plan.max_delay, 1024), dtype=np.uint8)
    sp.debug_staging_fault(16, 20000)
    try:
        gu.dev_dedisperse(plan, x)
        torch.cuda.synchronize()
    finally:
        sp.debug_staging_fault(0, 1 << 31)
    assert plan.status(clear=True) & sp.SP_STATUS_STAGING_TIMEOUT
    got = gu.dev_dedisperse(plan, x)
    assert torch.equal(got, gu.dev_dedisperse(sp.Plan(f, synth.TSAMP, dms, shape=1), x))
    assert plan.status() == 0
