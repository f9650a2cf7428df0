"""Which dedispersion kernel a call runs, and that its result is the direct
kernel's (a plan of shape 1 never has the shared-sum tables) bit for bit."""
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


def _dms(kind, n):
    start, step = {"fine": (0.0, 0.1), "mid": (300.0, 0.3), "coarse": (900.0, 1.0)}[kind]
    return start + step * np.arange(n)


def _sums_launches(call):
    before = sp.sums_launch_count()
    out = call()
    torch.cuda.synchronize()
    return sp.sums_launch_count() - before, out


# Direct and shared-sum time of each on one GB300, us: 290 and 172; 294 and 226; 1134 and 347; 1109 and 924; 1109 and
# 923; 843 and 917; 210 and 333; 26 and 41 (no tables).  The last has no tables either.
@pytest.mark.parametrize("nchan,kind,ndm,n_out,sums", [
    (1024, "fine", 512, 1025, 1), (1024, "mid", 512, 1500, 1), (4096, "fine", 64, 513, 1),
    (4096, "coarse", 129, 20001, 1), (4096, "coarse", 256, 12288, 1), (4096, "coarse", 129, 700, 0),
    (1024, "coarse", 256, 1500, 0), (64, "fine", 512, 2048, 0), (64, "coarse", 96, 2048, 0),
])
def test_kernel_of_a_call(nchan, kind, ndm, n_out, sums):
    f, dms = synth.band_freqs(nchan), _dms(kind, ndm)
    plan, direct = sp.Plan(f, synth.TSAMP, dms), sp.Plan(f, synth.TSAMP, dms, shape=1)
    rng = np.random.default_rng(nchan + ndm)
    x = rng.integers(0, 256, size=(n_out + plan.max_delay, nchan), dtype=np.uint8)
    ran, got = _sums_launches(lambda: gu.dev_dedisperse(plan, x))
    assert ran == sums
    ran, want = _sums_launches(lambda: gu.dev_dedisperse(direct, x))
    assert ran == 0
    assert torch.equal(got, want)
    rows = [0, ndm // 2, ndm - 1]
    assert np.array_equal(got[rows].cpu().numpy(), oracle.dedisperse(x, oracle.delays(f, synth.TSAMP, dms[rows]), n_out))


def _stream_batch(plan, nbeams, gulp):
    """A gulp of each of nbeams beams, pushed one after the other."""
    s = sp.Stream(plan, nbeams, gulp, [1, 2, 4], 1e9, 0, 64, 4 << 30, max_batch=4)
    g = torch.randint(0, 256, (gulp, plan.nchan), dtype=torch.uint8).pin_memory()
    for b in range(nbeams):
        s.history(b, torch.zeros((plan.max_delay, plan.nchan), dtype=torch.uint8).pin_memory())
    for b in range(nbeams):
        s.push(b, g)
    assert all(r.status == sp.SP_OK for r, _ in s.drain())
    s.close()


def test_a_stream_decides_for_each_batch():
    """One gulp runs shorter on the direct kernel (283 and 335 us measured), two or
    more in a batch on the shared-sum kernel (432 items: 505, 335)."""
    plan = sp.Plan(synth.band_freqs(1024), synth.TSAMP, _dms("coarse", 256))
    ran, _ = _sums_launches(lambda: _stream_batch(plan, 1, 12288))
    assert ran == 0
    ran, _ = _sums_launches(lambda: _stream_batch(plan, 6, 12288))
    assert ran >= 1


def test_batches_graphs_and_streams_are_counted():
    f = synth.band_freqs(1024)
    fine, coarse = sp.Plan(f, synth.TSAMP, _dms("fine", 128)), sp.Plan(f, synth.TSAMP, _dms("coarse", 128))
    for plan, sums in ((fine, 1), (coarse, 0)):
        batch = sp.Batch([plan], [0, 0], [1500, 1100], [1, 2, 4], 1e9, 0, 64, 4 << 30)
        st = torch.cuda.Stream()
        ran, _ = _sums_launches(lambda: batch.run(stream=st))
        assert ran == sums * batch.ngroups
        ran, _ = _sums_launches(lambda: batch.capture(stream=st))
        assert ran == 0
        ran, _ = _sums_launches(lambda: [batch.launch(stream=st) for _ in range(3)])
        assert ran == 3 * sums * batch.ngroups
        batch.close()
        ran, _ = _sums_launches(lambda: _stream_batch(plan, 1, 1500))
        assert ran == sums
