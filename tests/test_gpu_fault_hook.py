"""The largest value the staging test hook accepts (1 MiB) stays inside what a
barrier can count: the waits run out and are reported, later calls are right."""
import numpy as np
import pytest
import torch

import paper_2606_27262_gb300 as sp
import synth
from paper_2606_27262_gb300 import build as spbuild
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [0, 1])  # shared sums, direct
def test_largest_hook_value(shape):
    spbuild.build()
    f, dms, n_out = synth.band_freqs(1024), 0.1 * np.arange(70), 1500
    plan = sp.Plan(f, synth.TSAMP, dms, shape=shape)
    x = np.random.default_rng(shape).integers(0, 256, size=(n_out + plan.max_delay, 1024), dtype=np.uint8)
    want = gu.dev_dedisperse(plan, x)
    sp.debug_staging_fault(1 << 20, 20000)
    try:
        gu.dev_dedisperse(plan, x)
    finally:
        sp.debug_staging_fault(0, 1 << 31)
    assert plan.status(clear=True) & sp.SP_STATUS_STAGING_TIMEOUT
    assert torch.equal(gu.dev_dedisperse(plan, x), want) and plan.status() == 0
