"""The streamed best-S/N map is the tile kernel's bit for bit: a candidate search
of a beam whose length is not a multiple of four runs the tile kernel, so its
candidates are the 3 x 3 peaks of the map, with the map's S/N bits and widths.
(Small planes with one block or one width are tiles for the map as well.)"""
import numpy as np
import pytest
import torch

from paper_2606_27262_gb300 import build as spbuild
from tests import gpu_util as gu
from tests.test_gpu_sps_map import MIXED, POW2, _plane

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    spbuild.build()


def _peaks_of(gb, gk):
    pad = np.pad(gb, 1, constant_values=-np.inf)
    keep = np.isfinite(gb)
    ndm, n = gb.shape
    for i in range(3):
        for j in range(3):
            if (i, j) != (1, 1):
                u = pad[i:i + ndm, j:j + n]
                keep &= gb > u if (i, j) < (1, 1) else gb >= u
    return [(int(d), int(t), int(gb[d, t:t + 1].view(np.int32)[0]), int(gk[d, t])) for d, t in np.argwhere(keep)]


@pytest.mark.parametrize("ndm,n_out,widths,block,bright", [
    (13, 511, [1], 0, False), (301, 9003, [1], 1024, True), (97, 24001, [4], 0, False), (300, 5003, POW2, 0, False),
    (29, 4099, MIXED, 512, False), (15, 523, POW2, 0, False), (29, 781, POW2, 256, False), (2, 1021, MIXED, 512, False),
    (31, 4101, MIXED, 1024, True), (43, 8193, POW2, 4096, True), (17, 5003, POW2, 768, True), (70, 20011, MIXED, 8192, False)])
def test_search_of_an_odd_length_finds_the_peaks_of_the_map(ndm, n_out, widths, block, bright):
    dmt = torch.from_numpy(_plane(ndm, n_out, 3 * ndm + n_out, bright)).cuda()
    gb, gk = gu.dev_best_map(dmt, widths, block)
    got, n = gu.dev_candidates(dmt, widths, -1e30, block)
    got = sorted((int(c["dm_idx"]), int(c["t"]), int(c["snr"].view(np.int32)), int(c["width_idx"])) for c in got)
    assert len(got) == n and got == _peaks_of(gb, gk)
