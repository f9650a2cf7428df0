"""The streamed best-S/N map at its edges (beams one sample around the shortest
it takes, rows that are not 16-byte aligned, row groups of 13 to 15, blocks of one chunk,
tiles left to the tile kernel for their values), against the float64 oracle
with the bounds of every other map; and the windowed peak filter against the
oracle's filter on the same map, exactly."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_27262_gb300 as sp
from paper_2606_27262_gb300 import build as spbuild
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

POW2 = [1, 2, 4, 8, 16, 32, 64, 128, 256]
MIXED = [1, 3, 7, 12, 50, 200]


@pytest.fixture(scope="module", autouse=True)
def _built():
    spbuild.build()


def _plane(ndm, n_out, seed, bright):
    rng = np.random.default_rng(seed)
    x = rng.normal(5000.0, 60.0, size=(ndm, n_out)).astype(np.int32)
    if bright:  # samples that take a tile (2^22 / 256 from the mean) and a 32-bit sum (2^31 / 256) out of range
        for d, t, v in ((1, n_out // 3, 30000), (ndm // 2, n_out // 2, 40000000), (ndm - 1, n_out - 3, 25000)):
            x[d, t] = v
    return x


@pytest.mark.parametrize("ndm,n_out,widths,block,bright", [
    (13, 511, [1], 0, False), (14, 512, [1], 0, False), (15, 523, POW2, 0, False), (15, 524, POW2, 0, False),
    (29, 780, POW2, 256, False), (2, 1021, MIXED, 512, False), (31, 4101, MIXED, 1024, True),
    (43, 8192, POW2, 4096, True), (17, 5003, POW2, 768, True), (16, 2050, [1, 2, 300], 512, False),
    (16, 2050, MIXED, 300, False)])
def test_map_edges(ndm, n_out, widths, block, bright):
    x = _plane(ndm, n_out, ndm + n_out, bright)
    gb, gk = gu.dev_best_map(torch.from_numpy(x).cuda(), widths, block)
    ob, ok = oracle.best(x, widths, block)
    gu.check_best_map(gb, gk, ob, ok, oracle.boxcar_snr(x, widths, block))


@pytest.mark.parametrize("ndm,n_out,radius,thr", [
    (1, 511, 5, 1.0), (9, 512, 2, 0.5), (8, 513, 5, -1e30), (25, 1500, 3, 2.0), (70, 4099, 4, 1.5), (33, 2048, 5, 6.0)])
def test_window_peaks_equal_the_filter_of_the_map(ndm, n_out, radius, thr):
    x = _plane(ndm, n_out, n_out, False)
    x[ndm // 2, n_out // 2: n_out // 2 + 8] += 400
    x[0, 10] = x[0, 12]  # equal values inside a window
    dmt = torch.from_numpy(x).cuda()
    gb, gk = gu.dev_best_map(dmt, POW2, 0)
    cap = ndm * n_out
    cands = torch.zeros((cap, 4), dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    work = torch.empty(sp.sps_window_workspace_bytes(ndm, n_out, len(POW2), 0, radius), dtype=torch.uint8, device="cuda")
    sp.single_pulse_search_window(dmt, POW2, thr, 0, radius, work, cands, count)
    torch.cuda.synchronize()
    got = sp.cands_to_numpy(cands.cpu().numpy(), int(count.item()))
    want = set()
    pad = np.pad(gb, radius, constant_values=-np.inf)
    for d, t in np.argwhere(gb >= thr):
        w = pad[d: d + 2 * radius + 1, t: t + 2 * radius + 1].ravel()
        mid = w.size // 2
        if (gb[d, t] > w[:mid]).all() and (gb[d, t] >= w[mid + 1:]).all():
            want.add((d, t, float(gb[d, t]), int(gk[d, t])))
    assert {(int(c["dm_idx"]), int(c["t"]), float(c["snr"]), int(c["width_idx"])) for c in got} == want
    assert len(got) == len(want)
