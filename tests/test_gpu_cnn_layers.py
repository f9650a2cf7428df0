"""The convolutions' gradients at the edges of their tiles: batches whose last
layer fills half a tile (1), one and a half (3), and one at which every layer's
pixels are split between thread blocks unevenly (19).  Against the float64
oracle, which rounds to bf16 where the GPU stores bf16; what differs is a value
whose fp32 sum rounds the other way, one unit of 2^-8 at most, in few places:
2 % of a layer's norm, as for the whole step."""
import numpy as np
import pytest
import torch

import paper_2606_27262_gb300 as sp
from oracle import cnn as ocnn
from paper_2606_27262_gb300 import build as spbuild

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 3, 19])
def test_gradients_at_tile_edges(batch):
    spbuild.build()
    rng = np.random.default_rng(batch)
    ft, dmt = (torch.from_numpy(rng.normal(size=(batch, 256, 256)).astype(np.float32)).to(torch.bfloat16).cuda()
               for _ in range(2))
    labels = np.zeros(batch, np.float32)  # one sign of dloss: sums over examples do not cancel
    clf = sp.Classifier(max_batch=batch + 1, seed=batch)
    flat = clf.params()
    grads = []
    for _ in range(2):
        clf.backward(ft, dmt, torch.from_numpy(labels).cuda())
        grads.append(clf.grads())
    assert np.array_equal(grads[0], grads[1])  # no order of sums depends on scheduling
    as64 = [t.float().cpu().numpy().astype(np.float64) for t in (ft, dmt)]
    want = ocnn.forward_backward(flat, as64[0], as64[1], labels.astype(np.float64))[2]
    n, o = ocnn.num_params_branch(), 0
    for cin, cout in ((1, 16), (16, 32), (32, 64), (64, 128), (128, 256)):
        for size in (cout * 9 * cin, cout):
            for branch in range(2):
                s = slice(branch * n + o, branch * n + o + size)
                err = np.linalg.norm(grads[0][s] - want[s]) / np.linalg.norm(want[s])
                assert err <= 0.02, (cin, size, branch, err)
            o += size


@pytest.mark.parametrize("batch", [20, 77])
def test_split_layers_equal_whole_ones(batch):
    """A few tiles' output channels are shared by several thread blocks; layer 3
    stops at batch 19, layer 4 at 76.  Either way the same sums in the same order."""
    spbuild.build()
    gen = torch.Generator(device="cuda").manual_seed(batch)
    ft, dmt = (torch.randn((batch, 256, 256), device="cuda", generator=gen).to(torch.bfloat16) for _ in range(2))
    clf = sp.Classifier(max_batch=batch, seed=3)
    whole, part = torch.empty(batch, device="cuda"), torch.empty(2, device="cuda")
    clf.forward(ft, dmt, whole)
    for i in (0, batch - 2):
        clf.forward(ft[i:i + 2].contiguous(), dmt[i:i + 2].contiguous(), part)
        torch.cuda.synchronize()
        assert torch.equal(whole[i:i + 2], part)
