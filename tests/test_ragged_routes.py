"""The three routes of boys_eval_ragged by the size of the workspace: the persistent
kernel (256 bytes), the tile table built on the device, and the persistent kernel
behind a table that does not fit.  All give the bits of flat boys_eval."""
import numpy as np
import pytest
import torch

import paper_2512_10059_gb300 as pb
from paper_2512_10059_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("kmaxes", [(0,), (32,), (3, 17), (0, 1, 31, 32), tuple(range(33))])
def test_routes_bitwise(kmaxes):
    rng = np.random.default_rng(len(kmaxes))
    lens = rng.choice([0, 1, 31, 127, 128, 129, 300], size=45000, p=[.1, .7, .1, .03, .03, .03, .01])
    kmax = rng.choice(kmaxes, size=lens.size).astype(np.int32)
    off = np.zeros(lens.size + 1, dtype=np.int64)
    np.cumsum(lens, out=off[1:])
    x = W.mixture_c1(int(off[-1]), seed=4)
    xt, ot, kt = (torch.from_numpy(a).to(DEV) for a in (x, off, kmax))
    out_off, total = pb.api.ragged_layout(ot, kt)
    tiles = int(np.sum((lens + 127) // 128))
    assert tiles > 40000
    outs = []
    for nbytes in (256, 512 + 16 * 39999, 512 + 16 * 40000, 512 + 16 * tiles):
        ws = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
        out = torch.full((total,), float("nan"), dtype=torch.float64, device=DEV)
        pb.boys_eval_ragged(xt, ot, kt, out=out, out_off=out_off, workspace=ws)
        assert pb.ragged_status(ws) is False
        outs.append(out)
    for k in kmaxes:
        seg = np.flatnonzero((kmax == k) & (lens > 0))[:2000]
        pos = np.concatenate([np.arange(off[s], off[s + 1]) for s in seg])
        flat = pb.boys_eval(xt[torch.from_numpy(pos).to(DEV)], int(k)).cpu().numpy()
        host, oo = outs[0].cpu().numpy(), out_off.cpu().numpy()
        a = 0
        for s in seg:
            n = lens[s]
            assert np.array_equal(host[oo[s]:oo[s] + (k + 1) * n].reshape(k + 1, n), flat[:, a:a + n])
            a += n
    for o in outs[1:]:
        assert torch.equal(o, outs[0])
