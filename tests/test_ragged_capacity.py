"""boys_eval_ragged where the workspace holds the tile table just so, one tile short of it,
and one tile only: the table's route and the persistent one behind it, same bits."""
import numpy as np
import pytest
import torch

import paper_2512_10059_gb300 as pb
from paper_2512_10059_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("lens", [[1], [128], [129], [0, 0, 5], [300, 0, 128, 1, 127, 129, 4000], [7] * 500])
def test_capacity_border(lens):
    lens = np.array(lens)
    kmax = (np.arange(lens.size) * 7 % 33).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    x = W.mixture_c1(int(off[-1]), seed=lens.size)
    xt, ot, kt = (torch.from_numpy(a).to(DEV) for a in (x, off, kmax))
    out_off, total = pb.api.ragged_layout(ot, kt)
    flat = torch.cat([pb.boys_eval(xt[off[s]:off[s + 1]].clone(), int(kmax[s])).reshape(-1) for s in range(lens.size)])
    tiles = int(np.sum((lens + 127) // 128))
    for nbytes in sorted({256, 528, 512 + 16 * tiles - 16, 512 + 16 * tiles - 1, 512 + 16 * tiles, 512 + 16 * tiles + 16}):
        ws = torch.full((max(nbytes, 256),), 0xAB, dtype=torch.uint8, device=DEV)
        out = torch.full((total,), float("nan"), dtype=torch.float64, device=DEV)
        pb.boys_eval_ragged(xt, ot, kt, out=out, out_off=out_off, workspace=ws)
        assert pb.ragged_status(ws) is False
        assert torch.equal(out, flat)
