"""Layer budgets at the edges of how layers are put into a warp's lanes (32, 128, 256) and sequences into
a block (32, 8 or 4, beyond which a second kernel makes the row offsets): exact against the oracle."""
import numpy as np
import pytest
import torch

import paper_2509_09754_b200 as lava
from oracle import lava_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,batch", [(1, 1), (31, 32), (32, 33), (33, 8), (80, 9), (128, 1), (129, 4),
                                          (256, 5), (2, 1024)])
def test_budgets_at_the_edges_of_the_layout(layers, batch):
    rng = np.random.RandomState(layers + batch)
    e = rng.rand(layers, batch) ** 3
    e[:, 0] = 0.0
    if layers > 3:
        e[1::2, batch - 1] = e[0, batch - 1]  # equal remainders: ties go to the lower layer
    lo = rng.randint(0, 50, size=batch)
    hi = lo + rng.randint(1, 400, size=batch)
    total = np.array([rng.randint(layers * lo[b], layers * hi[b] + 1) for b in range(batch)])
    for mode in (lava.LAVA_BUDGET_DYNAMIC, lava.LAVA_BUDGET_UNIFORM, lava.LAVA_BUDGET_PYRAMID):
        out = torch.empty((layers, batch), dtype=torch.int64, device="cuda")
        off = torch.empty(layers * batch + 1, dtype=torch.int64, device="cuda")
        lava.lava_layer_budgets(layers, batch, torch.from_numpy(e).cuda(), torch.from_numpy(total).cuda(),
                                torch.from_numpy(lo).cuda(), torch.from_numpy(hi).cuda(), mode, out, off)
        got = out.cpu().numpy()
        for b in range(batch):
            want = O.layer_budgets(list(e[:, b]), int(total[b]), int(lo[b]), int(hi[b]), mode)
            assert [int(x) for x in got[:, b]] == want, (mode, b)
        np.testing.assert_array_equal(off.cpu().numpy(), np.concatenate([[0], np.cumsum(got.reshape(-1))]))
