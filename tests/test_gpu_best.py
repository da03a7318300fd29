"""perch_best at the edges of its blocks and rounds, with ties, caller ids and costs
aligned to 4 bytes only, against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2008_00326_gb300 import build, perch
    build.build()
    perch.load()
    return perch


@pytest.mark.parametrize("n", [1, 2, 31, 255, 257, 1023, 1024, 1025, 300001, 608 * 1024, 608 * 1024 + 1, 1300003])
@pytest.mark.parametrize("span", [1, 3, 5000])
def test_best_device(P, oracle, n, span):
    import torch
    rng = np.random.default_rng(n + span)
    costs = rng.integers(0, span, (n, 2)).astype(np.int32)
    ids = rng.permutation(n).astype(np.uint64) * np.uint64(3 << 31) + np.uint64(5)
    s = torch.cuda.Stream()
    with P.Context(0) as ctx, torch.cuda.stream(s):
        for shift in (0, 1):                    # the second: costs on a 4-byte boundary
            buf = torch.zeros(2 * n + 2, dtype=torch.int32, device="cuda")
            dc = buf[shift:shift + 2 * n]
            dc.copy_(torch.from_numpy(costs.reshape(-1)))
            for i in (None, ids, ids // np.uint64(7 << 31)):      # the last has equal ids too
                bi = torch.zeros(1, dtype=torch.int64, device="cuda")
                bc = torch.zeros(1, dtype=torch.int32, device="cuda")
                di = None if i is None else torch.from_numpy(i.view(np.int64)).cuda()
                ctx.best(dc, di, stream=s, out_index=bi, out_cost=bc)
                s.synchronize()
                J = costs.astype(np.int64).sum(1)
                at = np.flatnonzero(J == J.min())
                k = at[np.argmin(i[at])] if i is not None else at[0]
                assert (int(bi.item()), int(bc.item())) == (int(k), int(J.min()))
                assert oracle.best(costs, ids=i) == (int(k), int(J.min()))
