"""FXAA where its search and its lists are at their edges: columns shorter than
the search, neighbours of very different length, blocks that are all edge or
end in the middle of a block, against the oracle."""

import numpy as np
import pytest

import oracle
from parity import check_guards, lp_slots, to_device_lp

pytestmark = pytest.mark.gpu

POSE = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, -3.0]])


@pytest.mark.parametrize("e_max, delta", [(0.04, None), (0.15, None), (0.7, None), (3.0, None),
                                          (0.7, (3.0, 0.2, 0.2, 0.2, 0.2)), (2.0, (0.02, 1.5, 1.5, 1.5, 1.5))])
@pytest.mark.parametrize("density", [0.5, 0.02])
def test_small_layouts(V, torch_mod, e_max, delta, density):
    torch = torch_mod
    P, F = oracle.PAPER_PIVOTS_DEG, oracle.PAPER_PIVOTS_CPD
    lay = oracle.lp_layout(oracle.Acuity(P, F, delta=delta), e_max=e_max)
    s = V.vafr_session_create(V.make_session_desc(512, 512, 90.0, [POSE],
                                                  acuity=V.make_acuity(P, F, e_max_deg=e_max, delta=delta)))
    rng = np.random.default_rng(int(e_max * 100))
    for _ in range(4):
        # stretches of equal texels, so that searches run to their end
        on = np.cumsum(rng.random(lay.total) < density) % 2
        lp = (0.1 + 0.8 * on[:, None] * rng.uniform(0.9, 1.0, (lay.total, 4))).astype(np.float32)
        dev = torch.from_numpy(np.ascontiguousarray(to_device_lp(lp, V, s))).cuda()
        out = torch.full_like(dev, float("nan"))
        V.vafr_fxaa_lp(s, 0, dev, out)
        slot, _, counts, offs = lp_slots(V, s)
        assert np.array_equal(counts, lay.n_col)
        got = out.cpu().numpy()
        check_guards(got, counts, offs)
        assert np.abs(got[slot] - oracle.fxaa_lp(lp.astype(np.float64), lay)).max() < 1e-5
    V.vafr_session_destroy(s)
