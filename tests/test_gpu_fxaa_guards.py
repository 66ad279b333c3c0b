"""FXAA takes the lumas of a column's ends from the texels that the guard slots
stand for: a buffer whose own guard slots were never filled gives the same
texels, except where the blend itself reads a guard slot."""

import numpy as np
import pytest

import oracle
from parity import lp_slots, to_device_lp

pytestmark = pytest.mark.gpu

POSE = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, -3.0]])


@pytest.mark.parametrize("fill", [float("nan"), 0.0, 5.0])
@pytest.mark.parametrize("e_max, half", [(0.15, False), (3.0, True), (60.0, False)])
def test_unfilled_guards(V, torch_mod, e_max, half, fill):
    torch = torch_mod
    P, F = oracle.PAPER_PIVOTS_DEG, oracle.PAPER_PIVOTS_CPD
    lay = oracle.lp_layout(e_max=e_max)
    s = V.vafr_session_create(V.make_session_desc(512, 512, 90.0, [POSE], int(half), 0,
                                                  acuity=V.make_acuity(P, F, e_max_deg=e_max)))
    slot, n_slots, counts, offs = lp_slots(V, s)
    rng = np.random.default_rng(7)
    lp = to_device_lp(rng.uniform(0.0, 1.0, (lay.total, 4)).astype(np.float16 if half else np.float32), V, s)
    guards = np.concatenate([offs - 1, offs + counts])
    bare = lp.copy()
    bare[guards] = fill
    out = []
    for buf in (lp, bare):
        dev = torch.from_numpy(np.ascontiguousarray(buf)).cuda()
        res = torch.full_like(dev, 9.0)
        V.vafr_fxaa_lp(s, 0, dev, res)
        out.append(res.float().cpu().numpy()[slot])
    V.vafr_session_destroy(s)
    differ = (out[0] != out[1]).any(1)
    ends = np.zeros(n_slots, bool)
    ends[np.concatenate([offs, offs + counts - 1])] = True
    assert not differ[~ends[slot]].any()
    # at the ends the luma and every decision are the same; a blend along the angle takes its
    # colour from the guard slot (about half of the blends)
    assert differ[ends[slot]].mean() < 0.75
