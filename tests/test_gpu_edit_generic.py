"""Edits fused into the generic passes' first kernel (images narrower than 23 pixels,
rows above the compiled lengths, plans kept off the register-resident passes): the
bits of the standalone edit followed by a solve, in every storage type; and the
corrected solve on such plans is the two-step flow."""
import numpy as np
import pytest
import torch

from paper_1902_00176_gb300 import gfc, synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(autouse=True)
def _lib(gfc_lib):
    yield


@pytest.mark.parametrize("dt", [torch.float32, torch.float16, torch.bfloat16])
@pytest.mark.parametrize("H,W,C,B,force", [(70, 20, 2, 2, False), (37, 22, 1, 3, False), (40, 2100, 1, 1, False),
                                           (40, 56, 1, 3, True), (65, 501, 1, 2, True)])
def test_edits_in_the_generic_passes(H, W, C, B, force, dt, monkeypatch):
    if force:
        monkeypatch.setenv("GFC_FORCE_GENERIC", "1")
    img, gx, gy, edges = synth.edit_batch(B, C, H, W, seed=6600)
    p = gfc.Plan(H, W, C=C, batch=B, dtype=dt, device=DEV)
    dx, dy, de, di = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV).to(dt) for a in (gx, gy, edges, img))
    monkeypatch.setenv("GFC_FORCE_GENERIC", "1")
    gen = gfc.Plan(H, W, C=C, batch=B, dtype=dt, device=DEV)  # (solves of long rows have passes of their own)
    m, s = p.field_stats(di)
    for edit, kw in (("threshold", dict(frac=0.1)), ("threshold", dict(frac=0.3, ref=1.0)),
                     ("merge", dict(alpha=0.5, edges=de))):
        ex, ey = p.gradient_threshold(dx, dy, kw["frac"], kw.get("ref", 0.0)) if edit == "threshold" else \
            p.gradient_merge(dx, dy, de, 0.5)
        one = p.solve_edited(dx, dy, edit, **kw)
        assert torch.equal(one, gen.solve_from_gradient(ex, ey)), (edit, kw)
        corrected = p.solve_corrected(dx, dy, m, s, edit=edit, **kw)
        p.color_correct(one, m, s)
        assert torch.equal(corrected, one), (edit, kw)
    p.close()
    gen.close()
