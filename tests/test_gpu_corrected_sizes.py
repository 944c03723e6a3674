"""gfc_solve_corrected on images with more items of row pairs than the one-call flow
has room for (146 a field): the two-step flow's bits above the limit, its values to
FP32 rounding below it, and the oracle's flow on both sides."""
import numpy as np
import pytest
import torch

import oracle.gfc_edit_oracle as E
import oracle.gfc_oracle as O
from paper_1902_00176_gb300 import gfc, synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
F32, F16, BF16 = torch.float32, torch.float16, torch.bfloat16


@pytest.fixture(autouse=True)
def _lib(gfc_lib):
    yield


# (H, W, storage type, two-step flow); row pairs per item: 2 at N = 1960 and 2058, 3 at
# 980, 4 at 1568, 5 at 1250, 7 at 270, 9 at 140
CASES = [(584, 1930, F32, False), (585, 1930, F32, True), (1080, 1920, F32, True), (876, 960, F32, False),
         (960, 960, F32, True), (1168, 1540, F32, False), (1169, 1540, F32, True), (1200, 1560, BF16, True),
         (1461, 1200, F16, True), (2045, 250, F32, True), (2044, 250, BF16, False), (2628, 132, F32, False),
         (2629, 132, F32, True), (3000, 64, F32, True), (600, 2050, F32, True)]


@pytest.mark.parametrize("H,W,dt,two_step", CASES)
def test_corrected_solve_on_both_sides_of_the_item_limit(H, W, dt, two_step):
    img, gx, gy, _ = synth.edit_batch(1, 1, H, W, seed=6500)
    p = gfc.Plan(H, W, batch=1, dtype=dt, device=DEV)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV).to(dt)  # noqa: E731
    dx, dy = dev(gx), dev(gy)
    m, s = p.field_stats(dev(img))
    for edit, kw in (("threshold", dict(frac=0.1)), ("none", {})):
        one = p.solve_corrected(dx, dy, m, s, edit=edit, **kw)
        two = p.solve_edited(dx, dy, edit, **kw)
        p.color_correct(two, m, s)
        if two_step:
            assert torch.equal(one, two)
        else:  # FP32 rounding of the statistics, once more rounded to 16 bits
            lim = 1e-6 if dt == F32 else 4e-3
            assert float((one.double() - two.double()).norm()) <= lim * float(two.double().norm())
    if dt == F32:
        x, y = (t.cpu().numpy()[0, 0] for t in (dx, dy))
        ic = O.solve_from_gradient(x.astype(np.float64), y.astype(np.float64), p.M, p.N, p.pad)
        ref = E.color_correct_with(ic, float(m), float(s))
        got = one.double().cpu().numpy()[0, 0]
        assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
    p.close()
