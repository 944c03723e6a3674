"""Images of more than 2030 rows, whose row pairs outnumber the adjoint's slots of
partial sums: solves keep the register-resident passes, the adjoint runs the generic
ones. On both sides of the limit at one short, one odd and one long row length, and
at the tallest image."""
import numpy as np
import pytest
import torch

import fp32_reference
import oracle.gfc_oracle as O
from paper_1902_00176_gb300 import gfc, synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
REL_F32, MAXABS = 1e-5, 1e-4
F32, F16, BF16 = torch.float32, torch.float16, torch.bfloat16
UNIT = {F16: 2.0 ** -11, BF16: 2.0 ** -8}

CASES = [(2029, 64, F32), (2046, 64, F32), (2047, 64, BF16), (2200, 24, F32), (2046, 101, F16), (2050, 245, F32),
         (2050, 501, F32), (2047, 900, BF16), (2200, 1240, F32), (2100, 1555, F16), (4088, 40, F32), (4088, 333, BF16),
         (4087, 2049, F32)]


@pytest.fixture(autouse=True)
def _lib(gfc_lib):
    yield


def _rel(got, ref):
    return float(np.linalg.norm(got - ref) / max(np.linalg.norm(ref), 1e-300))


def _np(t):
    return t.double().cpu().numpy()


def _assert_near(got, ref, dt, rel):
    """FP32: relative L2. 16 bits: every element within the rounding of its storage
    and 1e-4 of the largest for the FP32 arithmetic."""
    if dt == F32:
        assert _rel(got, ref) <= rel
    else:
        assert np.all(np.abs(got - ref) <= UNIT[dt] * np.abs(ref) + 2.0 ** -25 + MAXABS * np.abs(ref).max())


@pytest.mark.parametrize("H,W,dt", CASES)
def test_tall_image_matches_oracle(H, W, dt, monkeypatch):
    rng = np.random.default_rng(9700 + H + W)
    img = np.add.outer(np.sin(np.arange(H) * 0.05), np.cos(np.arange(W) * 0.04))
    gx, gy = np.zeros((1, 1, H, W)), np.zeros((1, 1, H, W))
    gx[..., :-1] = np.diff(img, axis=1)
    gy[..., :-1, :] = np.diff(img, axis=0)
    gx += rng.uniform(-0.05, 0.05, (1, 1, 1, 1))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV).to(dt)  # noqa: E731
    tx, ty, tg = dev(gx), dev(gy), dev(synth.upstream_gradient((1, 1, H, W), seed=9800 + W))
    p = gfc.Plan(H, W, 1, 1, dtype=dt, device=DEV)
    out, lap = p.solve_from_gradient(tx, ty), p.solve_from_laplacian(tg)
    bx, by = p.backward(tg)
    edited = p.solve_edited(tx, ty, "threshold", frac=0.0)
    g = _np(tg)[0, 0]
    ref, rl = O.solve_from_gradient(_np(tx)[0, 0], _np(ty)[0, 0], p.M, p.N, p.pad), \
        O.solve_from_laplacian(g, p.M, p.N, p.pad)
    rx, ry = O.backward(g, p.M, p.N, p.pad)
    to = tl = tbx = tby = REL_F32
    if dt == F32:  # tall and narrow tori amplify FP32 rounding: within the bound of a plain FP32 transform
        div = O.divergence_torus(*(O.zero_extend(_np(t)[0, 0], p.M, p.N, p.pad) for t in (tx, ty)))
        div = div[p.pad:p.pad + H + 1, p.pad:p.pad + W + 1]
        fo = fp32_reference.torch_fp32_laplacian_solve(div, p.M, p.N, p.pad, DEV)[:H, :W]
        fl = fp32_reference.torch_fp32_laplacian_solve(g, p.M, p.N, p.pad, DEV)
        fx, fy = fp32_reference.torch_fp32_adjoint(g, p.M, p.N, p.pad, DEV)
        to, tl, tbx, tby = (max(REL_F32, 3.0 * _rel(f, r)) for f, r in ((fo, ref), (fl, rl), (fx, rx), (fy, ry)))
    _assert_near(_np(out)[0, 0], ref, dt, to)
    _assert_near(_np(edited)[0, 0], ref, dt, to)
    _assert_near(_np(lap)[0, 0], rl, dt, tl)
    _assert_near(_np(bx)[0, 0], rx, dt, tbx)
    _assert_near(_np(by)[0, 0], ry, dt, tby)
    monkeypatch.setenv("GFC_FORCE_GENERIC", "1")
    gen = gfc.Plan(H, W, 1, 1, dtype=dt, device=DEV)
    if H >= 2046:  # the generic adjoint's bits
        for a, b in zip((bx, by), gen.backward(tg)):
            assert torch.equal(a, b)
    gen.close()
    p.close()


def test_ragged_batch_with_a_tall_item():
    items = [(1, 300, 320), (2, 2300, 150), (1, 2100, 40)]
    rng = np.random.default_rng(9900)
    for dt in (F32, BF16):
        rp = gfc.RaggedPlan(items, dt, device=DEV)
        x, y = (rp.pack([torch.from_numpy(rng.standard_normal(s).astype(np.float32)) for s in items]) for _ in range(2))
        for (C, H, W), gx, gy, got in zip(items, rp.unpack(x), rp.unpack(y), rp.unpack(rp.solve_from_gradient(x, y))):
            p = gfc.Plan(H, W, C, 1, dtype=dt, device=DEV)
            want = p.solve_from_gradient(gx, gy)[0].double()
            unit = UNIT.get(dt, 2.0 ** -24)
            assert torch.all((got.double() - want).abs() <= 2 * unit * want.abs() + MAXABS * want.abs().max())
            p.close()
        rp.close()
