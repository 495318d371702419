"""The streaming 3-D step under every kind of plan, one and two shots, against the brick kernel,
which covers a grid without a plan and gives the same bits.  Kinds, with fewer tile columns than
CTAs: every column in equal parts, one to a CTA ("equal"); equal parts whose leftovers are cut over
all CTAs ("cut"); longer first parts, leftovers to the CTAs with a last part ("longer").  With more
columns than CTAs: rounds of whole columns ("columns") or of parts of columns ("parts"), each with
leftovers cut again."""
import numpy as np
import pytest

from paper_1912_08063_gb300 import synth
from test_schedule_cpu import build_check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NB = 8
# rows of a tile column, forward modes and reverse (64 columns each)
TILE_ROWS = {8: (32, 16), 16: (16, 32)}


def _kind(check, order, computed, shots, rows, ctas):
    columns = -(-computed[2] // 64) * -(-computed[1] // rows) * shots
    rounds, zparts, rem_ctas, rem_first, _ = map(int, check(order // 2, computed[0], columns, ctas).split())
    if columns >= ctas:
        return "parts" if zparts > 1 else "columns"
    return "longer" if rem_first else "cut" if rem_ctas else "equal"


@pytest.mark.parametrize("order,computed,shots,forward,reverse", [
    (8, (200, 260, 130), 1, "equal", "longer"),
    (8, (240, 340, 250), 1, "longer", "cut"),
    (8, (100, 240, 250), 2, "longer", "longer"),
    (8, (72, 816, 576), 1, "cut", "parts"),
    (8, (72, 1136, 832), 1, "parts", "columns"),
    (16, (200, 180, 250), 1, "equal", "equal"),
    (16, (160, 240, 250), 2, "equal", "longer"),
    (16, (160, 340, 380), 1, "cut", "cut"),
    (16, (240, 260, 380), 1, "longer", "cut"),
    (16, (80, 852, 852), 1, "columns", "columns"),
    (16, (160, 1136, 832), 1, "parts", "parts"),
])
def test_planned_step_matches_bricks(order, computed, shots, forward, reverse, monkeypatch, tmp_path):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(order + shots)
    nt, h = 24, 10.0
    shape = tuple(n - 2 * NB for n in computed)
    gen = torch.Generator("cuda").manual_seed(order + shots)
    v = torch.rand(shape, device="cuda", generator=gen) * 2800.0 + 1600.0
    dt = 0.3 * h / 4600.0
    src = np.stack([np.array(shape) // 2 + 3 * k for k in range(shots)]).astype(np.int32)
    yy, xx = np.meshgrid(np.arange(-4, 5, 2), np.arange(-4, 5, 2), indexing="ij")
    rec = np.stack([0 * yy.ravel() + shape[0] // 2 + 2, yy.ravel() + shape[1] // 2, xx.ravel() + shape[2] // 2],
                   1).astype(np.int32)
    acq = fwi.Acquisition(src, rec)
    wav = torch.from_numpy(np.stack([synth.ricker(60.0, dt, nt)] * shots).astype(np.float32)).cuda()
    dobs = torch.from_numpy(rng.standard_normal((shots, nt, len(rec))).astype(np.float32) * 1e-7).cuda()
    outs = []
    for brick in ("0", "1"):
        monkeypatch.setenv("FWI_STEP3D_BRICK", brick)
        m = fwi.FwiModel(v, h, dt, nt, order=order, nb=NB, snap_dtype="fp32", sponge_vref=4600.0)
        tr = m.forward(acq, wav)
        phi, g = m.gradient(acq, wav, dobs)
        outs.append((tr, phi, g))
        ctas = m.info()["step_ctas"]
        m.close()
    check = build_check(tmp_path)
    rows = TILE_ROWS[order]
    kinds = [_kind(check, order, computed, shots, rows[i], c) for i, c in zip((0, 1, 0), ctas)]
    assert kinds == [forward, reverse, forward], (kinds, ctas)
    # traces and misfit bit for bit; the gradient too, summed in the same order
    for a, b in zip(*outs):
        assert a.abs().max() > 0
        assert torch.equal(a, b)
