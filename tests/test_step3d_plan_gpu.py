"""The streaming 3-D step under its plan just above the brick kernel's size: tile columns in equal
parts without leftovers, and in parts whose leftovers are cut again, one and two shots; against
the brick kernel, which covers the grid without a plan and gives the same bits."""
import numpy as np
import pytest

from paper_1912_08063_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,shape,shots", [
    (8, (121, 117, 131), 1), (8, (88, 85, 152), 2), (8, (130, 120, 152), 1), (16, (140, 121, 133), 1),
])
def test_planned_step_matches_bricks(order, shape, shots, monkeypatch):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(order + shots)
    nt, h = 24, 10.0
    v = torch.from_numpy(rng.uniform(1600.0, 4400.0, shape).astype(np.float32)).cuda()
    dt = 0.3 * h / 4600.0
    src = np.stack([np.array(shape) // 2 + 3 * k for k in range(shots)]).astype(np.int32)
    yy, xx = np.meshgrid(np.arange(-4, 5, 2), np.arange(-4, 5, 2), indexing="ij")
    rec = np.stack([0 * yy.ravel() + shape[0] // 2 + 2, yy.ravel() + shape[1] // 2, xx.ravel() + shape[2] // 2],
                   1).astype(np.int32)
    acq = fwi.Acquisition(src, rec)
    wav = torch.from_numpy(np.stack([synth.ricker(60.0, dt, nt)] * shots).astype(np.float32)).cuda()
    dobs = torch.from_numpy(rng.standard_normal((shots, nt, len(rec))).astype(np.float32) * 1e-7).cuda()
    outs = []
    for brick in (None, "1"):
        if brick:
            monkeypatch.setenv("FWI_STEP3D_BRICK", brick)
        m = fwi.FwiModel(v, h, dt, nt, order=order, snap_dtype="fp32", sponge_vref=4600.0)
        tr = m.forward(acq, wav)
        phi, g = m.gradient(acq, wav, dobs)
        outs.append([x.double().cpu().numpy() for x in (tr, phi, g)])
        m.close()
    # traces and misfit bit for bit; the gradient too, summed in the same order
    for a, b in zip(*outs):
        assert np.abs(b).max() > 0
        assert np.array_equal(a, b)
