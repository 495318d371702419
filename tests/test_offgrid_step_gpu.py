"""Off-grid sources added inside the 3-D brick step (with the step's own receiver samples,
checkpoint maxima and stores) against the separate injection after the streaming step, bit
for bit: taps that straddle bricks, that reach into the sponge, several shots; and off-grid
receivers against the node samples they interpolate at integer positions."""
import numpy as np
import pytest

from paper_1912_08063_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,snap,slots", [(8, "fp16", 0), (16, "bf16", 8), (8, "fp32", 6)])
def test_source_taps_in_the_step(order, snap, slots, monkeypatch):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(order + slots)
    shape, nb, nt, h = (20, 22, 50), 6, 40, 10.0
    v = synth.smooth_random(rng, shape, h, ell=80.0)
    dt = 0.35 * h / 4600.0
    src = np.array([[7.3, 10.6, 31.5], [0.2, 21.0, 0.7], [10.0, 8.0, 24.0]])
    yy, xx = np.meshgrid(range(0, 22, 3), range(0, 50, 3), indexing="ij")
    rec = np.stack([np.full(yy.size, 8), yy.ravel(), xx.ravel()], 1).astype(np.int32)
    acq = fwi.Acquisition(rec=rec, src_pos=src)
    wav = torch.from_numpy(np.stack([synth.ricker(50.0, dt, nt)] * 3).astype(np.float32)).cuda()
    dobs = torch.from_numpy(rng.standard_normal((3, nt, len(rec))).astype(np.float32) * 1e-7).cuda()
    field = -(-32 * 34 * 64 // 64) * 64
    outs = []
    for brick in ("0", "1"):
        monkeypatch.setenv("FWI_STEP3D_BRICK", brick)
        m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, order=order, nb=nb, snap_dtype=snap,
                         sponge_vref=4600.0,
                         snap_budget_bytes=slots * 3 * field * (4 if snap == "fp32" else 2))
        tr, fin = m.forward(acq, wav, final_state=True)
        phi, _ = m.gradient(acq, wav, dobs)
        outs.append([x.cpu().numpy() for x in (tr, fin, phi)] + [m.gradient(acq, wav, dobs)[1].cpu().numpy()])
        m.close()
    for a, b in zip(outs[0][:3], outs[1][:3]):
        assert np.array_equal(a, b)
    # the sources' image terms are atomic adds of one FP32 product per tap and step: 8 taps a
    # row, 512 a shot, in any order
    assert np.allclose(outs[0][3], outs[1][3], rtol=0, atol=2e-6 * np.abs(outs[0][3]).max())


@pytest.mark.parametrize("shape", [(40, 150), (18, 25, 40)])
def test_receiver_samples_at_integer_positions(shape):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(9)
    v = rng.uniform(1600.0, 4400.0, shape).astype(np.float32)
    h, nt = 10.0, 25
    dt = 0.35 * h / 4600.0
    hi = shape if len(shape) == 3 else (shape[0], 1, shape[1])
    src = np.array([[n // 2 for n in hi]], dtype=np.int32)
    rec = np.stack([np.clip(n // 2 + rng.integers(-4, 5, 13), 0, n - 1) for n in hi], 1).astype(np.int32)
    wav = torch.from_numpy(synth.ricker(50.0, dt, nt)[None].astype(np.float32)).cuda()
    m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, nb=5, sponge_vref=4600.0)
    node = m.forward(fwi.Acquisition(src, rec), wav)
    pos = m.forward(fwi.Acquisition(src, rec_pos=rec.astype(np.float64)), wav)
    assert torch.equal(node, pos) and node.abs().max() > 0
    m.close()


@pytest.mark.parametrize("shape", [(40, 150), (18, 25, 40)])
def test_tap_weights_match_the_oracle(shape):
    """Samples of the last state at the corners, edges and random positions of the grid, against
    the oracle's taps applied to that state."""
    import oracle
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(4)
    v = rng.uniform(1600.0, 4400.0, shape).astype(np.float32)
    h, nt, nb = 10.0, 60, 5
    dt = 0.35 * h / 4600.0
    hi = np.array(shape if len(shape) == 3 else (shape[0], 1, shape[1]))
    src = (hi // 2)[None].astype(np.int32)
    frac = np.array([[0, 0, 0], [1, 1, 1], [0, 1, 0.5], [1, 0, 0.25]] + rng.random((40, 3)).tolist())
    pos = frac * (hi - 1)
    pos[10:20] = np.floor(pos[10:20]) + [0.5, 0.0 if hi[1] == 1 else 0.5, 1e-9]
    pos = np.minimum(pos, hi - 1)
    wav = torch.from_numpy(synth.ricker(50.0, dt, nt)[None].astype(np.float32)).cuda()
    m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, nb=nb, sponge_vref=4600.0)
    tr, fin = m.forward(fwi.Acquisition(src, rec_pos=pos), wav, final_state=True)
    u = fin.cpu().numpy()[0, 0].astype(np.float64).ravel()   # u^nt, the last trace row's state
    got = tr.cpu().numpy()[0, -1]
    for p, g in zip(pos, got):
        idx, w = oracle.point_taps(shape, p if len(shape) == 3 else p[[0, 2]], nb=nb)
        ref, mag = np.sum(w * u[idx]), np.sum(np.abs(w * u[idx]))
        # each weight is a product of FP32-rounded factors, the sum is in FP32: 64 or 512 terms
        # in chains of at most 8 and a tree of at most 6, and three roundings a weight
        assert abs(g - ref) <= (8 + 6 + 3) * 2.0 ** -24 * mag * 2 + 1e-30
    assert np.abs(got).max() > 0
    m.close()
