"""The brick form of the 3-D step against the streaming kernels, bit for bit, where its
tiling can go wrong: grids smaller than the stencil radius, exact bricks (32 x 8 x 4), one
cell more in each direction, a partial last group of four columns, several shots, anisotropic
weights, receivers in the step and in separate kernels, every checkpoint format, with and
without recomputation."""
import numpy as np
import pytest

from paper_1912_08063_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [8, 16])
@pytest.mark.parametrize("shape,nb,h,nshots,snap,slots", [
    ((3, 2, 5), 0, (10.0, 10.0, 10.0), 1, "fp32", 0),
    ((8, 16, 64), 0, (10.0, 10.0, 10.0), 1, "fp16", 0),
    ((9, 17, 65), 0, (8.0, 10.0, 12.0), 2, "bf16", 0),
    ((5, 15, 30), 3, (10.0, 10.0, 10.0), 3, "fp32", 0),
    ((21, 33, 47), 4, (10.0, 10.0, 10.0), 1, "fp16", 6),
    ((40, 20, 70), 6, (8.0, 8.0, 10.0), 2, "bf16", 5),
])
def test_brick_equals_streaming(order, shape, nb, h, nshots, snap, slots, monkeypatch):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(sum(shape) + order)
    v = rng.uniform(1600.0, 4400.0, shape).astype(np.float32)
    nt, dt = 30, 0.35 * min(h) / 4600.0
    mid = np.array(shape) // 2
    src = np.clip(mid + rng.integers(-2, 3, (nshots, 3)), 0, np.array(shape) - 1).astype(np.int32)
    yy, xx = np.meshgrid(range(0, shape[1], 2), range(0, shape[2], 3), indexing="ij")
    rec = np.stack([np.full(yy.size, mid[0]), yy.ravel(), xx.ravel()], 1).astype(np.int32)
    acq = fwi.Acquisition(src, rec)
    wav = torch.from_numpy(np.stack([synth.ricker(60.0, dt, nt) * (1 + 0.2 * s) for s in range(nshots)])
                           .astype(np.float32)).cuda()
    dobs = torch.from_numpy(rng.standard_normal((nshots, nt, len(rec))).astype(np.float32) * 1e-7).cuda()
    c = [n + 2 * nb for n in shape]
    field = -(-c[0] * c[1] * (-(-c[2] // 8) * 8) // 64) * 64
    outs = []
    for brick, fuse in (("0", "1"), ("1", "1"), ("1", "0")):
        monkeypatch.setenv("FWI_STEP3D_BRICK", brick)
        monkeypatch.setenv("FWI_STEP3D_REC_FUSE", fuse)
        m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, order=order, nb=nb if nb else -1,
                         snap_dtype=snap, sponge_vref=4600.0,
                         snap_budget_bytes=slots * nshots * field * (4 if snap == "fp32" else 2))
        tr, fin = m.forward(acq, wav, final_state=True)
        phi, g, g64 = m.gradient(acq, wav, dobs, want64=True)
        outs.append([x.cpu().numpy() for x in (tr, fin, phi, g, g64)])
        m.close()
    for other in outs[1:]:
        for a, b in zip(outs[0], other):
            assert np.array_equal(a, b)
    assert np.isfinite(outs[0][3]).all() and np.abs(outs[0][3]).max() > 0


@pytest.mark.parametrize("shape,shots,grad", [
    ((262200, 4, 4), 1, True),      # 65550 bricks in z
    ((4, 524320, 2), 1, True),      # 65540 in y
    ((4, 4, 4), 65600, False),      # one in z for each shot
])
def test_thin_grids_beyond_a_launch_grid_stream(shape, shots, grad, monkeypatch):
    """Few points, but more bricks along an axis than a launch grid takes: the streaming kernels
    run the call, as they do with bricks off."""
    from paper_1912_08063_gb300 import fwi
    nt, dt = 10, 0.3 * 10.0 / 4600.0
    v = torch.from_numpy(np.random.default_rng(5).uniform(1600.0, 4400.0, shape).astype(np.float32)).cuda()
    src = np.broadcast_to(np.array(shape) // 2, (shots, 3)).astype(np.int32)
    rec = src[:1] + np.array([[1, 0, 0]], np.int32)
    wav = torch.from_numpy(np.tile(synth.ricker(120.0, dt, nt), (shots, 1)).astype(np.float32)).cuda()
    outs = []
    for brick in (None, "0"):
        if brick:
            monkeypatch.setenv("FWI_STEP3D_BRICK", brick)
        m = fwi.FwiModel(v, 10.0, dt, nt, order=16, nb=0, sponge_vref=4600.0)
        acq = fwi.Acquisition(src, rec)
        tr = m.forward(acq, wav)
        outs.append([tr, *(m.gradient(acq, wav, tr * 0.5) if grad else ())])
        m.close()
    for a, b in zip(*outs):
        assert a.abs().max() > 0 and torch.equal(a, b)
