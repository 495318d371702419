"""2-D stepping on chip (one cluster of CTAs per shot) against single steps: same traces,
final states, misfits and gradients bit for bit, at the edges of what fits (bands of just M
rows, a partial group of four columns, one to three blocks per thread, the gradient on and
off chip), for one and several shots, every checkpoint format, checkpoint budgets with
and without recomputation, several folds of the gradient, and odd step counts."""
import numpy as np
import pytest

from paper_1912_08063_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,nx,nb,order,nshots,snap,slots,nt,fold", [
    (64, 33, 0, 8, 1, "fp32", 0, 31, 256),      # bands of exactly M rows
    (128, 18, 0, 16, 1, "bf16", 0, 40, 256),
    (70, 101, 6, 8, 2, "fp16", 0, 61, 16),      # ragged groups, three folds and a rest
    (90, 90, 9, 16, 1, "fp16", 9, 50, 7),       # clusters of 8; recomputation in short runs
    (40, 60, 0, 16, 1, "fp32", 0, 30, 256),     # clusters of 4
    (120, 340, 10, 8, 1, "bf16", 14, 64, 256),
    (250, 250, 10, 16, 1, "fp32", 0, 33, 256),  # forward on chip, gradient not
    (230, 220, 10, 8, 1, "bf16", 0, 25, 256),   # two blocks per thread
    (64, 1200, 20, 8, 1, "fp16", 0, 21, 256),   # wide: rows of 310 groups, forward on chip
])
def test_onchip_equals_single_steps(nz, nx, nb, order, nshots, snap, slots, nt, fold):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(nz + nx)
    v = synth.smooth_random(rng, (nz, nx), 10.0, ell=80.0)
    h, dt = 10.0, 0.4 * 10.0 / 4600.0
    # sources within 5 rows of the receivers: 20 steps carry the waves at least 6 cells, so
    # that the forward and reverse fields meet and the gradient is not zero
    src = np.stack([nz // 2 + rng.integers(-5, 6, nshots), np.zeros(nshots, int), rng.integers(0, nx, nshots)], 1)
    rec = np.array([[nz // 2, 0, x] for x in range(0, nx, 3)], dtype=np.int32)
    acq = fwi.Acquisition(src.astype(np.int32), rec)
    wav = torch.from_numpy(np.stack([synth.ricker(30.0, dt, nt) * (1 + 0.2 * s) for s in range(nshots)])
                           .astype(np.float32)).cuda()
    dobs = torch.from_numpy(rng.standard_normal((nshots, nt, len(rec))).astype(np.float32) * 1e-6).cuda()
    field = -(-(nz + 2 * nb) * (-(-(nx + 2 * nb) // 8) * 8) // 64) * 64
    outs = []
    for tb in (1, 0):   # 1: single steps; 0: on chip where it fits
        m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, order=order, nb=nb if nb else -1,
                         snap_dtype=snap, fold_every=fold, temporal_blocking=tb, sponge_vref=4600.0,
                         snap_budget_bytes=slots * nshots * field * (4 if snap == "fp32" else 2))
        tr, fin = m.forward(acq, wav, final_state=True)
        phi, g, g64 = m.gradient(acq, wav, dobs, want64=True)
        i = m.info()
        outs.append(([x.cpu().numpy() for x in (tr, fin, phi, g, g64)], i["kernel_launches"]))
        if slots:
            assert i["snap_slots"] < nt - 1
        stats = {k: i[k] for k in ("last_forward_steps", "last_adjoint_steps", "last_snap_stores",
                                   "last_snap_restores", "snap_slots")}
        outs[-1] += (stats,)
        m.close()
    for x, y in zip(outs[0][0], outs[1][0]):
        assert np.array_equal(x, y)
    assert outs[0][2] == outs[1][2]
    assert np.isfinite(outs[1][0][3]).all() and np.abs(outs[1][0][3]).max() > 0
    assert outs[1][1] < outs[0][1]      # the on-chip calls launched fewer kernels
