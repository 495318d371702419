"""The 2-D step on halo tiles at the sizes where its tiling can go wrong: one cell, grids
smaller than the stencil radius, exact tiles (128 columns by 8 or 6 rows), one cell more, a
partial last group of four columns; one and several shots, receivers on one row (sampled and
injected by the step) and scattered (separate kernels), every checkpoint format."""
import numpy as np
import pytest

import oracle
from paper_1912_08063_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("order", [8, 16])
@pytest.mark.parametrize("nz,nx,nb,nshots,snap", [
    (1, 1, 0, 1, "fp32"), (3, 7, 0, 2, "fp32"), (6, 128, 0, 1, "fp16"), (7, 129, 0, 3, "fp32"),
    (8, 132, 0, 1, "bf16"), (9, 255, 0, 2, "fp16"), (33, 118, 5, 1, "fp32"), (24, 261, 6, 2, "bf16"),
])
def test_tile_step_matches_oracle(order, nz, nx, nb, nshots, snap, monkeypatch):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(nz * 1000 + nx + order)
    v = rng.uniform(1600.0, 4400.0, (nz, nx)).astype(np.float32)
    h, nt = 10.0, 45
    dt = 0.4 * h / 4500.0
    at = rng.integers(0, nx, nshots)
    # 45 steps carry the wavefield at least 1600 m/s * 45 dt = 6.4 cells: sources lie within
    # 4 rows of the receiver row and receivers around the first source's column, so that the
    # traces hold the wave and not its rounding tail ahead of the front
    src = np.stack([rng.integers(0, min(nz, 6), nshots), 0 * at, at], 1).astype(np.int32)
    cols = np.unique(np.clip(at[0] + np.array([-5, -4, -1, 0, 1, 2, 3, 6]), 0, nx - 1))
    row = np.stack([np.full(cols.size, min(2, nz - 1)), 0 * cols, cols], 1).astype(np.int32)
    wav = np.stack([synth.ricker(40.0, dt, nt) * (1 + 0.1 * s) for s in range(nshots)]).astype(np.float32)
    p = oracle.Problem(v, h, dt, nt, order=order, nb=nb, vref=4600.0, src=src, rec=row, wavelet=wav)
    ref, rfin = p.forward(final=True)
    dobs = (0.7 * ref).astype(np.float32)
    _, rg = p.gradient(dobs.astype(np.float64))
    outs = []
    for fuse in ("1", "0"):   # receivers in the step, or in the separate kernels
        monkeypatch.setenv("FWI_STEP3D_REC_FUSE", fuse)
        m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, order=order, nb=nb if nb else -1,
                         snap_dtype=snap, sponge_vref=4600.0)
        acq, w = fwi.Acquisition(src, row), torch.from_numpy(wav).cuda()
        tr, fin = m.forward(acq, w, final_state=True)
        phi, g = m.gradient(acq, w, torch.from_numpy(dobs).cuda())
        outs.append([x.cpu().numpy() for x in (tr, fin, phi, g)])
        m.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
    tr, fin, phi, g = outs[0]
    # the bars of the other parity tests: FP32 time stepping, and the checkpoint's rounding
    e = (_rel(tr, ref), _rel(fin.reshape(rfin.shape), rfin), _rel(g, np.asarray(rg).reshape(g.shape)))
    print(f"tile {nz}x{nx} nb {nb} o{order} {snap}: traces {e[0]:.1e} final {e[1]:.1e} grad {e[2]:.1e}")
    assert e[0] <= 1e-4 and e[1] <= 1e-4 and e[2] <= (1e-3 if snap == "fp32" else 1e-2)


@pytest.mark.parametrize("order,lo,hi,row", [
    (8, 523984, 524384, 524268),    # tile rows beyond 65535 of 8 rows: forward modes
    (16, 523984, 524384, 524276),
    (8, 393000, 393400, 393200),    # beyond 65535 of 6 rows: the reverse step
])
def test_more_tile_rows_than_a_launch_holds(order, lo, hi, row):
    """A grid of 524,400 computed rows: the rows around the last tile of a launch equal those of a
    model of rows lo .. hi - 1 alone, whose faces the waves do not reach (12 steps carry them at
    most 96 rows), bit for bit."""
    from paper_1912_08063_gb300 import fwi
    nz, nx, nb, nt, h = 524384, 12, 8, 12, 10.0
    dt = 0.3 * h / 4600.0
    v = np.random.default_rng(order).uniform(1600.0, 4400.0, (nz, nx)).astype(np.float32)
    wav = torch.from_numpy(synth.ricker(120.0, dt, nt)[None].astype(np.float32)).cuda()
    outs = []
    for a, b in ((0, nz), (lo, hi)):
        m = fwi.FwiModel(torch.from_numpy(v[a:b]).cuda(), h, dt, nt, order=order, nb=nb, sponge_vref=4600.0)
        src = np.array([[row - a, 0, nx // 2]], dtype=np.int32)
        rec = np.array([[row - a + 8, 0, x] for x in range(nx)], dtype=np.int32)
        acq = fwi.Acquisition(src, rec)
        tr, fin = m.forward(acq, wav, final_state=True)
        phi, g = m.gradient(acq, wav, tr * 0.5)
        fin = fin.reshape(-1, nx + 2 * nb)[nb + lo - a:nb + hi - a]
        outs.append([x.cpu().numpy() for x in (tr, fin, phi, g[lo - a:hi - a])])
        m.close()
    for x, y in zip(*outs):
        assert np.abs(x).max() > 0 and np.array_equal(x, y)
