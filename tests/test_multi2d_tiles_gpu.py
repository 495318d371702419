"""The serving loop's shared 2-D launch at the edges of its tiles (128 columns by 8 rows of the
computed grid): requests of several sizes in one table, receivers on two rows (sampled by the
sampling kernel) and on one row of a grid too large to step on chip (sampled by the step),
against direct calls bit for bit."""
import numpy as np
import pytest

from paper_1912_08063_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [8, 16])
def test_shared_launch_tiles_equal_direct_calls(order):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(order)
    nb, nt, h = 20, 30, 10.0
    dt = 0.35 * h / 4600.0
    wav = synth.ricker(50.0, dt, nt).astype(np.float32)
    reqs = []
    # computed sizes 1 + 2 nb and tile multiples, one less and one more
    for nz, nx in ((1, 1), (8, 88), (7, 89), (9, 87), (24, 92), (25, 217), (560, 530)):
        v = rng.uniform(1600.0, 4400.0, (nz, nx)).astype(np.float32)
        cols = np.unique(np.clip(nx // 2 + np.arange(-4, 5), 0, nx - 1))
        row = np.stack([0 * cols + min(1, nz - 1), 0 * cols, cols], 1)
        rec = row if nz > 500 else np.concatenate([row, row[:1] + [nz - 1 - min(1, nz - 1), 0, 0]])
        reqs.append({"kind": "forward", "v": v, "h": h, "dt": dt, "nt": nt, "order": order, "snap_dtype": "bf16",
                     "src": [min(2, nz - 1), 0, nx // 2], "rec": rec.astype(np.int32), "wavelet": wav,
                     "d_obs": None, "arrival": 0.0})
    res, out = fwi.fwi_serve(reqs, max_active=len(reqs), steps_per_turn=4, nb=nb)
    for r, x, o in zip(reqs, res, out):
        assert x["status"] == 0 and x["shared_launch"]
        m = fwi.FwiModel(torch.from_numpy(r["v"]).cuda(), h, dt, nt, order=order, nb=nb)
        tr = m.forward(fwi.Acquisition(np.array([r["src"]], np.int32), r["rec"]),
                       torch.from_numpy(wav[None]).cuda())
        assert np.abs(o).max() > 0 and np.array_equal(o, tr[0].cpu().numpy())
        m.close()
