"""The gradient finish (fold of the sponge cells onto the physical cells they replicate,
sum over shots) where its work splits: rows on and off the z and y faces, one and many
shots, no sponge, extents of one and two cells, rows of one, two and several column
chunks."""
import numpy as np
import pytest

import oracle
from paper_1912_08063_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,nshots,nb", [
    ((1, 40), 1, 9), ((2, 33), 9, 5), ((37, 1), 3, 8), ((12, 270), 8, 7), ((20, 65), 2, 0),
    ((3, 1, 40), 1, 6), ((2, 2, 30), 2, 7), ((9, 12, 257), 1, 4), ((8, 7, 34), 9, 3),
])
def test_finish_matches_oracle(shape, nshots, nb):
    from paper_1912_08063_gb300 import fwi
    rng = np.random.default_rng(51)
    ndim = len(shape)
    v = rng.uniform(1600.0, 4400.0, shape).astype(np.float32)
    h, nt = 10.0, 40
    dt = 0.4 * h / 4500.0
    hi = shape if ndim == 3 else (shape[0], 1, shape[1])
    # sources and receivers within a few cells of one another, so that 40 steps carry signal
    # between them, at the end of the row (its fold and the last column chunk included)
    lo = [max(0, n - 12) for n in hi]
    src = np.stack([rng.integers(a, n, nshots) for a, n in zip(lo, hi)], 1).astype(np.int32)
    rec = np.stack([rng.integers(a, n, 5) for a, n in zip(lo, hi)], 1).astype(np.int32)
    rec = np.unique(rec, axis=0)
    wav = np.broadcast_to(synth.ricker(40.0, dt, nt), (nshots, nt)).astype(np.float32).copy()
    p = oracle.Problem(v, h, dt, nt, order=8, nb=nb, vref=4600.0, src=src, rec=rec, wavelet=wav)
    dobs = (0.8 * p.forward()).astype(np.float32)
    _, rg = p.gradient(dobs.astype(np.float64))
    m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, nb=nb if nb else -1, sponge_vref=4600.0)
    _, g, g64 = m.gradient(fwi.Acquisition(src, rec), torch.from_numpy(wav).cuda(),
                           torch.from_numpy(dobs).cuda(), want64=True)
    rg = np.asarray(rg).reshape(shape)
    # FP32 wavefields over 40 steps: the bar of the other FP32-checkpoint gradients
    e = np.linalg.norm(g64.cpu().numpy() - rg) / np.linalg.norm(rg)
    print(f"finish {shape} shots {nshots} nb {nb}: rel-L2 {e:.2e}")
    assert e <= 1e-3
    assert torch.equal(g, g64.float())
    m.close()
