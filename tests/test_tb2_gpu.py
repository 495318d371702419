"""2-D stepping on chip (fwi_opts.temporal_blocking) against single steps and the oracle.  A
batch of more shots than clusters of CTAs run at once goes step by step, its shots one at a time
go on chip, many steps per launch with the states in shared memory: traces and final states are
equal bit for bit, for odd step counts too."""
import numpy as np
import pytest

import oracle
from paper_1912_08063_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(order, nshots, nt, seed):
    rng = np.random.default_rng(seed)
    nz, nx = 96, 200
    h = 10.0
    v = synth.smooth_random(rng, (nz, nx), h, ell=150.0)
    dt = 0.4 * h / 4500.0
    src = np.stack([np.full(nshots, 6), np.zeros(nshots, int),
                    rng.integers(0, nx, nshots)], 1).astype(np.int32)
    rec = np.stack([np.full(40, 3), np.zeros(40, int), np.linspace(0, nx - 1, 40).astype(int)],
                   1).astype(np.int32)
    wav = np.stack([synth.ricker(25.0, dt, nt) * (1 + 0.01 * s) for s in range(nshots)])
    return v, h, dt, src, rec, wav.astype(np.float32)


@pytest.mark.parametrize("order,nshots,nt", [(8, 48, 61), (16, 80, 40)])
def test_batch_in_single_steps_equals_shots_on_chip(order, nshots, nt):
    from paper_1912_08063_gb300 import fwi
    v, h, dt, src, rec, wav = _case(order, nshots, nt, seed=order)
    m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, order=order, sponge_vref=4600.0,
                     temporal_blocking=True)
    tr, fin = m.forward(fwi.Acquisition(src, rec), torch.from_numpy(wav).cuda(), final_state=True)
    tr, fin = tr.cpu().numpy(), fin.cpu().numpy()
    launches = m.info()["kernel_launches"]
    assert launches >= nt                       # a launch or more per step
    for s in (0, nshots // 2, nshots - 1):
        t1, f1 = m.forward(fwi.Acquisition(src[s:s + 1], rec), torch.from_numpy(wav[s:s + 1]).cuda(),
                           final_state=True)
        assert np.array_equal(tr[s], t1.cpu().numpy()[0])
        assert np.array_equal(fin[s], f1.cpu().numpy()[0])
    assert m.info()["kernel_launches"] - launches < nt   # three calls of a few launches


def test_batch_of_shots_matches_oracle():
    from paper_1912_08063_gb300 import fwi
    nshots, nt = 48, 50
    v, h, dt, src, rec, wav = _case(8, nshots, nt, seed=3)
    m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, order=8, sponge_vref=4600.0,
                     temporal_blocking=True)
    tr = m.forward(fwi.Acquisition(src, rec), torch.from_numpy(wav).cuda()).cpu().numpy()
    pick = [0, 17, 47]
    P = oracle.Problem(v, (h, h), dt, nt, order=8, nb=20, vref=4600.0, src=src[pick], rec=rec,
                       wavelet=wav[pick].astype(np.float64))
    ref = P.forward()
    e = np.linalg.norm(tr[pick] - ref) / np.linalg.norm(ref)
    print(f"batch traces vs oracle: rel-L2 {e:.2e}")
    assert e <= 1e-4


@pytest.mark.parametrize("shape,order", [((60, 90), 8), ((131, 77), 16), ((300, 280), 8)])
def test_onchip_blocking_equals_single_steps(shape, order):
    """temporal_blocking 0 and 2 run a one-shot 2-D forward with receivers on one row on chip:
    traces and the final state equal those of single steps (1) bit for bit, in fewer launches,
    and the traces match the oracle."""
    from paper_1912_08063_gb300 import fwi
    import oracle
    rng = np.random.default_rng(41)
    nz, nx = shape
    v = synth.smooth_random(rng, shape, 10.0, ell=80.0)
    h, nt = 10.0, 150
    dt = 0.5 / fwi.fwi_cfl_number(2, order, (h, h, h), float(v.max()), 1.0)
    src = np.array([[3, 0, nx // 2]], dtype=np.int32)
    rec = np.array([[2, 0, x] for x in range(nx)], dtype=np.int32)
    wav = synth.ricker(25.0, dt, nt)[None].astype(np.float32)
    acq = fwi.Acquisition(src, rec)
    outs, launches = [], []
    for tb in (1, 0, 2):
        m = fwi.FwiModel(torch.from_numpy(v).cuda(), h, dt, nt, order=order, nb=20,
                         temporal_blocking=tb)
        tr, fin = m.forward(acq, torch.from_numpy(wav).cuda(), final_state=True)
        outs.append((tr.cpu().numpy(), fin.cpu().numpy()))
        launches.append(m.info()["kernel_launches"])
        m.close()
    for other in outs[1:]:
        assert np.array_equal(outs[0][0], other[0]) and np.array_equal(outs[0][1], other[1])
    assert launches[1] == launches[2] < nt <= launches[0]
    ref = oracle.Problem(v, h, dt, nt, order=order, nb=20, src=src, rec=rec,
                         wavelet=wav).forward()
    e = np.linalg.norm(outs[1][0] - ref) / np.linalg.norm(ref)
    print(f"on-chip blocking {shape} order {order}: traces rel-L2 {e:.2e}")
    assert e <= 1e-4
