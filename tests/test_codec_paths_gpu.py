"""fwi_snapshot_encode where its path changes: one CTA or several launches, 16-byte or scalar
loads (length and alignment), every format, zero and non-finite input; scales and codes
against the definition evaluated with torch."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _reference(a, b, half, texp):
    codes, scales = [], []
    for x in (a, a - b):
        top = float(x.abs().max()) if x.numel() else 0.0
        m, e = math.frexp(top)
        s = 1.0 if top == 0.0 else 2.0 ** max(-126, min(127, texp - (e - 1) - (1 if m > 0.5 else 0)))
        scales.append(s)
        codes.append((x * s).to(half).view(torch.int16))
    return torch.cat(codes), scales


@pytest.mark.parametrize("dtype", ["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("n,shift", [(1, 0), (3, 1), (1000, 0), (32768, 1), (32769, 0), (32772, 0), (32772, 1),
                                     (300000, 0), (300001, 0), (2000004, 0)])
def test_encode_paths(n, shift, dtype):
    from paper_1912_08063_gb300 import fwi
    g = torch.Generator("cuda").manual_seed(n)
    a = (torch.randn(n + shift, generator=g, device="cuda") * 1e-6)[shift:]
    b = (torch.randn(n + shift, generator=g, device="cuda") * 1e-6)[shift:]
    code_dt = fwi.SNAP_DTYPES[dtype]
    code = torch.zeros(2 * n, dtype=torch.float32 if dtype == "fp32" else torch.int16, device="cuda")
    scale = torch.full((2,), 7.0, device="cuda")
    fwi.fwi_snapshot_encode(a, b, n, code_dt, code, scale)
    if dtype == "fp32":
        assert torch.equal(code, torch.cat([a, b])) and scale.tolist() == [1.0, 1.0]
    else:
        ref, s = _reference(a, b, torch.bfloat16 if dtype == "bf16" else torch.float16, 0 if dtype == "bf16" else 14)
        assert scale.tolist() == s and torch.equal(code, ref)
    a2, b2 = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    fwi.fwi_snapshot_decode(code, scale, n, code_dt, a2, b2)
    assert torch.isfinite(a2).all() and torch.isfinite(b2).all()


@pytest.mark.parametrize("n", [100, 50000])
@pytest.mark.parametrize("value,where", [(float("nan"), "a"), (float("inf"), "b"), (float("-inf"), "a"), (0.0, "all")])
def test_encode_special_values(n, value, where):
    from paper_1912_08063_gb300 import fwi
    a, b = torch.full((n,), 2.0, device="cuda"), torch.full((n,), 1.5, device="cuda")
    if where == "all":
        a.zero_()
        b.zero_()
    else:
        (a if where == "a" else b)[n - 1] = value
    code, scale = torch.zeros(2 * n, dtype=torch.int16, device="cuda"), torch.zeros(2, device="cuda")
    fwi.fwi_snapshot_encode(a, b, n, 2, code, scale)
    if where == "all":
        assert scale.tolist() == [1.0, 1.0] and not code.any()
    else:
        assert torch.isnan(scale).all()
