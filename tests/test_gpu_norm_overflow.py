"""The gradient norm of a diverged step: finite gradients whose squares or sums of squares leave fp32
give infinity (and AdamW then takes a step from the moments alone), never NaN."""
import pytest

from paper_2406_06385_gb300 import lrqat as LQ
from paper_2406_06385_gb300 import workloads as WL

from gpu_util import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k,r", [(4096, 4096, 32), (2048, 4096, 256)])
def test_norm_of_large_gradients(m, k, r):
    """Half powers of two from 2^46 to 2^62 against the sum in doubles: its fp32 value (2^-23 relative)
    where that is finite, else infinity."""
    t = torch()
    L = LQ.Layer.from_spec(WL.LayerSpec("n", m, k, r, float(r), 4, 0, WL.PHI_QFIXED))
    g = t.Generator(device="cuda").manual_seed(r)
    unit = [t.rand(n, generator=g, device="cuda") * 0.5 + 0.5 for n in (m * r, r * k, m)]
    for e in range(92, 125):
        dA, dB, ds = (u * 2.0 ** (e / 2) for u in unit)
        sq = t.zeros(1, device="cuda")
        LQ.grad_sqnorm(L, dA, dB, ds, sq)
        want = sum(x.double().square().sum() for x in (dA, dB, ds))
        if t.isinf(want.float()):
            assert t.isinf(sq).item(), (e, sq.item())
        else:
            assert abs(sq.double().item() - want.item()) <= 2.0 ** -23 * want.item(), e


@pytest.mark.parametrize("log2", [58.5, 59.0, 59.75, 61.0])
def test_diverged_step_is_clipped_to_nothing(log2):
    """An infinite norm clips by 0: the moments only decay, and finite parameters stay finite."""
    t = torch()
    m, k, r = 4096, 4096, 32
    L = LQ.Layer.from_spec(WL.LayerSpec("n", m, k, r, float(r), 4, 0, WL.PHI_QFIXED))
    n = {"A": m * r, "B": r * k, "s": m}
    grad = {key: t.full((size,), 2.0 ** log2, device="cuda") for key, size in n.items()}
    par = {key: t.full((size,), 0.5, device="cuda") for key, size in n.items()}
    mom = {key: t.full((size,), 0.25, device="cuda") for key, size in n.items()}
    var = {key: t.full((size,), 0.0625, device="cuda") for key, size in n.items()}
    A, B = (t.zeros(n[key], dtype=t.bfloat16, device="cuda") for key in ("A", "B"))
    sq = t.zeros(1, device="cuda")
    LQ.grad_sqnorm(L, grad["A"], grad["B"], grad["s"], sq)
    assert t.isinf(sq).item()
    opt = LQ.AdamW.make(1e-3, 1e-5, step=10, max_grad_norm=1.0)
    LQ.adamw_step(L, opt, sq, grad["A"], grad["B"], grad["s"],
                  dict(A32=par["A"], mA=mom["A"], vA=var["A"], B32=par["B"], mB=mom["B"], vB=var["B"],
                       ms=mom["s"], vs=var["s"]), par["s"], A, B)
    for key in n:
        # one fp32 product each
        assert t.equal(mom[key], t.full_like(mom[key], 0.25) * opt.beta1), key
        assert t.equal(var[key], t.full_like(var[key], 0.0625) * opt.beta2), key
        assert t.isfinite(par[key]).all().item(), key
