"""Edges of the optimizer kernels: squares out of the fp32 range, non-finite and unaligned
gradients, unaligned parameters and state."""
import pytest

from paper_2406_06385_gb300 import lrqat as LQ
from paper_2406_06385_gb300 import workloads as WL

from gpu_util import torch

pytestmark = pytest.mark.gpu


def _spec(m, k, r):
    return WL.LayerSpec("e", m, k, r, float(r), 4, 0, WL.PHI_QFIXED)


@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e19])
@pytest.mark.parametrize("shift", [0, 1])
def test_gradient_norm_range_and_alignment(scale, shift):
    """Squares that overflow or vanish in fp32 are summed in doubles; unaligned gradients give the
    same sum (fp32 result of a sum of about 48 bits: 2^-23 relative)."""
    t = torch()
    m, k, r = 384, 640, 20
    g = t.Generator(device="cuda").manual_seed(1)
    mk = lambda n: (t.randn(n + 1, generator=g, device="cuda") * scale)[shift:shift + n]
    dA, dB, ds = mk(m * r), mk(r * k), mk(m)
    sq = t.zeros(1, device="cuda")
    L = LQ.Layer.from_spec(_spec(m, k, r))
    LQ.grad_sqnorm(L, dA, dB, ds, sq)
    want = sum(x.double().square().sum() for x in (dA, dB, ds)).float()
    if t.isinf(want):
        assert t.isinf(sq).item()
    else:
        assert abs(sq.item() - want.item()) <= 2.0 ** -23 * want.item() + 1e-45
    dB[7] = float("inf")
    sq.zero_()
    LQ.grad_sqnorm(L, dA, dB, ds, sq)
    assert t.isinf(sq).item()
    ds[3] = float("nan")
    LQ.grad_sqnorm(L, dA, dB, ds, sq)
    assert t.isnan(sq).item()


@pytest.mark.parametrize("m,k,r", [(128, 128, 1), (4096, 2048, 130), (2048, 4096, 256)])
@pytest.mark.parametrize("shift", [0, 3])
def test_gradient_norm_sizes(m, k, r, shift):
    """From less than one 16-byte item per thread to several batches of loads, the arrays' borders inside
    a batch; 2^-23 relative as above, over values of very different size in the three arrays."""
    t = torch()
    g = t.Generator(device="cuda").manual_seed(m + r)
    mk = lambda n, f: (t.randn(n + shift, generator=g, device="cuda") * f)[shift:]
    dA, dB, ds = mk(m * r, 1.0), mk(r * k, 1e-3), mk(m, 30.0)
    sq = t.zeros(1, device="cuda")
    LQ.grad_sqnorm(LQ.Layer.from_spec(_spec(m, k, r)), dA, dB, ds, sq)
    want = sum(x.double().square().sum() for x in (dA, dB, ds)).item()
    assert abs(sq.item() - want) <= 2.0 ** -23 * want


@pytest.mark.parametrize("r", [1, 20])
def test_adamw_of_unaligned_arrays(r):
    """Arrays that start off a 16-byte boundary take the one-element kernel: same values."""
    t = torch()
    m, k = 128, 256
    n = {"A": m * r, "B": r * k, "s": m}
    L = LQ.Layer.from_spec(_spec(m, k, r))
    opt = LQ.AdamW.make(1e-3, 1e-4, step=3, weight_decay_ab=0.1)
    got = []
    for off in (0, 1):
        g = t.Generator(device="cuda").manual_seed(5)
        mk = lambda size, f=1.0: t.nn.functional.pad(t.randn(size, generator=g, device="cuda") * f, (off, 0))[off:]
        st, grads, half = {}, {}, {}
        for key in ("A", "B", "s"):
            grads[key] = mk(n[key])
            st[key] = (mk(n[key]), mk(n[key], 0.1), mk(n[key], 0.1).square_())
        for key in ("A", "B"):
            half[key] = t.zeros(n[key] + off, dtype=t.bfloat16, device="cuda")[off:]
        sq = t.full((1,), 9.0, device="cuda")
        LQ.adamw_step(L, opt, sq, grads["A"], grads["B"], grads["s"],
                      dict(A32=st["A"][0], mA=st["A"][1], vA=st["A"][2], B32=st["B"][0], mB=st["B"][1], vB=st["B"][2],
                           ms=st["s"][1], vs=st["s"][2]), st["s"][0], half["A"], half["B"])
        got.append([x.clone() for key in ("A", "B", "s") for x in st[key]] + [half["A"].clone(), half["B"].clone()])
    for a, b in zip(*got):
        assert t.equal(a, b)
