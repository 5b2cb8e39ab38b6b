"""Edges of the range-setting and downcast kernels: candidate counts around whole warps and
blocks, short and long segments, values on rounding boundaries, extreme scales and non-finite
weights."""
import numpy as np
import pytest

import oracle as O
from paper_2406_06385_gb300 import lrqat as LQ
from paper_2406_06385_gb300 import workloads as WL

from gpu_util import phi_buffer, torch

pytestmark = pytest.mark.gpu


def _spec(m, k, bits=4, group=0, phi=WL.PHI_QFIXED, r=8):
    return WL.LayerSpec("e", m, k, r, float(r), bits, group, phi)


@pytest.mark.parametrize("n", [1, 31, 33, 100, 129, 256])
@pytest.mark.parametrize("m,k,group,p", [(128, 640, 0, 2.0), (256, 256, 128, 3.0), (128, 1152, 0, 2.4)])
def test_lp_range_candidate_counts(n, m, k, group, p):
    """The chosen scale's exact loss is the smallest over the candidates up to 1e-4 (fp32 sums
    may order nearly equal candidates differently), for every block shape."""
    t = torch()
    g = t.Generator(device="cuda").manual_seed(n + k)
    W = t.randn((m, k), generator=g, device="cuda") * 0.02
    W[3] = 0.0
    spec = _spec(m, k, group=group)
    s = t.empty((m, k // group) if group else (m,), device="cuda")
    LQ.range_lp(LQ.Layer.from_spec(spec), W, s, p, n)
    w = W.reshape(m, -1, group or k).double()
    a = w.abs().amax(-1)
    s_max = t.where(a > 0, a / 7, t.ones_like(a)).float().double()

    def loss(sc):
        q = t.round((w / sc.unsqueeze(-1)).float().double()).clamp(-8, 7)
        return (w - sc.unsqueeze(-1) * q).abs().pow(p).sum(-1)

    best = t.stack([loss((s_max * (j + 1) / n).float().double()) for j in range(n)]).amin(0)
    got = loss(s.reshape(best.shape).double())
    assert bool((got <= best * (1 + 1e-4)).all())


@pytest.mark.parametrize("bits,phi", [(2, WL.PHI_QFIXED), (4, WL.PHI_INT_PACKED), (7, WL.PHI_QFIXED), (8, WL.PHI_BF16)])
@pytest.mark.parametrize("scale", [1.0, 0.0137, 2.0 ** -128, 2.0 ** 112])
def test_lp_range_on_rounding_boundaries(bits, phi, scale):
    """Weights at and next to the half steps of the full scale (one candidate in two of which the other is
    the full scale itself), at ordinary and extreme scales: the summed |error| of the chosen scale is
    the smallest up to the rounding of the fp32 sums (640 values: 640 * 2^-24 < 1e-4)."""
    t = torch()
    m, k, n = 128, 640, 2
    top = 2 ** (bits - 1) - 1
    rng = np.random.default_rng(bits)
    W = (rng.integers(-2 * top, 2 * top + 1, size=(m, k)) / 2 * scale).astype(np.float32)
    W = np.where(rng.random((m, k)) < 0.5, np.nextafter(W, np.float32(0)), W).astype(np.float32)
    W[:, 0] = np.float32(top * scale)
    s = t.empty(m, device="cuda")
    LQ.range_lp(LQ.Layer.from_spec(_spec(m, k, bits=bits, phi=phi)), t.from_numpy(W).cuda(), s, 1.0, n)
    s_max = (np.abs(W).max(1) / np.float32(top)).astype(np.float64)

    def loss(sc):
        sc = sc[:, None]
        q = np.clip(np.rint((W / sc.astype(np.float32)).astype(np.float32)), -top - 1, top)
        return np.abs(W - sc * q).sum(1)

    got = s.cpu().numpy().astype(np.float64)
    best = np.minimum(loss((s_max / 2).astype(np.float32).astype(np.float64)), loss(s_max))
    assert (loss(got) <= best * (1 + 1e-4)).all()


@pytest.mark.parametrize("phi,bits", [(WL.PHI_QFIXED, 4), (WL.PHI_QFIXED, 7), (WL.PHI_INT_PACKED, 3),
                                      (WL.PHI_FP8_E4M3, 4), (WL.PHI_BF16, 4)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -130, 2.0 ** 100, 0.0137])
def test_downcast_on_rounding_boundaries(phi, bits, scale):
    """Weights at and next to every half step of the stored grid, in and beyond its range, at
    ordinary and extreme scales: the stored base equals the oracle's bit for bit."""
    t = torch()
    m, k = 128, 1152   # a row of more than one block and a ragged one
    spec = _spec(m, k, bits=bits, phi=phi)
    rng = np.random.default_rng(3)
    step = 2.0 ** -(8 - bits) if phi == WL.PHI_QFIXED else 1.0
    half = rng.integers(-600, 600, size=(m, k)).astype(np.float64) * (step / 2)
    W = (half * scale).astype(np.float32)
    W = np.where(rng.random((m, k)) < 0.3, np.nextafter(W, np.float32(0)), W).astype(np.float32)
    s0 = np.full(m, scale, dtype=np.float32)
    L = LQ.Layer.from_spec(spec)
    out = phi_buffer(spec)
    LQ.downcast(L, t.from_numpy(W).cuda(), t.from_numpy(s0).cuda(), out)
    OL = O.Layer(m, k, 8, 8.0, bits, 0, phi, 0)
    want = O.downcast(W, s0, OL)
    np.testing.assert_array_equal(out.cpu().numpy().view(want.dtype), want)


def test_range_and_downcast_of_non_finite_weights():
    """NaN weights leave min-max untouched; they and infinities clip to the grid's ends in the
    fixed-point base, and a NaN is the zero code of the packed base."""
    t = torch()
    m, k = 128, 256
    W = t.randn((m, k), device="cuda").clamp(-2, 2)
    want = W.abs().amax(1) / 7
    W[:, 5] = float("nan")
    keep = W.abs().nan_to_num(0).amax(1) / 7
    s = t.empty(m, device="cuda")
    LQ.range_minmax(LQ.Layer.from_spec(_spec(m, k)), W, s)
    assert t.equal(s, t.where(keep == want, want, keep))
    W[:, 9], W[:, 10] = float("inf"), float("-inf")
    q = t.empty((m, k), dtype=t.int8, device="cuda")
    LQ.downcast(LQ.Layer.from_spec(_spec(m, k)), W, s, q)
    assert bool((q[:, 5] == -128).all() and (q[:, 9] == 112).all() and (q[:, 10] == -128).all())
    p = t.empty((m, k // 2), dtype=t.uint8, device="cuda")
    LQ.downcast(LQ.Layer.from_spec(_spec(m, k, phi=WL.PHI_INT_PACKED)), W, s, p)
    assert bool(((p[:, 2] >> 4) == 0).all() and ((p[:, 4] >> 4) == 7).all() and ((p[:, 5] & 15) == 8).all())
