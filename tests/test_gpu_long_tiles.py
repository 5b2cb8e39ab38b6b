"""The GEMMs with the low-rank tile in the stage at token counts where the pair kernel takes its largest
tile (448 tokens in two accumulators, one producer group), and just above and below: against the
product with the merged codes, bit for bit.  The adapters are small multiples of 1/4, the tokens small
integers and the scales powers of two, so every sum is exact in fp32 in any order."""
import pytest

from paper_2406_06385_gb300 import lrqat as LQ
from paper_2406_06385_gb300 import workloads as WL

from gpu_util import DeviceLayer, torch

pytestmark = pytest.mark.gpu


def _spec(m, k, r, bits=4, group=0, phi=WL.PHI_QFIXED, asym=False, ub=False):
    return WL.LayerSpec("t", m, k, r, float(r), bits, group, phi, asym=asym, w_row_shift=0.03 if asym else 0.0, u_bf16=ub)


# 76 pairs: two or four 256-row blocks of 448-token tiles fill one round up to 17024 or 8512 tokens, where
# smaller tiles take two or more; one token more makes it two rounds for every tile
CASES = [
    ("q44", _spec(512, 256, 32), 17000),
    ("q44_full_round", _spec(512, 128, 8), 17024),
    ("q44_next_round", _spec(512, 128, 8), 17025),
    ("odd_rows_r20", _spec(384, 384, 20), 16801),
    ("two_rounds_r64", _spec(1024, 256, 64), 16999),
    ("int3_r48", _spec(512, 256, 48, bits=3, phi=WL.PHI_INT_PACKED), 16900),
    ("int2_asym", _spec(512, 384, 16, bits=2, asym=True), 17001),
    ("int2_asym_group", _spec(512, 512, 16, bits=2, group=128, asym=True), 16931),
    ("packed_group", _spec(512, 512, 32, phi=WL.PHI_INT_PACKED, group=256), 17011),
    ("bf16", _spec(512, 256, 32, phi=WL.PHI_BF16), 16999),
    ("bf16_group_odd", _spec(384, 256, 64, phi=WL.PHI_BF16, group=128), 17007),
    ("bf16_192_tokens", _spec(512, 256, 32, phi=WL.PHI_BF16), 7200),
    ("fp16", _spec(512, 384, 8, phi=WL.PHI_FP16), 17003),
    ("e4m3_ubf16", _spec(512, 256, 32, phi=WL.PHI_FP8_E4M3, ub=True), 16990),
    ("bf16_ubf16", _spec(512, 256, 32, phi=WL.PHI_BF16, ub=True), 16995),
]


def _layer(spec, T, wide):
    """A layer with exact arithmetic, `wide` tokens [T, k] or [T, m], and its merged integer weights."""
    t = torch()
    dl = DeviceLayer(WL.make_layer(spec, 1, seed=3, with_activations=False))
    g = t.Generator(device="cuda").manual_seed(7)
    pick = lambda shape, lo, hi: t.randint(lo, hi + 1, shape, generator=g, device="cuda").float()
    dl.A = (pick((spec.m, spec.r), -1, 1) / 4).to(t.bfloat16)
    dl.B = (pick((spec.r, spec.k), -1, 1) / 4).to(t.bfloat16)
    dl.s = 2.0 ** -pick(tuple(dl.s0.shape), 0, 3)
    tok = pick((T, wide), -2, 2)
    w_z = t.empty((spec.m, spec.k), dtype=t.int8, device="cuda")
    LQ.merge(dl.layer, dl.phi0, dl.A, dl.B, w_z)
    spread = lambda v: v.repeat_interleave(spec.group_size, 1) if spec.group_size else v[:, None]
    w = w_z.float() if dl.z is None else w_z.float() - spread(dl.z)
    return dl, tok, (w * spread(dl.s)).double()


@pytest.mark.parametrize("cid,spec,T", CASES, ids=[c[0] for c in CASES])
def test_forward(cid, spec, T):
    t = torch()
    dl, X, w = _layer(spec, T, spec.k)
    Y = t.full((T + 1, spec.m), float("nan"), dtype=t.bfloat16, device="cuda")
    LQ.linear_fwd_noalloc(dl.layer, T, X.to(t.bfloat16), dl.phi0, dl.s, dl.A, dl.B, None, Y)
    LQ.get_device_status()
    assert t.isnan(Y[T]).all().item()
    assert t.equal(Y[:T], (X.double() @ w.t()).to(t.bfloat16))


@pytest.mark.parametrize("cid,spec,T", CASES, ids=[c[0] for c in CASES])
def test_input_gradient(cid, spec, T, lowrank_path):
    """The transposed layer's shapes: 512 (384, 1024) produced rows."""
    t = torch()
    lowrank_path("tile")
    group = 128 if spec.group_size else 0
    spec = WL.LayerSpec("t", spec.k, spec.m, spec.r, spec.alpha, spec.bits, group, spec.phi_format, asym=spec.asym,
                        w_row_shift=spec.w_row_shift, u_bf16=spec.u_bf16)
    dl, dY, w = _layer(spec, T, spec.m)
    X = t.zeros((T, spec.k), dtype=t.bfloat16, device="cuda")
    dX = t.full((T + 1, spec.k), float("nan"), dtype=t.bfloat16, device="cuda")
    dA, dB = t.empty((spec.m, spec.r), device="cuda"), t.empty((spec.r, spec.k), device="cuda")
    ws = t.empty(LQ.bwd_workspace_bytes(dl.layer, T), dtype=t.uint8, device="cuda")
    LQ.linear_bwd(dl.layer, T, dY.to(t.bfloat16), X, dl.phi0, dl.s, dl.A, dl.B, None, dX, dA, dB, t.empty_like(dl.s),
                  False, ws)
    LQ.get_device_status()
    assert t.isnan(dX[T]).all().item()
    assert t.equal(dX[:T], (dY.double() @ w).to(t.bfloat16))


@pytest.mark.parametrize("tile", range(32, 449, 32))
def test_every_tile_on_the_codes(tile, lowrank_path):
    """Four 256-row blocks and 19 token tiles fill one round of 76 pairs, so each token count here takes
    another tile; 12 stages, more than any ring holds.  Forward and dX."""
    t = torch()
    lowrank_path("codes")
    T = 19 * tile - 5
    spec = _spec(1024, 768, 16, group=256, phi=WL.PHI_INT_PACKED)
    dl, X, w = _layer(spec, T, spec.k)
    Y = t.full((T + 1, spec.m), float("nan"), dtype=t.bfloat16, device="cuda")
    ws = t.empty(LQ.fwd_workspace_bytes(dl.layer, T), dtype=t.uint8, device="cuda")
    LQ.linear_fwd(dl.layer, T, X.to(t.bfloat16), dl.phi0, dl.s, dl.A, dl.B, None, Y, ws)
    assert t.isnan(Y[T]).all().item()
    assert t.equal(Y[:T], (X.double() @ w.t()).to(t.bfloat16))

    spec = _spec(768, 1024, 16, bits=2, asym=True)
    dl, dY, w = _layer(spec, T, spec.m)
    X = t.zeros((T, spec.k), dtype=t.bfloat16, device="cuda")
    dX = t.full((T + 1, spec.k), float("nan"), dtype=t.bfloat16, device="cuda")
    dA, dB = t.empty((spec.m, spec.r), device="cuda"), t.empty((spec.r, spec.k), device="cuda")
    ws = t.empty(LQ.bwd_workspace_bytes(dl.layer, T), dtype=t.uint8, device="cuda")
    LQ.linear_bwd(dl.layer, T, dY.to(t.bfloat16), X, dl.phi0, dl.s, dl.A, dl.B, None, dX, dA, dB, t.empty_like(dl.s),
                  False, ws)
    LQ.get_device_status()
    assert t.isnan(dX[T]).all().item()
    assert t.equal(dX[:T], (dY.double() @ w).to(t.bfloat16))


@pytest.mark.parametrize("T", [1, 9, 16])
@pytest.mark.parametrize("cid,spec", [("bf16_r64", _spec(256, 4096, 64, phi=WL.PHI_BF16)),
                                      ("packed_r64_odd", _spec(384, 6144, 64, phi=WL.PHI_INT_PACKED)),
                                      ("fp16_group", _spec(128, 4096, 48, phi=WL.PHI_FP16, group=128)),
                                      ("q44_r8", _spec(128, 4096, 8))])
def test_few_tokens_on_long_contractions(cid, spec, T):
    """Where a call of a few tokens may leave the kernel made for them: the same product on every path."""
    t = torch()
    dl, X, w = _layer(spec, T, spec.k)
    want = (X.double() @ w.t()).to(t.bfloat16)
    for noalloc in (False, True):
        Y = t.full((T + 1, spec.m), float("nan"), dtype=t.bfloat16, device="cuda")
        args = (dl.layer, T, X.to(t.bfloat16), dl.phi0, dl.s, dl.A, dl.B, None, Y)
        if noalloc:
            LQ.linear_fwd_noalloc(*args)
        else:
            LQ.linear_fwd(*args, t.empty(LQ.fwd_workspace_bytes(dl.layer, T), dtype=t.uint8, device="cuda"))
        LQ.get_device_status()
        assert t.isnan(Y[T]).all().item()
        assert t.equal(Y[:T], want)
