"""The weight gradients from the code bytes of the codes pass (clip mask in the top bit) against the
kernels that recompute the low-rank tile: the same G, code and mask per weight, so dA, dB and ds
agree bit for bit, over both work schedules, ragged token counts, ranks of one to four K steps,
clipping grids, groups, zero offsets and several tiles per persistent CTA."""
import pytest

from paper_2406_06385_gb300 import lrqat as LQ
from paper_2406_06385_gb300 import workloads as WL

from gpu_util import DeviceLayer, to_dev, torch

pytestmark = pytest.mark.gpu


def _spec(m, k, r, bits=4, group=0, phi=WL.PHI_QFIXED, act=0, asym=False, ub=False, std=0.2):
    return WL.LayerSpec("c", m, k, r, float(r), bits, group, phi, act, a_std=std, b_std=std, asym=asym,
                        w_row_shift=0.03 if asym else 0.0, u_bf16=ub)


CASES = [
    ("one_tile_one_token", _spec(256, 256, 8), 1),
    ("rank_not_direct", _spec(256, 512, 20), 97),
    ("rank_48_clip", _spec(512, 256, 48, bits=2, std=1.0), 450),
    ("rank_64_group", _spec(256, 768, 64, group=128), 1000),
    ("int3_packed_a8", _spec(512, 512, 32, bits=3, phi=WL.PHI_INT_PACKED, act=8), 333),
    ("asym_group", _spec(256, 512, 16, bits=2, group=256, asym=True), 2070),
    ("bf16_base_ubf16", _spec(256, 512, 32, phi=WL.PHI_BF16, ub=True), 130),
    ("bits_7", _spec(256, 256, 32, bits=7), 64),
    ("many_tiles", _spec(2560, 2304, 32), 700),
]


def _grads(spec, T, dl, X, dY, s_x):
    t = torch()
    out = [t.empty((T, spec.k), dtype=t.int16, device="cuda"), t.empty((spec.m, spec.r), device="cuda"),
           t.empty((spec.r, spec.k), device="cuda"), t.empty_like(dl.s)]
    ws = t.empty(LQ.bwd_workspace_bytes(dl.layer, T), dtype=t.uint8, device="cuda")
    LQ.linear_bwd(dl.layer, T, dY, X, dl.phi0, dl.s, dl.A, dl.B, s_x, *out, False, ws)
    LQ.get_device_status()
    return out


@pytest.mark.parametrize("schedule", ["split", "tail"])
@pytest.mark.parametrize("cid,spec,T", CASES, ids=[c[0] for c in CASES])
def test_gradients_from_codes_equal_those_from_the_low_rank_tile(cid, spec, T, schedule, lowrank_path, dw_schedule):
    t = torch()
    dw_schedule(schedule)
    data = WL.make_layer(spec, T, seed=4)
    dl = DeviceLayer(data, 1.05)
    X, dY = to_dev(data.X_bits), to_dev(data.dY_bits)
    s_x = t.full((1,), 0.02, device="cuda") if spec.act_bits else None
    got = {}
    for path in ("tile", "codes"):
        lowrank_path(path)
        got[path] = _grads(spec, T, dl, X, dY, s_x)
    for name, a, b in zip(("dA", "dB", "ds"), got["tile"][1:], got["codes"][1:]):
        assert t.equal(a, b), name
    a, b = (got[p][0].view(t.bfloat16).float() for p in ("tile", "codes"))
    assert float((a - b).norm() / b.norm()) <= 4e-3


WIDE_CASES = [
    ("r96_few_tiles", _spec(512, 768, 96), 700),
    ("r72_not_direct_odd_tokens", _spec(2560, 2304, 68), 333),
    ("r256_mixed_parts", _spec(1280, 1536, 256), 1000),
    ("r128_group_asym", _spec(768, 2816, 128, bits=3, group=128, asym=True), 2081),
]


@pytest.mark.parametrize("schedule", ["auto", "split", "tail"])
@pytest.mark.parametrize("cid,spec,T", WIDE_CASES, ids=[c[0] for c in WIDE_CASES])
def test_pair_gradients_of_large_ranks(cid, spec, T, schedule, gemm_variant, dw_schedule):
    """Ranks above 64 on pairs against one SM: the same token ranges per 128 x 128 tile, so dU is the
    same bit for bit and only the order of fp32 sums of partials differs (2^-18 relative)."""
    t = torch()
    dw_schedule(schedule)
    data = WL.make_layer(spec, T, seed=4)
    dl = DeviceLayer(data, 1.05)
    X, dY = to_dev(data.X_bits), to_dev(data.dY_bits)
    got = {}
    for variant in ("single", "pair"):
        gemm_variant(variant)
        got[variant] = _grads(spec, T, dl, X, dY, None)[1:]
    for name, a, b in zip(("dA", "dB", "ds"), *got.values()):
        assert float((a - b).norm() / a.norm()) <= 2.0 ** -18, name


TILE_CASES = [
    # odd numbers of 128-row blocks in both directions, token counts around the tiles' edges
    ("odd_blocks", _spec(384, 640, 32), 225),
    ("one_block", _spec(128, 128, 8), 33),
    ("odd_group_asym", _spec(128, 384, 16, bits=3, group=128, asym=True), 449),
    ("two_rounds", _spec(640, 384, 32, group=128), 20011),
    ("bf16_8_bits", _spec(384, 256, 16, bits=8, phi=WL.PHI_BF16), 257),
]


@pytest.mark.parametrize("path", ["tile", "codes"])
@pytest.mark.parametrize("cid,spec,T", TILE_CASES, ids=[c[0] for c in TILE_CASES])
def test_pair_gemm_equals_the_one_sm_kernel(cid, spec, T, path, lowrank_path, gemm_variant):
    """Y and dX of the pair kernel against the one-SM kernel's: the same W_hat and products summed in
    the same K order, so bf16 outputs agree to a rounding of sums that differ in the last fp32 bits."""
    t = torch()
    lowrank_path(path)
    data = WL.make_layer(spec, T, seed=6)
    dl = DeviceLayer(data, 1.05)
    X, dY = to_dev(data.X_bits), to_dev(data.dY_bits)
    got = {}
    for variant in ("single", "pair"):
        gemm_variant(variant)
        Y = t.full((T + 1, spec.m), 0x7FC0, dtype=t.int16, device="cuda")
        ws = t.empty(LQ.fwd_workspace_bytes(dl.layer, T), dtype=t.uint8, device="cuda")
        LQ.linear_fwd(dl.layer, T, X, dl.phi0, dl.s, dl.A, dl.B, None, Y, ws)
        dX = _grads(spec, T, dl, X, dY, None)[0]
        assert bool((Y[T] == 0x7FC0).all())   # nothing is written past the last token
        got[variant] = [x.view(t.bfloat16).float() for x in (Y[:T], dX)]
    for a, b in zip(*got.values()):
        assert bool(t.isfinite(b).all())
        assert float((a - b).norm() / a.norm()) <= 2.0 ** -9


def test_codes_of_unaligned_factors_and_outputs():
    """The merge writes the same codes from padded factors, and to a 16-byte aligned output that is
    not 32-byte aligned."""
    t = torch()
    spec = _spec(384, 640, 32, bits=3)
    dl = DeviceLayer(WL.make_layer(spec, 1, seed=2, with_activations=False))
    out = [t.empty(spec.m * spec.k + 16, dtype=t.int8, device="cuda")[o:o + spec.m * spec.k] for o in (0, 16)]
    for o in out:
        LQ.merge(dl.layer, dl.phi0, dl.A, dl.B, o)
    LQ.get_device_status()
    assert t.equal(out[0], out[1])
    assert int(out[0].min()) == -4 and int(out[0].max()) == 3
