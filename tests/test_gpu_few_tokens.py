"""The few-token forward (up to 16 tokens, ranks up to 64) against the pair GEMM with the in-stage
low-rank tile: the same codes and products, summed in another order."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2406_06385_gb300 import lrqat as LQ
from paper_2406_06385_gb300 import workloads as WL

from gpu_util import DeviceLayer, near_bf16_boundary, oracle_layer, to_dev, torch

pytestmark = pytest.mark.gpu


def _spec(m, k, r, bits=4, group=0, phi=WL.PHI_QFIXED, act=0, per_token=False, asym=False, ub=False, std=0.2):
    return WL.LayerSpec("f", m, k, r, float(r), bits, group, phi, act, a_std=std, b_std=std, asym=asym,
                        w_row_shift=0.03 if asym else 0.0, act_per_token=per_token, u_bf16=ub)


CASES = [
    ("q44", _spec(256, 1152, 32)),
    ("one_block_pair", _spec(128, 128, 8)),
    ("int3_r20", _spec(128, 640, 20, bits=3, phi=WL.PHI_INT_PACKED)),
    ("r48_group", _spec(384, 512, 48, group=256)),
    ("r64_clip_asym_group", _spec(128, 2304, 64, bits=2, group=128, asym=True, std=1.0)),
    ("asym_rows", _spec(128, 384, 16, bits=2, asym=True)),
    ("a8_tensor", _spec(128, 512, 32, act=8)),
    ("a8_token", _spec(128, 512, 32, act=8, per_token=True)),
    ("bf16_8_bits", _spec(128, 256, 16, bits=8, phi=WL.PHI_BF16)),
    ("fp16", _spec(128, 384, 32, phi=WL.PHI_FP16)),
    ("e4m3", _spec(128, 384, 32, phi=WL.PHI_FP8_E4M3)),
    ("e5m2_ubf16", _spec(128, 256, 32, phi=WL.PHI_FP8_E5M2, ub=True)),
]


def _forward(L, dl, T, X, s_x, m, noalloc):
    t = torch()
    Y = t.full((T + 1, m), 0x7FC0, dtype=t.int16, device="cuda")
    if noalloc:
        LQ.linear_fwd_noalloc(L, T, X, dl.phi0, dl.s, dl.A, dl.B, s_x, Y)
    else:
        ws = t.empty(LQ.fwd_workspace_bytes(L, T), dtype=t.uint8, device="cuda")
        LQ.linear_fwd(L, T, X, dl.phi0, dl.s, dl.A, dl.B, s_x, Y, ws)
    LQ.get_device_status()
    assert bool((Y[T] == 0x7FC0).all())   # nothing is written past the last token
    return Y[:T]


@pytest.mark.parametrize("T", [1, 7, 8, 9, 16, 17])
@pytest.mark.parametrize("cid,spec", CASES, ids=[c[0] for c in CASES])
def test_few_tokens_match_the_pair_gemm(cid, spec, T, lowrank_path):
    """Y within the bf16 rounding of sums in another order, plus the codes of exact products next to
    a rounding tie (2^-8 relative covers both)."""
    t = torch()
    data = WL.make_layer(spec, T, seed=8)
    dl = DeviceLayer(data, 1.05)
    X = to_dev(data.X_bits)
    s_x = t.full((1,), 0.02, device="cuda") if spec.act_bits and not spec.act_per_token else None
    lowrank_path("auto")
    few = _forward(dl.layer, dl, T, X, s_x, spec.m, False)
    if T <= 16:   # (17 tokens are past the kernel's range: the pair GEMM on either path)
        assert t.equal(few, _forward(dl.layer, dl, T, X, s_x, spec.m, True))
    lowrank_path("tile")
    ref = _forward(dl.layer, dl, T, X, s_x, spec.m, False).view(t.bfloat16).float()
    few = few.view(t.bfloat16).float()
    assert bool(t.isfinite(few).all())
    assert float((few - ref).norm() / ref.norm()) <= 2.0 ** -8


@pytest.mark.parametrize("zero_B", [True, False], ids=["ties", "lowrank"])
@pytest.mark.parametrize("cid,spec", [c for c in CASES if not c[1].act_bits], ids=[c[0] for c in CASES if not c[1].act_bits])
def test_few_token_codes(cid, spec, zero_B):
    """With s = 1 and rows of the identity as tokens, Y holds the codes (minus the zero offsets):
    equal to the oracle's outside near-ties, and with B = 0 on exact ties too."""
    t = torch()
    data = WL.make_layer(spec, 1, seed=5, with_activations=False, zero_B=zero_B)
    dl = DeviceLayer(data)
    z = dl.z
    dl.s = t.ones_like(dl.s)
    eye = t.eye(spec.k, dtype=t.bfloat16, device="cuda").view(t.int16)
    rows = [_forward(dl.layer, dl, 16, eye[i:i + 16].contiguous(), None, spec.m, False) for i in range(0, spec.k, 16)]
    got = t.cat(rows).view(t.bfloat16).float().cpu().numpy().T
    OL = oracle_layer(spec)
    if spec.asym:
        s0, z0 = O.minmax_range_asym(data.W0, OL)
        phi = O.downcast(data.W0, s0, OL, z0)
    else:
        s0, z0 = O.minmax_scale(data.W0, OL), None
        phi = O.downcast(data.W0, s0, OL)
    fq = O.fake_quant_weight(phi, np.ones_like(s0), data.A, data.B, OL, z0)
    differ = got != fq["cz"]
    exempt = np.zeros_like(differ) if zero_B else O.near_tie(fq["u"])
    if spec.u_bf16 and not zero_B:
        exempt |= near_bf16_boundary(data.A, data.B)
    assert not (differ & ~exempt).any()
