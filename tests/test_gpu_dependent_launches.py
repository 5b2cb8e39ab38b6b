"""Kernels of one call overlap at their ends (programmatic dependent launches): calls issued back to
back on shared workspaces give the same bits as with every kernel run to its end before the next
starts (tracing puts an event between any two), eagerly and from a CUDA graph."""
import pytest

from paper_2406_06385_gb300 import lrqat as LQ
from paper_2406_06385_gb300 import workloads as WL

from gpu_util import phi_buffer, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k,r,T,group,act", [
    (256, 256, 4, 64, 0, 0),        # six short kernels: the shortest overlaps; adapter layouts first
    (512, 768, 32, 7, 0, 0),        # the few-token forward
    (1024, 1280, 96, 300, 128, 0),  # group-wise, rounds of ranks
    (2048, 1024, 32, 1000, 0, 8),   # the activation quantizer between the kernels
])
def test_back_to_back_calls_match_serialised_ones(m, k, r, T, group, act):
    t = torch()
    spec = WL.LayerSpec("d", m, k, r, float(r), 4, group, WL.PHI_QFIXED, act)
    L = LQ.Layer.from_spec(spec)
    g = t.Generator(device="cuda").manual_seed(m + T)
    rnd = lambda *n, f=1.0: (t.randn(n, generator=g, device="cuda") * f).to(t.bfloat16)
    s = t.empty((m, k // group) if group else (m,), device="cuda")
    phi = phi_buffer(spec)
    W = t.randn((m, k), generator=g, device="cuda") * 0.02
    LQ.range_minmax(L, W, s)
    LQ.downcast(L, W, s, phi)
    batches = [(rnd(T, k), rnd(T, m), rnd(m, r, f=1 / 64), rnd(r, k, f=1e-3)) for _ in range(4)]
    s_x = t.full((1,), 0.03, device="cuda") if act else None
    wf = t.empty(max(LQ.fwd_workspace_bytes(L, T), 16), dtype=t.uint8, device="cuda")
    wb = t.empty(LQ.bwd_workspace_bytes(L, T), dtype=t.uint8, device="cuda")
    empty = lambda *n, dtype=t.bfloat16: t.zeros(n, dtype=dtype, device="cuda")
    outs = [dict(Y=empty(T, m), dX=empty(T, k), dA=empty(m, r, dtype=t.float32), dB=empty(r, k, dtype=t.float32),
                 ds=t.zeros_like(s)) for _ in batches]

    def run():
        for (X, dY, A, B), o in zip(batches, outs):
            LQ.linear_fwd(L, T, X, phi, s, A, B, s_x, o["Y"], wf)
            LQ.linear_bwd(L, T, dY, X, phi, s, A, B, s_x, o["dX"], o["dA"], o["dB"], o["ds"], False, wb)

    def take():
        t.cuda.synchronize()
        got = [{n: x.clone() for n, x in o.items()} for o in outs]
        for o in outs:
            for x in o.values():
                x.zero_()
        t.cuda.synchronize()
        return got

    LQ.trace_enable(True)
    run()
    want = take()
    LQ.trace_read()
    LQ.trace_enable(False)
    graph, side = t.cuda.CUDAGraph(), t.cuda.Stream()
    with t.cuda.graph(graph, stream=side):
        run()
    take()
    for go in [run] * 5 + [graph.replay] * 5:
        go()
        for a, b in zip(take(), want):
            for n in a:
                assert t.equal(a[n], b[n]), n
    LQ.get_device_status()
