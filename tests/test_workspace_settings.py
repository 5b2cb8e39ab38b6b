"""A backward workspace of a layer of rank above 64 serves every setting of lrqat_set_gemm_variant, whichever was
set when its size was asked for."""
import pytest

from paper_2406_06385_gb300 import lrqat as LQ


@pytest.mark.parametrize("r", [65, 96, 128, 256])
@pytest.mark.parametrize("m,k", [(256, 256), (4096, 4096), (13824, 5120), (384, 640), (256, 384)])
def test_backward_size_of_high_ranks_covers_the_gemm_variants(m, k, r, gemm_variant):
    L = LQ.Layer(m, k, r, float(r), 4, 0, LQ.PHI_QFIXED, 0, None, 0, 0)
    for T in (1, 64, 1000, 1024, 2048, 8192):
        sizes = set()
        for variant in ("auto", "single", "pair"):
            gemm_variant(variant)
            sizes.add(LQ.bwd_workspace_bytes(L, T))
        assert len(sizes) == 1 and sizes.pop() > 0, T
