"""Sizes that the library asks its callers for, on both sides of the rules that choose a kernel."""
import pytest

import paper_2609_07816_gb300 as kdn


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_07816_gb300 import build
    build.build()


def _desc(B, T, H, out=kdn.KDN_BF16, **kw):
    return kdn.make_desc(B, T, H, 128, 128, kdn.KDN_BF16, out_dtype=out, **kw)


@pytest.mark.parametrize("out", [kdn.KDN_F32, kdn.KDN_BF16])
@pytest.mark.parametrize("B,T,H", [(2, 130, 3), (1, 449, 14), (8, 4096, 16), (8, 4095, 16), (2, 1999, 16),
                                   (64, 1000, 32)])
def test_saved_context_is_one_record_a_chunk(B, T, H, out):
    """162 KB and 128 floats per 64-token chunk at every size: no kernel choice adds to it."""
    for variant in (0, 1):
        assert kdn.saved_bytes(_desc(B, T, H, out), variant) == B * H * ((T + 63) // 64) * (165888 + 512)
