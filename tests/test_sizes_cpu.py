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


@pytest.mark.parametrize("B,T,H", [(8, 4095, 16), (64, 1000, 32), (33, 191, 2), (8, 4096, 16)])
def test_a_forward_pays_for_no_backward(B, T, H):
    """More sequences than the parallel forward takes: a status word, at any length; the ragged
    training backward asks for its partial last chunk (80 KB a sequence) by itself."""
    d = _desc(B, T, H)
    assert kdn.workspace_bytes(d, 0) == 256
    two = kdn.kdn_kernel_launches(d, 0, 6) > 1
    assert two or (B, H) != (8, 16)
    assert kdn.workspace_bytes(d, 0, "saved") == 256 + (B * H * 81920 if T % 64 and two else 0)
    assert kdn.workspace_bytes(_desc(B, T, H, kdn.KDN_F32), 0, "saved") == 256
    assert kdn.workspace_bytes(d, 1, "saved") == 256


@pytest.mark.parametrize("B,T,H", [(1, 65472, 16), (1, 131008, 16), (2, 40001, 16), (1, 1 << 20, 1), (7, 20001, 8)])
def test_the_parallel_forward_is_bounded(B, T, H):
    """Few sequences of any length: the records of at most 2048 chunks and a state per sequence."""
    n = kdn.workspace_bytes(_desc(B, T, H), 0)
    if T != 1 << 20:  # (that one is cut into segments)
        assert n <= 256 + 2048 * (66560 + 516) + 512 + B * H * (128 * 129 * 4)


def test_launch_counts():
    n = kdn.kdn_kernel_launches
    for d, bf in ((_desc(8, 4096, 16), True), (_desc(8, 4096, 16, kdn.KDN_F32), False), (_desc(2, 1999, 16), True)):
        assert [n(d, 0, op) for op in (1, 3, 4)] == [2, 1, 1]
        assert n(d, 0, 6) == (3 if bf else 1)  # tiles, memory, chunks; or the sweep
        assert n(d, 1, 6) == 1
    assert n(_desc(2, 130, 3), 0, 6) == 1  # too few chunks for the two-kernel backward
    assert n(_desc(2, 130, 3, chunk=32), 0, 6) == -1
    # the parallel forward of few sequences: one launch a slice (2048 chunks of all sequences)
    assert n(_desc(2, 1999, 16), 0, 0) == 1 and n(_desc(2, 5000, 16), 0, 0) == 2 and n(_desc(1, 65472, 16), 0, 0) == 8
