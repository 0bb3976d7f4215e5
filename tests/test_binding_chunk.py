"""``chunk`` is a whole number: a fraction is refused, not cut off."""
import numpy as np
import pytest

import paper_2609_07816_gb300 as kdn
from test_binding_cpu import acts, fake, fake_tensor  # noqa: F401


@pytest.mark.parametrize("chunk", [32.5, 32.0, "32"])
def test_chunk_must_be_a_whole_number(fake, chunk):  # noqa: F811
    x = acts("diag", 1, 70, 2, 128, 128)
    n = len(fake.calls)
    with pytest.raises(TypeError):
        kdn.kdn_diag_fwd(*x, chunk=chunk)
    assert len(fake.calls) == n
    kdn.kdn_diag_fwd(*x, chunk=np.int64(32))
    assert len(fake.calls) == n + 1
