"""Decode attention (a few query vectors per KV head): how its launches are laid out."""
import pytest

from paper_2606_10944_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype_code", [binding.ELM_F32, binding.ELM_BF16])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("vectors", [1, 2, 4, 5, 8])
def test_split_grid_is_resident_at_once(dtype_code, d, vectors):
    """A long list is split over as many CTAs as the device holds, not over more (they would be a second wave)."""
    for problems in (1, 8, 64, 296):
        ctas, resident = binding.debug_decode_grid(problems, vectors, 1, 20000, d, 20000, dtype_code=dtype_code)
        assert problems <= ctas <= resident
