"""Sizes of the caller's scratch, on the host: a buffer that was sized for the largest batch, the most draft
tokens or the longest row does for everything smaller."""
import pytest

from paper_2603_12617_b200 import binding as b


@pytest.mark.parametrize("dtype", [b.SD_DTYPE_F32, b.SD_DTYPE_BF16])
@pytest.mark.parametrize("size", [b.sd_workspace_bytes, b.sd_hint_workspace_bytes])
@pytest.mark.parametrize("k,V", [(1, 8), (1, 5500008), (4, 4097), (5, 50257), (8, 128256), (3, 32000), (64, 65544)])
def test_more_sequences_never_need_less(size, dtype, k, V):
    sizes = [size(B, k, V, dtype) for B in list(range(1, 400)) + [2 ** n for n in range(9, 15)]]
    assert sizes[0] > 0 and all(p <= q for p, q in zip(sizes, sizes[1:]))


@pytest.mark.parametrize("dtype", [b.SD_DTYPE_F32, b.SD_DTYPE_BF16])
@pytest.mark.parametrize("size", [b.sd_workspace_bytes, b.sd_hint_workspace_bytes])
@pytest.mark.parametrize("B", [1, 13, 256])
def test_longer_rows_and_more_tokens_never_need_less(size, dtype, B):
    sizes = [size(B, 5, V, dtype) for V in list(range(1, 3000)) + list(range(3000, 160000, 37))]
    assert all(p <= q for p, q in zip(sizes, sizes[1:]))
    sizes = [size(B, k, 50257, dtype) for k in range(1, 65)]
    assert all(p <= q for p, q in zip(sizes, sizes[1:]))


@pytest.mark.parametrize("dtype", [b.SD_DTYPE_F32, b.SD_DTYPE_BF16])
def test_smaller_ensembles_never_need_more(dtype):
    """Fewer sequences, tokens, entries or learners: scratch for the larger call does."""
    size = b._lib.sd_ensemble_workspace_bytes
    for k, V, N in [(1, 8, 1), (8, 128256, 3), (4, 151936, 3), (3, 32000, 8), (64, 65544, 2), (2, 5500008, 5)]:
        sizes = [size(B, k, V, dtype, N) for B in list(range(1, 400)) + [2 ** n for n in range(9, 15)]]
        assert sizes[0] > 0 and all(p <= q for p, q in zip(sizes, sizes[1:]))
        sizes = [size(6, k, V, dtype, n) for n in range(1, 9)]
        assert all(p <= q for p, q in zip(sizes, sizes[1:]))
    for B in (1, 5, 13, 256):
        sizes = [size(B, 5, V, dtype, 3) for V in list(range(1, 3000)) + list(range(3000, 160000, 37))]
        assert all(p <= q for p, q in zip(sizes, sizes[1:]))
        sizes = [size(B, k, 50264, dtype, 3) for k in range(1, 65)]
        assert all(p <= q for p, q in zip(sizes, sizes[1:]))
