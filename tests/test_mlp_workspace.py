"""Workspace of the coefficient-forecasting MLP (a host-side computation)."""
import ctypes

import pytest

from paper_1406_4254_gb300 import etics


def need(dims, batch):
    return etics.load().etics_mlp_workspace_bytes(ctypes.byref(etics.MlpShape.of(dims)), batch)


@pytest.mark.parametrize("width", [4, 256, 1024, 1028, 65536])
@pytest.mark.parametrize("batch", [1, 1000, 4865, 19440])
def test_a_wide_layer_needs_no_sums_per_chunk_of_rows(width, batch):
    """One layer 8 -> width: its output, two errors in FP32 and bf16 and one
    product (4 + 8 + 4 + 4 bytes per column and row), 304 rows of FP64 column
    sums (or one per 128 rows) and the K slices of the weight gradient, as many
    as bring its tiles of 64 columns to 304 blocks, 64 at most.  The narrow kernels' 304 partial gradients, 8 x 4 bytes per column
    each, may come on top only up to 1024 columns."""
    columns = max(304, (batch + 127) // 128) * 8 + min(64, -(-304 // -(-width // 64))) * 8 * 4
    narrow = 304 * 8 * 4 if width <= 1024 else 0
    rows = batch * (8 * width + 12 * max(8, width))      # the errors are as wide as the widest
    assert need([8, width], batch) <= rows + width * (columns + narrow) + (1 << 16)


@pytest.mark.parametrize("dims", [[8, 64, 64, 3], [8, 1024], [64, 64, 64, 64, 64], [4, 8, 8],
                                  [8, 4096, 8], [16, 3], [8, 16, 1], [8, 256, 256, 3], [256, 256],
                                  [9720, 256, 256, 1215], [1000, 70, 500, 63], [2000, 64]])
def test_workspace_does_not_shrink_with_more_rows(dims):
    """A workspace sized for the largest batch serves every smaller one."""
    sizes = [need(dims, b) for b in range(1, 42000)]
    assert all(b >= a for a, b in zip(sizes, sizes[1:]))


@pytest.mark.gpu
@pytest.mark.parametrize("dims,batch", [([8, 1024, 3], 33), ([8, 1028, 3], 33), ([3, 2048], 130)])
def test_layers_around_the_widest_narrow_one_match_oracle(dims, batch):
    """Both routes of the input layer's weight gradient, on either side of 1024."""
    import test_surrogate
    test_surrogate.test_gradient_matches_oracle(dims, batch)
