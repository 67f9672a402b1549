"""The two forms of the fused FP32 kernel's chunks with knots: group 4 takes one or the other by tile, split, rows
and items per CTA, groups 2 and 8 always the plain one.  Both do the same operations in the same order, so
log L agrees bit for bit over the groups, on either side of each line of the rule."""
import numpy as np
import pytest

from tests import _forms
from tests._workloads import gpu_eval

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_channels,sgwb", [(2, 0), (3, 1), (3, 2)])
@pytest.mark.parametrize("n_bins,n_states,tile_bins", [
    (4001, 64, 512),       # split items of two rows
    (2000, 20, 512),       # rows of bins, few items
    (66, 20, 64),
    (9000, 300, 384),      # the plain form's tiles, split and not
    (60001, 300, 384),
    (60001, 300, 512),     # fewer than two items per CTA
    (40000, 2100, 512),    # more
    (40000, 2100, 416),
])
def test_groups_agree_bit_for_bit(n_bins, n_states, tile_bins, n_channels, sgwb):
    wl, P = _forms.chunk_workload(n_bins, n_states, n_channels, sgwb)
    ref = None
    for group in (4, 2, 8):
        L, St = gpu_eval(wl, P, 0, tiling=dict(tile_bins=tile_bins, states_per_cta=128, group=group))
        if ref is None:
            ref = L, St   # (some -inf: close knots overshoot by hundreds of decades)
            assert np.isfinite(L).mean() > 0.5
        np.testing.assert_array_equal(St, ref[1])
        np.testing.assert_array_equal(L, ref[0])
