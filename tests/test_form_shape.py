"""form_shape keeps its answers; what it refuses, it refuses after an equal key too (no GPU needed)."""
import ctypes

import numpy as np
import pytest


@pytest.mark.parametrize("form", [0.0, np.float64(0)])
def test_refused_types_stay_refused(form):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1103_0066_gb300 as fem
    fem.form_shape.cache_clear()
    with pytest.raises(ctypes.ArgumentError):
        fem.form_shape(form, 3)
    assert fem.form_shape(0, 3) == fem.form_shape(np.int64(0), 3) == (4, 4)  # an integer of any kind is one
    with pytest.raises(ctypes.ArgumentError):
        fem.form_shape(form, 3)
