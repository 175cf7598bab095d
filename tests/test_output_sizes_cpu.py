"""hg_evaluate refuses result arrays that hold fewer than 3 m values before it calls the
library (no GPU): device arrays are written by a kernel, which nothing would stop."""
import numpy as np
import pytest

from paper_1207_2367_gb300 import binding as hg


@pytest.mark.parametrize("which", range(3))
@pytest.mark.parametrize("shape", [(4, 3), (14,), (0,), (5, 2)])
def test_short_results_are_refused(which, shape):
    out = [None, np.empty((5, 3)), np.empty(20)]
    out[which] = np.empty(shape)
    with pytest.raises(ValueError, match="values"):
        hg.hg_evaluate(None, None, 5, *out)


def test_room_for_the_results_is_enough():
    """Exactly 3 m values, more of them, or no array: on to the library, which refuses the
    missing context."""
    for out in ([np.empty((5, 3))] * 3, [np.empty(40), None, np.empty((5, 3, 2))], [None] * 3):
        with pytest.raises(hg.HGError):
            hg.hg_evaluate(None, None, 5, *out)
