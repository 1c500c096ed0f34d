"""code_params() takes a length in any form that equals it."""
import numpy as np
import pytest
import torch

from paper_1412_6862_gb300 import hd


@pytest.mark.parametrize("form", [int, np.int64, np.uint8, float, np.array, torch.tensor])
def test_forms_of_a_length(form):
    for m in range(2, 9):
        n = (1 << m) - 1
        assert hd.code_params(form(n)) == (m, n - m)
    for n in (0, 1, 8, 100):
        with pytest.raises(hd.HDError) as e:
            hd.code_params(form(n))
        assert e.value.status == hd.HD_ERR_INVALID_N
