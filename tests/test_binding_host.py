"""What the binding takes for a tensor."""
import numpy as np
import pytest
import torch

from paper_2608_21308_b200 import binding as E


class Lookalike:
    is_cuda, dtype, shape = True, torch.float32, (1, 1, 16, 64)
    is_contiguous = staticmethod(lambda: True)
    data_ptr = staticmethod(lambda: 1 << 40)


@pytest.mark.parametrize("x", [Lookalike(), np.zeros((1, 1, 16, 64), np.float32), 1 << 40, "q"], ids=["lookalike", "array", "address", "text"])
def test_binding_takes_tensors_only(x):
    """Something that answers like a CUDA tensor is not one: what it calls its address is nobody's to use."""
    with pytest.raises(TypeError):
        E._ptr(x, torch.float32, (1, 1, 16, 64), "q")
