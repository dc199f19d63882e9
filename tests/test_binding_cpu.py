"""What the binding accepts as a frame: anything with a tensor's methods, its
shape a tuple or a list."""
import pytest

import paper_2110_14934_gb300 as G


class Frame:
    def __init__(self, shape, size):
        self.shape, self._size = shape, size

    def element_size(self):
        return self._size


@pytest.mark.parametrize("kind", [tuple, list])
def test_shapes_as_tuples_and_lists(kind):
    G._check_frame(Frame(kind((4, 5, 3)), 1), Frame(kind((4, 5)), 2), 4, 5)
    G._check_frame(Frame(kind((1, 4, 5, 3)), 1), Frame(kind((1, 4, 5)), 2), 4, 5)
    with pytest.raises(ValueError):
        G._check_frame(Frame(kind((5, 4, 3)), 1), Frame(kind((4, 5)), 2), 4, 5)
    with pytest.raises(ValueError):
        G._check_frame(Frame(kind((4, 5, 3)), 1), Frame(kind((5, 4)), 2), 4, 5)
