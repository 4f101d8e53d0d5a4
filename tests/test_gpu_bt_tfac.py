"""The triangular factors of the blocked back-transformation: panels of 128 reflectors,
a last panel of one, of a part of a lane's four columns and of all but one, checked
through B (Q orthogonal, B D^2 B^T = C)."""
import pytest

from parity_util import have_gpu
from test_gpu_trd_reduce import check, decompose

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a GPU")]


# reflectors n - 1: one panel more than full ones by 1, 2, 5, 64, 65, 127 and 0
@pytest.mark.parametrize("n", [258, 259, 262, 321, 322, 384, 385, 641])
def test_last_panel(n):
    check(decompose([n], "spread")[0], n)


def test_panels_of_a_batch():
    for n, g in zip([520, 300, 700], decompose([520, 300, 700], "spread")):
        check(g, n)
