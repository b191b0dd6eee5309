"""The shapes the tensor-core descriptors take, which the library decides before any device work (no recipes: nothing
runs).  Beyond them the ring of operand blocks is shorter than the way between two tasks of a warp."""
from types import SimpleNamespace

import pytest

from paper_1806_09819_gb300 import build as B
from paper_1806_09819_gb300 import leea


def _ask(dims):
    B.build()
    leea.leea_descriptors(4, dims, leea.Params(precision=1), 1, 1, *([None] * 7), 0, None, 32, None, stream=SimpleNamespace(cuda_stream=None))


@pytest.mark.parametrize("dims", [[784, 112, 10], [1024, 16, 10], [960, 64, 10], [832, 128, 10], [16, 16, 10]], ids=str)
def test_accepted(dims):
    _ask(dims)


@pytest.mark.parametrize("dims", [[1440, 16, 10], [1360, 32, 10], [1296, 48, 10], [1280, 64, 10], [1040, 16, 10],
                                  [848, 128, 10], [784, 144, 10], [792, 16, 10]], ids=str)
def test_refused(dims):
    with pytest.raises(leea.LeeaError, match="descriptors need"):
        _ask(dims)
