"""Arguments that the torch entry points refuse, with the error that says why."""
import pytest

torch = pytest.importorskip("torch")

import paper_2002_03258_gb300 as pkg  # noqa: E402


def colmajor(rows, cols, dtype=torch.float64):
    return torch.zeros((cols, rows), dtype=dtype).t()


@pytest.mark.parametrize("f,x,y", [(pkg.tsm2r, (8, 4), (4, 2)), (pkg.tsm2l, (8, 4), (4, 2)), (pkg.tsm2r_t, (8, 4), (8, 2)),
                                   (pkg.rankk, (8, 2), (4, 2))])
def test_tensors_on_the_host_are_refused(f, x, y):
    with pytest.raises(ValueError, match="CUDA device"):
        f(colmajor(*x), colmajor(*y))
    with pytest.raises(TypeError, match="both"):
        f(colmajor(*x), colmajor(*y, dtype=torch.float32))
