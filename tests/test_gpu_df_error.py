"""The rounding error of double-float composite solves, averaged over seeds, is no larger than that of the block-index
evaluation (FFTs of the block indices around FFTs within the blocks), which the line transforms replaced.

Bounds: the block-index evaluation's mean relative 2-norm error on the same inputs (measured once on a GB300, against the
same 64-bit values), plus 5 % for the spread of the means over seeds."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def ring(levels, nxy, nz, res, sigma, n_ext):
    return dict(kind="amr", levels=levels, nxy=nxy, nz=nz, res=res, sigma=sigma, n_ext=n_ext, precision="df32")


@pytest.mark.parametrize("case,seeds,block_form", [(ring(3, 192, 96, 64, 0.2, 16), 24, 5.31e-15),
                                                   (ring(3, 144, 96, 46, 0.141, 8), 2, 5.34e-15),
                                                   (ring(2, 144, 80, 45, 0.142, 8), 2, 4.81e-15)])
def test_composite_error(case, seeds, block_form):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import perf.cases as C
    total = 0.0
    for seed in range(1, seeds + 1):
        state = C.prepare(case, seed)
        got = C.run(state)
        torch.cuda.synchronize()
        ref = C.exact(case, seed)
        total += float(torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref))
        del state, got, ref
    assert total / seeds <= 1.05 * block_form
