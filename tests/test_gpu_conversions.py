"""Double-float to double: hi + lo correctly rounded, also just below a power of two, where the ulp of the sum is half that of
the high part.  A heat apply with alpha = 0 returns its input."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2010_13213_gb300.lgf as L
    L.load()
    return L


def round_trip(L, v):
    f = torch.zeros(8 ** 3, dtype=torch.float64, device="cuda")
    f[:len(v)] = torch.from_numpy(v)
    g = torch.full_like(f, float("nan"))
    L.lgf_heat_apply(0, L.Mesh([np.array([[0, 0, 0]])], 8, 1.0), 1, f.data_ptr(), g.data_ptr(), L.LGF_F64, 0.0,
                     L.make_opts(precision=L.LGF_PREC_DF32))
    torch.cuda.synchronize()
    return g.cpu().numpy()[:len(v)]


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("e", [-70, -1, 0, 1, 40, 110])
def test_values_that_two_floats_hold_come_back_equal(L, e, sign):
    """2^e (1 + k ulp) from either side, and odd high parts: the low part has at most 24 bits in each."""
    near = [1.0 - k * 2.0 ** -53 for k in (0, 1, 2, 3, 5, 2 ** 20 + 1, 2 ** 23 - 1, 2 ** 23 + 1)]
    near += [1.0 + k * 2.0 ** -52 for k in (1, 2, 3, 5, 2 ** 20 + 1, 2 ** 23 - 1)]
    odd = [1.0 + j * 2.0 ** -23 + k * 2.0 ** -47 for j in (1, 2, 2 ** 22, 2 ** 23 - 1) for k in (-3, -1, 0, 1, 3, 2 ** 20)]
    v = sign * np.array(near + odd) * 2.0 ** e
    assert np.array_equal(round_trip(L, v), v)
