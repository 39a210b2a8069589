"""Callers' fields at any alignment, and kept scratch: the four-cell loads and stores of restriction and heat store fall
back to single cells where a field does not start on 16 bytes; the velocity refresh keeps its plan and scratch."""
import numpy as np
import pytest

import lgf_synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2010_13213_gb300.lgf as L
    L.load()
    return L


@pytest.fixture(scope="module")
def table(L):
    t = L.lgf_table_create(8, (12, 12, 12), L.LGF_TBL_BOX_ONLY)
    yield t
    L.lgf_table_destroy(t)


def placed(v, shift, dtype):
    """A copy of v that starts `shift` elements into an allocation."""
    buf = torch.zeros(v.size + 4, dtype=dtype, device="cuda")
    out = buf[shift:shift + v.size].view(v.shape)
    out.copy_(torch.from_numpy(v))
    return out


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("code,dtype", [(0, torch.float64), (1, torch.float32)])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_any_field_alignment(L, table, precision, code, dtype, shift):
    """Same bits from a field and output that start 1, 2 or 3 elements past a 16-byte boundary."""
    rng = np.random.default_rng(3)
    coarse = S.box_blocks((24, 16, 16), 8)
    fine = np.array([(1, 1, 2), (2, 1, 2), (1, 2, 3)], np.int32)
    v = rng.standard_normal((2, len(coarse) + len(fine), 8, 8, 8))
    m = L.Mesh([coarse, fine], 8, 1.0, n_ext=3)
    got = []
    for s in (0, shift):
        f, phi, g = placed(v, s, dtype), placed(np.zeros_like(v), s, dtype), placed(np.zeros_like(v), s, dtype)
        o = L.make_opts(precision=precision)
        L.lgf_poisson_solve(table, m, 2, f.data_ptr(), phi.data_ptr(), code, o)
        L.lgf_heat_apply(table, m, 2, f.data_ptr(), g.data_ptr(), code, 0.05, o)
        torch.cuda.synchronize()
        got.append((phi.cpu().clone(), g.cpu().clone()))
    for a, b in zip(*got):
        assert torch.isfinite(a).all() and torch.equal(a, b)


def test_refresh_keeps_its_plans(L, table):
    """Two meshes in turn on two streams: every call gives what the first call of its mesh gave."""
    rng = np.random.default_rng(9)
    cases = []
    for shape in ((16, 24, 16), (8, 16, 32)):
        blocks = S.box_blocks(shape, 8)
        om = torch.from_numpy(rng.standard_normal((3, len(blocks), 8, 8, 8))).cuda()
        cases.append((L.Mesh([blocks], 8, 0.5), om))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    first = {}
    for k in range(8):
        i, st = k % 2, streams[(k // 2) % 2]
        m, om = cases[i]
        with torch.cuda.stream(st):
            u = torch.full_like(om, float("nan"))
            L.lgf_velocity_refresh(table, m, om.data_ptr(), u.data_ptr(), L.LGF_F64, L.make_opts(precision=2), None,
                                   st.cuda_stream)
        torch.cuda.synchronize()
        assert torch.isfinite(u).all()
        assert torch.equal(first.setdefault(i, u.clone()), u)
