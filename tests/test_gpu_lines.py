"""Line transforms of the block-index FFT mode (csrc/lines.cuh) and the double-float conversions, at the sizes where
they can go wrong: every block count 1..16 of both block sizes (8^3 boxes of odd counts use 8-point second steps),
one-block axes, complex and Hermitian-half fields, more fields than one launch takes, lines without sources.

Tolerances, relative to the largest value of the field: a solve passes at most 6 * 9 butterfly levels (lines of up to
512 points, forward and inverse) and 9 products, each rounding by u at most four times, on values up to 10 times the
rms: 60 * 4 * 10 u = 2.4e3 u with u = 2^-53, 2^-24 and, for double-float, 2^-46."""
import numpy as np
import pytest

import lgf_synth as S
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {0: 2.4e3 * 2.0 ** -53, 1: 2.4e3 * 2.0 ** -24, 2: 2.4e3 * 2.0 ** -46}


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2010_13213_gb300.lgf as L
    L.load()
    return L


@pytest.fixture(scope="module")
def tables(L):
    t = {B: L.lgf_table_create(B, (15, 15, 15), L.LGF_TBL_BOX_ONLY) for B in (8, 16)}
    yield t
    for h in t.values():
        L.lgf_table_destroy(h)


def check(L, tables, B, nb, ncomp, precision, dtype=False, sources=None):
    shape = tuple(B * n for n in nb[::-1])
    blocks = S.box_blocks(shape, B)
    box = S.random_box(shape, sum(nb) + 31 * ncomp, ncomp)
    f = S.box_to_blocks(box, blocks, B)
    roles = None
    if sources is not None:
        on = np.array([sources(*b) for b in blocks])
        roles = np.where(on, 3, 2).astype(np.uint8)
        box = S.blocks_to_box(f * on[None, :, None, None, None], blocks, B, shape)
    ref = oracle.solve_box_fft(box, 0.5)
    td = torch.float32 if dtype else torch.float64
    if dtype:
        ref = oracle.solve_box_fft(box.astype(np.float32).astype(np.float64), 0.5)
    ft = torch.from_numpy(f).to(td).cuda()
    phi = torch.full_like(ft, float("nan"))
    L.lgf_poisson_solve(tables[B], L.Mesh([blocks], B, 0.5, roles=roles), ncomp, ft.data_ptr(), phi.data_ptr(), L.LGF_F32 if dtype else L.LGF_F64,
                        L.make_opts(precision=precision, mac_mode=L.LGF_MAC_BOX))
    torch.cuda.synchronize()
    got = S.blocks_to_box(phi.double().cpu().numpy(), blocks, B, shape)
    tol = max(TOL[precision], 2.0 ** -23 if dtype else 0.0)
    for c in range(ncomp):
        assert np.abs(got[c] - ref[c]).max() <= tol * np.abs(ref[c]).max(), (B, nb, c)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("B,nb", [(8, (1, 2, 3)), (8, (5, 4, 7)), (8, (9, 11, 6)), (8, (13, 8, 15)), (8, (16, 1, 14)),
                                  (8, (10, 12, 1)), (16, (1, 1, 1)), (16, (2, 3, 5)), (16, (4, 7, 6)), (16, (3, 8, 2)),
                                  (16, (9, 1, 11)), (16, (1, 13, 15)), (16, (10, 2, 14)), (16, (12, 1, 16)),
                                  (16, (16, 12, 1)), (16, (11, 9, 1)), (16, (14, 16, 1)), (16, (15, 10, 1))])
def test_every_block_count(L, tables, B, nb, precision):
    check(L, tables, B, nb, 3, precision, dtype=precision == 1)  # FP32 takes the line passes on FP32 fields


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("ncomp", [1, 2, 9])
def test_field_groups(L, tables, ncomp, precision):
    """One real field, one complex field, and five fields over two launches."""
    check(L, tables, 8, (3, 2, 2), ncomp, precision, dtype=precision == 1)


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_float_storage(L, tables, precision):
    check(L, tables, 16, (2, 1, 3), 3, precision, dtype=True)


@pytest.mark.parametrize("B", [8, 16])
def test_lines_without_sources(L, tables, B):
    check(L, tables, B, (3, 3, 3), 2, 2, sources=lambda x, y, z: (x, y, z) == (1, 0, 2))


def test_conversions_round_trip(L):
    """A heat apply with alpha = 0 returns its input: double -> double-float -> double over the whole exponent range,
    at ties and next to powers of two.  hi + lo holds 48 bits where lo is a normal float."""
    rng = np.random.default_rng(5)
    v = rng.standard_normal((1, 2, 8, 8, 8)) * 10.0 ** rng.uniform(-28, 36, (1, 2, 8, 8, 8))
    flat = v.reshape(-1)
    e = np.arange(-95, 120)
    flat[:215] = 2.0 ** e
    flat[215:430] = -(2.0 ** e) * (1 - 2.0 ** -53)
    flat[430:645] = 2.0 ** e * (1 + 2.0 ** -24)  # half an ulp of the high part
    flat[645:650] = [0.0, -0.0, 1e-200, -1e-300, 5e-324]
    small = np.abs(v) < 1e-100
    f = torch.from_numpy(v).cuda()
    g = torch.full_like(f, float("nan"))
    m = L.Mesh([np.array([[0, 0, 0], [1, 0, 0]])], 8, 1.0)
    L.lgf_heat_apply(0, m, 1, f.data_ptr(), g.data_ptr(), L.LGF_F64, 0.0, L.make_opts(precision=L.LGF_PREC_DF32))
    torch.cuda.synchronize()
    got = g.cpu().numpy()
    assert (np.abs(got - v) <= 2.0 ** -48 * np.abs(v))[~small].all()
    assert (got[small] == 0.0).all()
