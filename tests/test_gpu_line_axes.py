"""Box convolutions with every line length on every axis (the x, y and z passes are kernels of their own), and the
block-index passes that FP32 arithmetic on FP64 fields runs.

Tolerance of the relative 2-norm: a solve passes at most 60 butterfly levels and products (lines of up to 512 points
along three axes, forward and inverse) of up to four roundings each; with independent signs about sqrt(240) = 16
roundings, doubled for products of unnormalised values: 32 u, u = 2^-53, 2^-24 and, for double-float, 2^-48."""
import numpy as np
import pytest

import lgf_synth as S
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = {0: 2.0 ** -53, 1: 2.0 ** -24, 2: 2.0 ** -48}


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


def check(L, tables, B, nb, ncomp, precision, single):
    shape = tuple(B * n for n in nb[::-1])
    blocks = S.box_blocks(shape, B)
    box = S.random_box(shape, sum(nb) + 17 * ncomp, ncomp)
    if precision == 1:
        box = box.astype(np.float32).astype(np.float64)
    ref = oracle.solve_box_fft(box, 0.5)
    f = torch.from_numpy(S.box_to_blocks(box, blocks, B)).to(torch.float32 if single else torch.float64).cuda()
    phi = torch.full_like(f, float("nan"))
    L.lgf_poisson_solve(tables[B], L.Mesh([blocks], B, 0.5), ncomp, f.data_ptr(), phi.data_ptr(),
                        L.LGF_F32 if single else L.LGF_F64, L.make_opts(precision=precision, mac_mode=L.LGF_MAC_BOX))
    torch.cuda.synchronize()
    got = S.blocks_to_box(phi.double().cpu().numpy(), blocks, B, shape)
    for c in range(ncomp):
        assert np.linalg.norm(got[c] - ref[c]) <= 32 * U[precision] * np.linalg.norm(ref[c]), (B, nb, c)


TRIPLES = [(8, (1, 2, 3)), (8, (5, 4, 7)), (8, (9, 11, 6)), (8, (13, 8, 15)), (8, (14, 2, 10)), (8, (12, 4, 16)),
           (16, (2, 3, 5)), (16, (4, 7, 6)), (16, (1, 8, 12)), (16, (9, 2, 11)), (16, (1, 13, 15)), (16, (10, 2, 14)),
           (16, (1, 16, 3))]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("turn", [0, 1, 2])
@pytest.mark.parametrize("B,nb", TRIPLES)
def test_every_length_on_every_axis(L, tables, B, nb, turn, precision):
    """A complex and a real field (three components); FP32 on FP32 fields runs the line passes."""
    check(L, tables, B, nb[turn:] + nb[:turn], 3, precision, precision == 1)


@pytest.mark.parametrize("ncomp", [1, 2])
@pytest.mark.parametrize("B,nb", [(16, (9, 2, 10)), (16, (3, 11, 12)), (16, (13, 1, 4)), (16, (2, 14, 5)),
                                  (16, (6, 15, 1)), (16, (16, 7, 1)), (16, (1, 3, 16)), (16, (8, 1, 9)),
                                  (8, (2, 3, 4)), (8, (9, 5, 1)), (8, (6, 7, 10)), (8, (16, 1, 8))])
def test_fp32_on_fp64_fields(L, tables, B, nb, ncomp):
    """The block-index passes (csrc/box_pass.cuh, csrc/box_fft.cuh), real and complex fields."""
    check(L, tables, B, nb, ncomp, 1, False)
