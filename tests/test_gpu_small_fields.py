"""Double-float solves of small fields: scaling the source by a power of two scales the result, as long as the low part of
the source itself stays a float.

Tolerance as in test_gpu_line_axes: 32 u in the relative 2-norm, u = 2^-48."""
import numpy as np
import pytest

import lgf_synth as S
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2010_13213_gb300.lgf as L
    L.load()
    return L


@pytest.mark.parametrize("e", [-96, -60, 0, 60])
@pytest.mark.parametrize("B,nb,ncomp", [(16, (3, 4, 2), 1), (16, (6, 5, 7), 2), (8, (3, 2, 4), 3)])
def test_scaled_sources(L, B, nb, ncomp, e):
    shape = tuple(B * n for n in nb[::-1])
    blocks = S.box_blocks(shape, B)
    box = S.random_box(shape, sum(nb), ncomp)
    ref = oracle.solve_box_fft(box, 0.5)
    f = torch.from_numpy(S.box_to_blocks(box, blocks, B) * 2.0 ** e).cuda()
    phi = torch.full_like(f, float("nan"))
    table = L.lgf_table_create(B, (7, 7, 7), L.LGF_TBL_BOX_ONLY)
    try:
        L.lgf_poisson_solve(table, L.Mesh([blocks], B, 0.5), ncomp, f.data_ptr(), phi.data_ptr(), L.LGF_F64,
                            L.make_opts(precision=L.LGF_PREC_DF32, mac_mode=L.LGF_MAC_BOX))
        torch.cuda.synchronize()
    finally:
        L.lgf_table_destroy(table)
    got = S.blocks_to_box(phi.cpu().numpy() * 2.0 ** -e, blocks, B, shape)
    for c in range(ncomp):
        assert np.linalg.norm(got[c] - ref[c]) <= 32 * 2.0 ** -48 * np.linalg.norm(ref[c])
