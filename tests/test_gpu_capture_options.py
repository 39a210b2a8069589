"""A mesh prepared with one set of options may be captured with another: the tables and the scratch of a box shape do not
depend on the evaluation that was asked for first."""
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


def single(L):
    blocks = S.box_blocks((48, 32, 80), 16)
    return L.Mesh([blocks], 16, 0.5), len(blocks)


def composite(L):
    coarse = S.box_blocks((32, 32, 48), 16)
    fine = np.array([(2, 1, 1), (3, 1, 1), (2, 2, 2)], np.int32)
    return L.Mesh([coarse, fine], 16, 0.5, n_ext=8), len(coarse) + len(fine)


@pytest.mark.parametrize("make", [single, composite])
@pytest.mark.parametrize("precision,slices", [(2, 0), (2, 5), (1, 0), (1, 2)])
def test_capture_after_preparing_with_other_options(L, make, precision, slices):
    mesh, n = make(L)
    f = torch.randn(3, n, 16, 16, 16, dtype=torch.float64, device="cuda")
    captured, eager = torch.zeros_like(f), torch.zeros_like(f)
    table = L.lgf_table_create(16, (12, 12, 12), L.LGF_TBL_BOX_ONLY)
    try:
        stream = torch.cuda.Stream()
        L.lgf_table_prepare(table, mesh, 3, L.LGF_F64, L.make_opts(precision=0), stream.cuda_stream)
        opts = L.make_opts(precision=precision, dft_slices=slices)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        failed = None
        with torch.cuda.graph(graph, stream=stream):
            try:
                L.lgf_poisson_solve(table, mesh, 3, f.data_ptr(), captured.data_ptr(), L.LGF_F64, opts, None,
                                    stream.cuda_stream)
            except L.LgfError as e:
                failed = e
        assert failed is None, failed
        graph.replay()
        torch.cuda.synchronize()
        L.lgf_poisson_solve(table, mesh, 3, f.data_ptr(), eager.data_ptr(), L.LGF_F64, opts, None, stream.cuda_stream)
        torch.cuda.synchronize()
        assert torch.isfinite(eager).all() and torch.equal(captured, eager)
    finally:
        L.lgf_table_destroy(table)
