"""Plans of new meshes built by one host thread and used by another on its own stream at once, and a captured refresh."""
import threading

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
    t = L.lgf_table_create(8, (10, 10, 10), L.LGF_TBL_BOX_ONLY)
    yield t
    L.lgf_table_destroy(t)


def new_meshes(L):
    out = []
    for shift in (3, 4, 5):  # shifted: not the plans of another test
        blocks = S.box_blocks((16, 24, 8 * shift), 8) + shift
        out.append((L.Mesh([blocks], 8, 0.5), len(blocks)))
        fine = np.array([(1, 1, 1), (2, 1, 1), (1, 2, 3)], np.int32) + 2 * shift
        out.append((L.Mesh([blocks, fine], 8, 0.5, n_ext=4), len(blocks) + len(fine)))
    return out


def test_solves_of_new_meshes_from_two_threads(L, table):
    meshes = new_meshes(L)
    f = [torch.randn(2, n, 8, 8, 8, dtype=torch.float64, device="cuda") for _, n in meshes]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = [[torch.zeros_like(v) for v in f] for _ in streams]
    torch.cuda.synchronize()
    start, failed = threading.Barrier(2), []

    def work(i):
        try:
            torch.cuda.set_device(0)
            start.wait()
            for (m, _), v, phi in zip(meshes, f, out[i]):
                L.lgf_poisson_solve(table, m, 2, v.data_ptr(), phi.data_ptr(), L.LGF_F64, L.make_opts(precision=2), None,
                                    streams[i].cuda_stream)
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for k, ((m, _), v) in enumerate(zip(meshes, f)):
        phi = torch.zeros_like(v)
        L.lgf_poisson_solve(table, m, 2, v.data_ptr(), phi.data_ptr(), L.LGF_F64, L.make_opts(precision=2))
        torch.cuda.synchronize()
        assert torch.isfinite(phi).all() and phi.abs().max() > 0
        assert torch.equal(out[0][k], phi) and torch.equal(out[1][k], phi)


def test_captured_refresh(L, table):
    """After one call on the stream a refresh can be captured; the replay reads the vorticity of the moment."""
    blocks = S.box_blocks((24, 16, 16), 8) - 2
    m = L.Mesh([blocks], 8, 0.5)
    om = torch.randn(3, len(blocks), 8, 8, 8, dtype=torch.float64, device="cuda")
    u, ref = torch.zeros_like(om), torch.zeros_like(om)
    opts, stream = L.make_opts(precision=2), torch.cuda.Stream()
    torch.cuda.synchronize()
    L.lgf_velocity_refresh(table, m, om.data_ptr(), u.data_ptr(), L.LGF_F64, opts, None, stream.cuda_stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        L.lgf_velocity_refresh(table, m, om.data_ptr(), u.data_ptr(), L.LGF_F64, opts, None, stream.cuda_stream)
    om.copy_(torch.randn_like(om))
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    L.lgf_velocity_refresh(table, m, om.data_ptr(), ref.data_ptr(), L.LGF_F64, opts)
    torch.cuda.synchronize()
    assert torch.isfinite(ref).all() and torch.equal(u, ref)
