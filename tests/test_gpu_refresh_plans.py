"""The velocity refresh's kept plans under several host threads and streams, without synchronisations between the calls."""
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


def test_new_plans_from_two_threads(L):
    """Two threads refresh the same new meshes on a stream each: whichever builds a mesh's plan, both get the values
    that a call after a synchronisation gives."""
    rng = np.random.default_rng(41)
    cases = []
    for k, shape in enumerate(((16, 24, 8), (24, 8, 16), (8, 8, 32), (16, 16, 24))):
        blocks = S.box_blocks(shape, 8)[::-1 if k % 2 else 1]
        om = torch.from_numpy(rng.standard_normal((3, len(blocks), 8, 8, 8))).cuda()
        cases.append((L.Mesh([blocks], 8, 0.5), om))
    table = L.lgf_table_create(8, (6, 6, 6), L.LGF_TBL_BOX_ONLY)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = [[torch.full_like(om, float("nan")) for _, om in cases] for _ in streams]
    torch.cuda.synchronize()
    start, failed = threading.Barrier(2), []

    def work(i):
        try:
            torch.cuda.set_device(0)
            start.wait()
            for (m, om), u in zip(cases, out[i]):
                L.lgf_velocity_refresh(table, m, om.data_ptr(), u.data_ptr(), L.LGF_F64, L.make_opts(precision=2), None,
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
    try:
        for k, (m, om) in enumerate(cases):
            u = torch.full_like(om, float("nan"))
            L.lgf_velocity_refresh(table, m, om.data_ptr(), u.data_ptr(), L.LGF_F64, L.make_opts(precision=2))
            torch.cuda.synchronize()
            assert torch.isfinite(u).all()
            assert torch.equal(out[0][k], u) and torch.equal(out[1][k], u)
    finally:
        L.lgf_table_destroy(table)
