"""The integrating-factor passes of both block sizes at every radius where their tiles change (no taps, fewer than one
window of eight, exactly one, two windows, the block edge, beyond it) against the oracle, with scratch that holds NaN
from an earlier call.

Tolerance of the relative 2-norm against the input: three passes of 2 r + 1 weighted sums and the interpolation, weights
of sum one.  A pass's partial sums stay below the largest input, so that its 2 r + 1 <= 41 roundings of independent sign
come to about sqrt(41) u / 2; three passes and the products' own roundings stay below 16 u, u = 2^-53, 2^-24 and, for
double-float, 2^-48."""
import numpy as np
import pytest

import lgf_synth as S
from oracle import amr, core

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


def meshes(B):
    coarse = S.box_blocks((2 * B, 2 * B, 2 * B), B)
    fine = np.array([(1, 1, 1), (2, 1, 1), (1, 2, 2), (3, 3, 2)], np.int32)  # not a box, not a union of coarse blocks
    large = [S.box_blocks((4 * B, 3 * B, 4 * B), B), S.box_blocks((3 * B, 4 * B, 3 * B), B) + 2]
    return [coarse, fine], large


def apply(L, levels, B, f, alpha, precision):
    m = L.Mesh(levels, B, 1.0, n_ext=4)
    g = torch.full_like(f, float("nan"))
    L.lgf_heat_apply(0, m, f.shape[0], f.data_ptr(), g.data_ptr(), L.LGF_F64, alpha, L.make_opts(precision=precision),
                     None, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return g


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("B", [8, 16])
@pytest.mark.parametrize("r,alpha", [(0, 0.0), (3, 1e-5), (7, 0.015), (8, 0.03), (9, 0.06), (10, 0.1), (16, 0.6),
                                     (17, 0.75)])
def test_every_radius(L, B, r, alpha, precision):
    assert len(core.heat_weights_1d(alpha)) - 1 == r
    levels, large = meshes(B)
    rng = np.random.default_rng(r + B)
    f = [rng.standard_normal((2, len(b), B, B, B)) for b in levels]
    if precision == 1:
        f = [v.astype(np.float32).astype(np.float64) for v in f]
    ft = torch.from_numpy(np.concatenate(f, axis=1)).cuda()
    nan = torch.full((2, sum(len(b) for b in large), B, B, B), float("nan"), dtype=torch.float64, device="cuda")
    apply(L, large, B, nan, alpha, precision)
    got = apply(L, levels, B, ft, alpha, precision).cpu().numpy()
    # the oracle's dense boxes reach n_ext + 8 cells beyond the blocks: they have to hold the kernel
    ref = np.concatenate(amr.fif_amr(dict(B=B, h0=1.0, n_ext=16, levels=levels), f, alpha), axis=1)
    on = np.isfinite(got)  # Omega_k: the cells that no finer block covers
    assert on[:, len(levels[0]):].all() and (ref[~on] == 0.0).all()
    fine = sum(len(b) for b in levels[1:]) * B ** 3
    assert on.sum() == 2 * (len(levels[0]) * B ** 3 - fine // 8 + fine)
    scale = np.linalg.norm(np.concatenate(f, axis=1))
    assert np.linalg.norm(got[on] - ref[on]) <= 16 * U[precision] * scale


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("B", [8, 16])
def test_projection_does_not_read_old_scratch(L, B, precision):
    """The same bits before and after a call whose fields are all NaN."""
    levels, large = meshes(B)
    table = L.lgf_table_create(B, (8, 8, 8), L.LGF_TBL_BOX_ONLY)
    try:
        rng = np.random.default_rng(B)
        r = torch.from_numpy(rng.standard_normal((3, sum(len(b) for b in levels), B, B, B))).cuda()
        nan = torch.full((3, sum(len(b) for b in large), B, B, B), float("nan"), dtype=torch.float64, device="cuda")
        out = []
        for lv, v in ((levels, r), (large, nan), (levels, r)):
            u, p = torch.zeros_like(v), torch.zeros_like(v[:1])
            L.lgf_stage_projection(table, L.Mesh(lv, B, 1.0, n_ext=4), v.data_ptr(), u.data_ptr(), p.data_ptr(),
                                   L.LGF_F64, 0.05, L.make_opts(precision=precision))
            torch.cuda.synchronize()
            out.append((u.cpu(), p.cpu()))
        assert torch.isfinite(out[0][0]).all() and torch.isfinite(out[0][1]).all()
        assert torch.equal(out[0][0], out[2][0]) and torch.equal(out[0][1], out[2][1])
    finally:
        L.lgf_table_destroy(table)
