"""The adjoint's tiles of segments on thin, narrow and odd grids: the gradient
of a cyclically relabelled state (x, y, z -> y, z, x) is the relabelled gradient,
so each tile form (segments along x; 8, 16 or 32 pencils side by side along y and
z) is held against the other two at the same sizes.  WENO5.  Bounds: the frames
are cyclic, so faces see the same numbers, and only the order of three-axis
sums differs: 1e-11 of a component's largest value in double (a few hundred
roundings through four stages), 1e-4 in float."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(1, 24, 20), (40, 9, 3), (70, 1, 1), (130, 2, 5), (17, 33, 1), (33, 12, 18), (3, 5, 270), (64, 16, 8)]


def gradient(shape, prec, cons, b, lq, lb):
    import torch
    from paper_1812_04278_gb300 import w5ct
    s = w5ct.Solver(shape, tuple(0.02 for _ in shape), w5ct.make_config(precision=prec, weno_variant=w5ct.W5CT_WENO_JS))
    s.set_state(cons, b)
    x, y = torch.from_numpy(lq).cuda(), torch.from_numpy(lb).cuda()
    gq, gb = torch.empty_like(x), torch.empty_like(y)
    w5ct.w5ct_adjoint_step(s.ctx, 2e-3, x, y, gq, gb)
    s.close()
    return gq.cpu().numpy(), gb.cpu().numpy()


def relabel(a):
    """planes (rho, m, E) or (b) in the axes (y, z, x)"""
    c = [0, 2, 3, 1, 4] if len(a) == 5 else [1, 2, 0]
    return np.ascontiguousarray(a[c].transpose(0, 3, 1, 2))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision, tol", [(0, 1e-11), (1, 1e-4)])
def test_relabelled_gradients(shape, precision, tol):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_04278_gb300 import inputs as I
    cons, b = I.random_smooth_state(shape, seed=21)
    rng = np.random.default_rng(1)
    args = [cons, b, rng.standard_normal(cons.shape), rng.standard_normal(b.shape)]
    want = gradient(shape, precision, *args)
    for _ in range(2):
        shape = (shape[1], shape[2], shape[0])
        args = [relabel(a) for a in args]
        want = [relabel(a) for a in want]
        for x, y in zip(gradient(shape, precision, *args), want):
            for f in range(len(x)):
                assert np.abs(x[f] - y[f]).max() <= tol * np.abs(y[f]).max()
