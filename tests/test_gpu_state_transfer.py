"""w5ct_set_state / w5ct_get_state: the one-launch device path against the
copies (host buffers, and device addresses a kernel may not touch), over odd
sizes, patches at odd offsets, NULL outputs and both arithmetic types."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_04278_gb300 import inputs, w5ct
    return torch, inputs, w5ct


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shapes", [[(7, 5, 3)], [(33, 9, 10)], [(7, 5, 3), (1, 1, 1), (16, 17, 9)]])
def test_device_path_equals_copies(env, precision, shapes):
    torch, I, w5 = env
    dxs = [tuple(1.0 / n for n in sh) for sh in shapes]
    cfg = w5.make_config(precision=precision)
    made = [w5.Batch(shapes, dxs, cfg) for _ in range(3)]
    states = [I.random_smooth_state(sh, seed=40 + p) if min(sh) > 1 else I.uniform_state(sh, B=(0.3, 0.2, 0.1))
              for p, sh in enumerate(shapes)]
    n = [sh[0] * sh[1] * sh[2] for sh in shapes]
    for p, (c, f) in enumerate(states):
        made[0].set_state(p, c, f)                                                   # host copies
        made[1].set_state(p, torch.from_numpy(c).cuda(), torch.from_numpy(f).cuda())   # one launch
        raw = torch.zeros(64 * n[p] + 8, dtype=torch.uint8, device="cuda")             # 4-byte aligned: copies
        raw[4:4 + 40 * n[p]] = torch.from_numpy(c.reshape(-1).view(np.uint8)).cuda()
        raw[4 + 40 * n[p]:4 + 64 * n[p]] = torch.from_numpy(f.reshape(-1).view(np.uint8)).cuda()
        torch.cuda.synchronize()
        w5.w5ct_set_state(made[2].ctx, raw.data_ptr() + 4, raw.data_ptr() + 4 + 40 * n[p], 1, patch=p)
        torch.cuda.synchronize()
    for b in made:
        b.step(1e-3)
    for p, sh in enumerate(shapes):
        want = made[0].get_state(p)
        for b in made[1:]:
            for x, y in zip(want, b.get_state(p)):
                assert np.array_equal(x, y)
            q = torch.full((5 * n[p],), 7.0, dtype=torch.float64, device="cuda")
            f = torch.full((3 * n[p],), 7.0, dtype=torch.float64, device="cuda")
            w5.w5ct_get_state(b.ctx, q, None, None, 1, patch=p)
            w5.w5ct_get_state(b.ctx, None, f, None, 1, patch=p)
            assert np.array_equal(q.cpu().numpy().reshape(want[0].shape), want[0])
            assert np.array_equal(f.cpu().numpy().reshape(want[1].shape), want[1])
            raw = torch.zeros(40 * n[p] + 8, dtype=torch.uint8, device="cuda")
            w5.w5ct_get_state(b.ctx, raw.data_ptr() + 4, None, None, 1, patch=p)
            assert np.array_equal(raw[4:4 + 40 * n[p]].cpu().numpy().view(np.float64).reshape(want[0].shape), want[0])
    for b in made:
        b.close()


def test_device_path_reports_a_nonphysical_state(env):
    torch, I, w5 = env
    c, f = I.random_smooth_state((8, 8, 8), seed=1)
    c[4, 2, 3, 4] = -1.0
    s = w5.Solver((8, 8, 8), 1.0 / 8, w5.make_config())
    s.set_state(torch.from_numpy(c).cuda(), torch.from_numpy(f).cuda())
    s.step(1e-4)
    q = torch.empty(c.shape, dtype=torch.float64, device="cuda")
    with pytest.raises(w5.W5ctError) as e:
        w5.w5ct_get_state(s.ctx, q, None, None, 1)
    assert e.value.code == w5.W5CT_ERR_NONPHYSICAL
    c, f = I.random_smooth_state((8, 8, 8), seed=1)
    s.set_state(torch.from_numpy(c).cuda(), torch.from_numpy(f).cuda())
    w5.w5ct_get_state(s.ctx, q, None, None, 1)
    assert np.array_equal(q.cpu().numpy(), c)
    s.close()
