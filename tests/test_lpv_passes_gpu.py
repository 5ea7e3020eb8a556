"""The passes of the load surrogate's loss, gradient and free run over the forms
they are built for: no, one and two scheduling variables; a state that ends
below or above column 8; one or two row groups per warp (more than 4,864
trajectories take two); chunks of 4 steps and work items of 16 and more.

Against a plain PyTorch FP64 evaluation of the same model (the loss by
autograd), with the tolerances of test_lpv_gpu.py: loss 1e-4 relative,
gradient and prediction 1e-3 of the largest entry.
"""
import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _model(rng, na, n_y, n_p, nu):
    nx = na * n_y
    W = np.zeros((1 + n_p, nx + n_y, nx + nu), dtype=np.float32)
    W[0, :nx, :nx] = rng.normal(0, 0.3 / np.sqrt(nx), (nx, nx)) + 0.5 * np.eye(nx)
    W[1:, :nx, :nx] = rng.normal(0, 0.02, (n_p, nx, nx))
    W[:, :nx, nx:] = rng.normal(0, 0.2, (1 + n_p, nx, nu))
    W[:, nx:, :nx] = rng.normal(0, 0.3, (1 + n_p, n_y, nx))
    scales = np.concatenate([rng.uniform(0.5, 2.0, nu + n_y), rng.normal(0, 0.2, n_p), rng.uniform(0.5, 2.0, n_p),
                             np.full(n_p, -5.0), np.full(n_p, 5.0)]).astype(np.float32)
    return W, scales


@pytest.mark.parametrize("na,n_y,n_p,nu,n,T", [(3, 4, 2, 3, 9, 33), (3, 4, 0, 3, 8, 4), (2, 3, 1, 3, 17, 65),
                                               (1, 3, 2, 2, 1, 1), (1, 7, 1, 4, 25, 3), (4, 3, 2, 3, 33, 18),
                                               (2, 3, 2, 3, 4870, 21), (3, 3, 1, 3, 4865, 6), (3, 4, 0, 2, 4999, 5)])
def test_passes_match_fp64(na, n_y, n_p, nu, n, T):
    torch = need_gpu()
    from paper_2604_12505_gb300 import lpv
    rng = np.random.default_rng(100 * na + 10 * n_y + n_p)
    nx, sigma2 = na * n_y, 1e-3
    W, sc = _model(rng, na, n_y, n_p, nu)
    u, y = rng.normal(size=(n, T, nu)).astype(np.float32), rng.normal(size=(n, T, n_y)).astype(np.float32)
    p = rng.uniform(-1, 1, (n, T, n_p)).astype(np.float32)
    m = lpv.Model(dict(n_x=nx, n_u=nu, n_y=n_y, n_p=n_p, na=na, sigma2=sigma2))
    m.set_params(W, sc)
    loss, g = m.loss_grad(u, y, p)
    yh = m.predict(u, p).cpu().numpy()
    m.close()

    Wt = torch.tensor(W, dtype=torch.float64, requires_grad=True)
    s = torch.tensor(sc, dtype=torch.float64)
    su, sy, pm, ps = s[:nu], s[nu:nu + n_y], s[nu + n_y:nu + n_y + n_p], s[nu + n_y + n_p:nu + n_y + 2 * n_p]
    ut, yt, pt = (torch.tensor(a, dtype=torch.float64) for a in (u, y, p))
    ut, pt = ut / su, (pt - pm) / ps
    x, out = torch.zeros((n, nx), dtype=torch.float64), []
    for k in range(T):
        z = torch.cat([x, ut[:, k]], 1)
        o = z @ Wt[0].T + sum(pt[:, k, i:i + 1] * (z @ Wt[1 + i].T) for i in range(n_p))
        x = o[:, :nx]
        out.append(o[:, nx:])
    yr = torch.stack(out, 1)
    ref = (yr - yt / sy).square().sum(2).mean() + 0.5 * sigma2 * Wt.square().sum()
    ref.backward()
    gr = Wt.grad.numpy().copy()
    gr[:, nx:, nx:] = 0.0
    ref, yr = float(ref.detach()), (yr.detach() * sy).numpy()
    assert abs(loss - ref) <= 1e-4 * ref
    assert np.abs(g - gr).max() <= 1e-3 * np.abs(gr).max()
    assert np.abs(yh - yr).max() <= 1e-3 * np.abs(yr).max()


@pytest.mark.parametrize("na,n_y,n_p,nu,B,T", [(3, 4, 2, 3, 1, 1), (3, 4, 2, 3, 19, 37), (2, 3, 1, 3, 8, 4), (1, 4, 0, 3, 5, 9),
                                               (2, 3, 2, 2, 4871, 6), (3, 4, 2, 3, 4866, 5), (4, 3, 0, 1, 33, 10)])
def test_closed_loop_matches_fp64(na, n_y, n_p, nu, B, T):
    torch = need_gpu()
    from paper_2604_12505_gb300 import lpv
    rng = np.random.default_rng(7 * B + T)
    nx = na * n_y
    W, sc = _model(rng, na, n_y, n_p, nu)
    body = dict(m=500.0, J=50.0, Ts=0.02, n_sub=10, ctrl_omega=0.2 * np.pi, ctrl_xi=0.7)
    F, tau = rng.uniform(-20, 20, (B, T, 2)), rng.uniform(-2, 2, (B, T))
    ref, fill = rng.uniform(-0.3, 0.3, (B, T)), rng.uniform(0.2, 0.8, B)
    F[0, 0] = 0.0, -0.0
    ref[:, T // 2] = 1e-42  # not a normal FP32 number
    m = lpv.Model(dict(n_x=nx, n_u=nu, n_y=n_y, n_p=n_p, na=na))
    m.set_params(W, sc)
    out = m.simulate(F, tau, ref, fill, body).cpu().numpy()
    m.close()

    Wd, s = W.astype(np.float64), sc.astype(np.float64)
    su, sy, pm, ps = s[:nu], s[nu:nu + n_y], s[nu + n_y:nu + n_y + n_p], s[nu + n_y + n_p:nu + n_y + 2 * n_p]
    x, q, v = np.zeros((B, nx)), np.zeros((B, 3)), np.zeros((B, 3))
    mass, w, want = np.array([500.0, 500.0, 50.0]), 0.2 * np.pi, np.zeros((B, T, 6))
    for k in range(T):
        want[:, k] = np.concatenate([q, v], 1)
        u = np.concatenate([F[:, k], (tau[:, k] + 50.0 * w * w * (ref[:, k] - q[:, 2]) - 1.4 * 50.0 * w * v[:, 2])[:, None]], 1)
        p = (np.clip(np.stack([fill, v[:, 2]], 1)[:, :n_p], -5.0, 5.0) - pm) / ps
        z = np.concatenate([x, u[:, :nu] / su], 1)
        o = z @ Wd[0].T + sum(p[:, i:i + 1] * (z @ Wd[1 + i].T) for i in range(n_p))
        x = o[:, :nx]
        a = (u + o[:, nx:nx + 3] * sy[:3]) / mass
        for _ in range(10):
            v = v + 0.002 * a
            q = q + 0.002 * v
    for blk in (slice(0, 3), slice(3, 6)):
        assert np.abs(out[:, :, blk] - want[:, :, blk]).max() <= 1e-3 * max(np.abs(want[:, :, blk]).max(), 1e-300)


@pytest.mark.parametrize("na,n_y,n_p", [(1, 3, 0), (2, 3, 1), (3, 4, 2)])
def test_closed_loop_is_the_same_in_either_row_split(na, n_y, n_p):
    """A warp carries 8 runs while they are few and 16 beyond: equal bit for bit."""
    torch = need_gpu()
    from paper_2604_12505_gb300 import lpv
    rng = np.random.default_rng(na)
    W, sc = _model(rng, na, n_y, n_p, 3)
    B, few, T = 5000, 45, 30
    body = dict(m=500.0, J=50.0, Ts=0.02, n_sub=10, ctrl_omega=0.2 * np.pi, ctrl_xi=0.7)
    F, tau = rng.uniform(-20, 20, (B, T, 2)), rng.uniform(-2, 2, (B, T))
    ref, fill = rng.uniform(-0.3, 0.3, (B, T)), rng.uniform(0.2, 0.8, B)
    m = lpv.Model(dict(n_x=na * n_y, n_u=3, n_y=n_y, n_p=n_p, na=na))
    m.set_params(W, sc)
    many = m.simulate(F, tau, ref, fill, body)[:few].cpu().numpy()
    alone = m.simulate(F[:few], tau[:few], ref[:few], fill[:few], body).cpu().numpy()
    m.close()
    np.testing.assert_array_equal(many, alone)
