"""The passes of the velocity-level surrogate's loss and gradient at the edges
of their chunks (32 samples of the state pass, 16 or 8 of the adjoint's, 64
and 128 of the sample and outer-product blocks), and over several windows of
the time axis (many trajectories), against the FP64 oracle.

Tolerances as in test_slpv_gpu.py: loss 1e-4 relative, gradient 1e-3 of the
largest entry.  The loss alone takes its sums in other parts: FP64 sums of the
same terms, 1e-12 relative.
"""
import numpy as np
import pytest

from oracle import slpv as S
from tests.gpu_util import need_gpu
from tests.test_slpv_gpu import _data, _theta

pytestmark = pytest.mark.gpu
SC = np.array([20.0, 20.0, 2.0, 0.1, 0.1, 0.05], dtype=np.float32)


# copies: the distinct trajectories repeated so often that the time axis is
# cut into windows (the mean over them does not change)
@pytest.mark.parametrize("nx,n,T,copies", [(2, 1, 1, 1), (2, 9, 32, 1), (4, 9, 33, 1), (4, 17, 127, 1), (6, 5, 64, 1),
                                           (6, 4, 9, 1), (8, 3, 31, 1), (8, 33, 8, 1), (4, 7, 40, 5000),
                                           (8, 5, 50, 2000),
                                           # the adjoint in segments: 4, 5 and 10 of a ragged
                                           # length, and of each of two windows
                                           (2, 2, 257, 1), (4, 9, 321, 1), (6, 3, 650, 1), (8, 2, 333, 1),
                                           (4, 2, 2500, 150)])
def test_passes_match_oracle(nx, n, T, copies):
    torch = need_gpu()
    from paper_2604_12505_gb300.slpv import VelocityModel
    th64, th32 = _theta(nx, 11 + nx)
    u, y = _data(n, T, 17 * n + T, SC)
    U = [u[i].astype(np.float64) / SC[:3] for i in range(n)]
    Y = [y[i].astype(np.float64) / SC[3:] for i in range(n)]
    sigma2 = 1e-3
    ref_l = S.loss(th64, U, Y, nx, sigma2)
    ref_g = S.loss_grad(th64, U, Y, nx, sigma2, S.d_mask(nx, 3, 3))
    m = VelocityModel(nx=nx, sigma2=sigma2)
    m.set_params(th32, SC)
    ud, yd = (torch.tensor(a, device="cuda").repeat(copies, 1, 1) for a in (u, y))
    loss, g = m.loss_grad(ud, yd)
    alone, _ = m.loss_grad(ud, yd, grad=False)
    loss, g = float(loss.item()), g.cpu().numpy()
    assert abs(loss - ref_l) <= 1e-4 * ref_l
    assert np.abs(g - ref_g).max() <= 1e-3 * np.abs(ref_g).max()
    assert abs(float(alone.item()) - loss) <= 1e-12 * loss
    m.close()


@pytest.mark.parametrize("nx,B,T", [(2, 1, 1), (4, 33, 5), (4, 64, 8), (6, 31, 7), (8, 40, 3)])
def test_closed_loop_matches_oracle_at_edge_sizes(nx, B, T):
    torch = need_gpu()
    from paper_2604_12505_gb300.slpv import VelocityModel
    th64, th32 = _theta(nx, 21, m1=0.2)
    rng = np.random.default_rng(B + T)
    F, tau, ref = rng.uniform(-20, 20, (B, T, 2)), rng.uniform(-2, 2, (B, T)), rng.uniform(-0.3, 0.3, (B, T))
    pd = dict(J=133.84, omega=0.2 * np.pi, xi=0.7)
    m = VelocityModel(nx=nx)
    m.set_params(th32, SC)
    # the second time from buffers that are 8-byte but not 16-byte aligned
    odd = torch.empty(2 * B * T + 1, dtype=torch.float64, device="cuda")[1:].view(B, T, 2)
    odd.copy_(torch.tensor(F))
    for f in (F, odd):
        out = m.simulate(f, tau, ref, 0.05, pd["J"], pd["omega"], pd["xi"]).cpu().numpy()
        want = np.stack([S.closed_loop(th64, nx, dict(u=SC[:3].astype(np.float64), y=SC[3:].astype(np.float64)), F[b],
                                       tau[b], ref[b], 0.05, pd) for b in range(B)])
        for blk in (slice(0, 3), slice(3, 6)):
            assert np.abs(out[:, :, blk] - want[:, :, blk]).max() <= 1e-3 * np.abs(want[:, :, blk]).max() + 1e-12
    m.close()


@pytest.mark.parametrize("nx,T", [(2, 9), (4, 8), (6, 3), (8, 21)])
def test_closed_loop_is_the_same_among_few_and_many_runs(nx, T):
    torch = need_gpu()
    from paper_2604_12505_gb300.slpv import VelocityModel
    _, th32 = _theta(nx, 21, m1=0.2)
    rng = np.random.default_rng(nx + T)
    B, few = 19500, 45
    F, tau, ref = (torch.tensor(a, device="cuda") for a in (rng.uniform(-20, 20, (B, T, 2)), rng.uniform(-2, 2, (B, T)),
                                                            rng.uniform(-0.3, 0.3, (B, T))))
    m = VelocityModel(nx=nx)
    m.set_params(th32, SC)
    many = m.simulate(F, tau, ref, 0.05, 133.84, 0.2 * np.pi, 0.7)[:few].cpu().numpy()
    alone = m.simulate(F[:few].contiguous(), tau[:few].contiguous(), ref[:few].contiguous(), 0.05, 133.84,
                       0.2 * np.pi, 0.7).cpu().numpy()
    m.close()
    np.testing.assert_array_equal(many, alone)
