"""Device memory of the load surrogate's loss and gradient: at most a row of 16
floats per sample (state and residuals), whatever the number of trajectories."""
import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,T", [(1, 300000), (9, 50000), (17, 20000), (4870, 100)])
def test_workspace_is_a_row_per_sample(n, T):
    torch = need_gpu()
    from paper_2604_12505_gb300.lpv import Model
    m = Model(dict(n_p=2))
    Wt = np.zeros(m.shape_W)
    Wt[0, :12, :12] = 0.5 * np.eye(12)
    Wt[0, :12, 12:] = Wt[0, 12:, :12].T[:, :3] = 0.1
    m.set_params(Wt, np.concatenate([np.ones(7), np.zeros(2), np.ones(2), [-9.0] * 2, [9.0] * 2]).astype(np.float32))
    u, y, p = (torch.randn(n, T, c, device="cuda") for c in (3, 4, 2))
    m.loss_grad(u[:, :4].contiguous(), y[:, :4].contiguous(), p[:, :4].contiguous())
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    loss, g = m.loss_grad(u, y, p)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    m.close()
    assert np.isfinite(loss) and np.isfinite(g).all()
    assert used <= 64 * n * T + (8 << 20)
