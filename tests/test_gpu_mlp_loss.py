"""GPU: the network's loss where the number of pass blocks and their fill change.

A pass block adds the terms of 8 samples (16 from 2432, 32 from 4864), the last
one padded, and one block of 256 threads adds the blocks' sums: one sample, both
sides of a full block, of each change of block size and of 256 blocks.  Bar as for
the gradient's test at one size: FP32 outputs, 1e-5 of the loss; a lost or doubled
sample changes it by 1/n >= 1.2e-4.
"""
import numpy as np
import pytest

from oracle import learned as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 8, 9, 2049, 2431, 2432, 2433, 4863, 4864, 4865, 8193])
def test_loss_at_kernel_edges(n):
    import torch

    from paper_1702_04910_gb300.binding import Mlp
    rng = np.random.default_rng(n)
    P = rng.normal(0.0, 0.08, L.N_PARAMS).astype(np.float32)
    X = rng.normal(0.0, 1.0, (n, L.N_IN)).astype(np.float32)
    T = rng.normal(0.0, 0.5, (n, L.N_OUT)).astype(np.float32)
    norm = np.concatenate([rng.normal(0.0, 0.1, 512), rng.uniform(0.5, 2.0, 512),
                           rng.uniform(0.5, 2.0, 6)]).astype(np.float32)
    m = Mlp()
    m.set_params(P)
    m.set_normalization(norm)
    x, t = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    _, loss = m.gradient(x.data_ptr(), t.data_ptr(), n)
    assert loss == pytest.approx(L.loss(P.astype(np.float64), norm.astype(np.float64), X, T), rel=1e-5)
    m.close()
