"""GPU: the network's gradient at the sizes where its kernels change shape.

One sample, the edges of a gradient chunk (128 samples) and of the samples a
pass block takes (8, 16 from 2432 samples, 32 from 4864), against the FP64
oracle.  Bar: a gradient entry is a sum of n products in order, so its error is
at most n 2^-24 of the sum of their magnitudes and, the roundings being
independent, about sqrt(n) 2^-24 = 4e-6 at the largest n; 1e-4 of a layer's
largest entry is the bar of the existing gradient test.
"""
import numpy as np
import pytest

from oracle import learned as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 8, 9, 127, 128, 129, 2431, 2433, 4865])
def test_gradient_at_kernel_edges(n):
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
    g, loss = m.gradient(x.data_ptr(), t.data_ptr(), n)
    ref = L.gradient(P.astype(np.float64), norm.astype(np.float64), X, T)
    at = 0
    for size in (512 * 64, 64, 64 * 64, 64, 64 * 6, 6):
        a, b = g[at:at + size], ref[at:at + size]
        assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b))
        at += size
    assert np.isfinite(loss) and loss > 0.0
    m.close()
