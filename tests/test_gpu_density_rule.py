"""The interior density's split polar rule on the GPU: the kernels of N_p <= 8
(moments of each azimuth line) against the kernel of N_p >= 9 (every node's
Zernike vector), which evaluates the same rule node by node and whose leading
coefficients are those of the smaller bases."""
import numpy as np
import pytest

from gpu_helpers import need_gpu
from paper_1608_04607_gb300.inputs import kuhn_cube_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    need_gpu()
    from paper_1608_04607_gb300 import dfm

    dfm.load()
    return dfm


# few tets (a warp per face) and many (sixteen lanes per face); even, odd, the
# smallest and the largest number of points; no, weak, strong damping
@pytest.mark.parametrize("n,nq", [(2, -24), (2, -3), (2, -2), (2, -64), (5, -24), (5, -7)])
@pytest.mark.parametrize("mu", [0.0, 0.3, 60.0, "tet"])
def test_line_moments_match_the_node_by_node_rule(D, n, nq, mu):
    """FP64 sums of at most 6 x 64^2 terms with coefficients that sum to 8.5:
    1e-12 of the largest entry leaves a factor of several over n_terms * eps."""
    import torch

    m = kuhn_cube_mesh(n, jitter=0.2, seed=9)
    mesh = D.Mesh(m.verts, m.tets, refl=1.0)
    rng = np.random.default_rng(3)
    tets = rng.integers(0, m.n_tets, size=m.n_tets + 3)  # some twice, an odd count
    w = rng.uniform(-1, 1, size=tets.size)
    if mu == "tet":
        mu = torch.from_numpy(rng.uniform(0, 5, size=m.n_tets)).cuda()
    ref = [v.reshape(m.n_rows, -1) for v in D.interior_density(mesh, 9, tets, weights=w, mu=mu, nq=nq)]
    for Np in range(9):
        nb = D.nbasis(Np)
        for got, want in zip(D.interior_density(mesh, Np, tets, weights=w, mu=mu, nq=nq), ref):
            want = want[:, :nb]
            assert float((got - want).abs().max()) <= 1e-12 * float(want.abs().max())
