"""FP32 operators applied to FP32 right-hand sides (tensor cores, both
operands split into TF32 parts) against the FP64-vector application of the same
blocks, which runs other kernels (compensated sums)."""
import numpy as np
import pytest

from gpu_helpers import need_gpu
from paper_1608_04607_gb300.inputs import kuhn_cube_mesh

pytestmark = pytest.mark.gpu

# worst case of a row: 22-bit products, sum |B||x| at most a few times max |y|
# for random x over up to 3 x 45 terms; typical errors are 50 times smaller
TOL = 3e-6


@pytest.fixture(scope="module")
def D():
    need_gpu()
    from paper_1608_04607_gb300 import dfm

    dfm.load()
    return dfm


def vectors(op, R, seed, scale=1.0):
    import torch

    g = torch.Generator(device="cuda").manual_seed(seed)
    return scale * torch.randn((R, op.n_rows, op.nb), generator=g, device="cuda")


def close(y, ref):
    # right-hand sides apart: one of tiny entries is held to its own size
    err = (y.double() - ref).abs().amax((1, 2)) / ref.abs().amax((1, 2))
    assert float(err.max()) <= TOL


# padded and unpadded bases, one and two column tiles with remainders, several
# passes, one tet group per block and more, walls on most faces (n = 1)
@pytest.mark.parametrize("Np", range(1, 9))
@pytest.mark.parametrize("n,R", [(1, 2), (3, 1), (3, 7), (3, 8), (3, 9), (2, 16), (2, 19), (6, 3)])
def test_several_right_hand_sides(D, Np, n, R):
    m = kuhn_cube_mesh(n, jitter=0.2 if n > 1 else 0.0, seed=8)
    op = D.Operator(D.Mesh(m.verts, m.tets, refl=0.9), Np, mu=0.1)
    x, x0 = vectors(op, R, 1), vectors(op, R, 2)
    x[R // 2] *= 1e-20  # each right-hand side keeps its own scale
    x0[R // 2] *= 1e-20
    close(op.apply(x), op.apply(x.double()))
    close(op.apply(x, x0=x0, alpha=-0.7), op.apply(x.double(), x0=x0.double(), alpha=-0.7))
    close(op.apply(x, x0=x, alpha=-1.0), op.apply(x.double(), x0=x.double(), alpha=-1.0))
    op.check_error()


@pytest.mark.parametrize("Np,K,R", [(1, 4, 9), (2, 3, 4), (3, 2, 5), (4, 3, 16), (4, 3, 17), (5, 4, 3), (6, 3, 8), (6, 4, 16), (8, 2, 4),
                                    (8, 3, 4)])
def test_combined_operators(D, Np, K, R):
    m = kuhn_cube_mesh(3, jitter=0.2, seed=8)
    mesh = D.Mesh(m.verts, m.tets, refl=0.9)
    ops = [D.Operator(mesh, Np, mu=0.1, moment=k) for k in range(K)]
    coef = np.random.default_rng(0).uniform(-1, 1, size=(R, K))
    x, x0 = vectors(ops[0], R, 3), vectors(ops[0], R, 4)
    ref = x0.double() + 0.5 * sum(coef_k[:, None, None] * o.apply(x.double())
                                  for coef_k, o in zip(__import__("torch").from_numpy(coef.T).cuda(), ops))
    close(D.apply_combo(ops, coef, x, x0=x0, alpha=0.5), ref)


def test_interface_reflections_accumulate_in_place(D):
    """The reflected part is applied with x0 = y, in place."""
    m = kuhn_cube_mesh(2, jitter=0.2, seed=8)
    rho = np.where(np.arange(m.n_tets) % 2, 1.0, 3.0)
    op = D.Operator(D.Mesh(m.verts, m.tets, refl=0.9), 4, mu=0.1, rho_f=rho)
    x = vectors(op, 5, 5)
    close(op.apply(x, x0=x), op.apply(x.double(), x0=x.double()))
