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


@pytest.mark.parametrize("Np,R,K", [(1, 8, 1), (2, 6, 1), (3, 5, 1), (4, 3, 1), (5, 1, 1), (6, 9, 1), (7, 2, 1), (8, 1, 1), (8, 16, 1),
                                    (2, 3, 2), (4, 2, 3), (8, 2, 2)])
def test_applications_have_no_common_loss(D, Np, R, K):
    """Results smaller by a common factor would be magnified by an iteration at
    little damping.  A nearly isotropic positive density, and one positive in all its
    coefficients: the mean relative error is at most the expected loss of one
    truncation towards zero, 2^-24 x 0.72 = 4.3e-8 (the mean of 1 / mantissa being
    0.72), and the mean of at least 3,888 results' own roundings, below 3e-9."""
    import torch

    m = kuhn_cube_mesh(6, jitter=0.2, seed=4)
    mesh = D.Mesh(m.verts, m.tets, refl=1.0)
    ops = [D.Operator(mesh, Np, mu=0.05, moment=k) for k in range(K)]
    coef = np.tile([1.0, -0.02, 0.01][:K], (R, 1))
    for spread in (0.05, 1.0):
        x = spread * vectors(ops[0], R, 7).abs()
        x[..., 0] = 1.0 + 0.2 * vectors(ops[0], R, 8)[..., 0].abs()
        if K == 1:
            y, ref = ops[0].apply(x), ops[0].apply(x.double())
        else:
            y = D.apply_combo(ops, coef, x)
            ref = sum(float(c) * o.apply(x.double()) for c, o in zip(coef[0].astype(np.float32), ops))
        d = y.double() - ref
        for part in (slice(0, 1), slice(None)):  # the isotropic coefficients, and all
            loss = float((d[..., part] * ref[..., part].sign()).sum() / ref[..., part].abs().sum())
            assert abs(loss) <= 4.6e-8, (spread, part, loss)


def test_coefficients_that_are_not_finite(D):
    """Infinities, NaN and numbers next to the largest one give what the same
    vectors give alone (N_b = 15: FP32 multiplications and additions)."""
    import torch

    m = kuhn_cube_mesh(3, jitter=0.2, seed=8)
    op = D.Operator(D.Mesh(m.verts, m.tets, refl=0.9), 4, mu=0.1)
    x = vectors(op, 6, 9)
    x[0, 100, 3] = float("inf")
    x[1, 100, 3] = -float("inf")
    x[1, 101, 5] = float("inf")
    x[2, 57, 0] = float("nan")
    x[3, 200, 0] = 3.4028234e38  # rounds up to infinity at 11 bits
    x[4, 200, 0] = torch.tensor([0x7F800001], dtype=torch.int32).view(torch.float32).item()
    y = op.apply(x)
    one = torch.cat([op.apply(x[r:r + 1]) for r in range(6)])
    assert bool((y.isnan() == one.isnan()).all())
    assert bool((y.isposinf() == one.isposinf()).all()) and bool((y.isneginf() == one.isneginf()).all())
    assert int((~one.isfinite()).sum()) > 0 and bool(one[3].isfinite().all()) and bool(one[5].isfinite().all())
    fin = one.isfinite()
    scale = x[:, :, :].abs().nan_to_num(posinf=0.0).amax((1, 2), keepdim=True)
    assert float(((y - one) / scale)[fin].abs().max()) <= TOL * float(op.blocks().abs().sum((1, 3)).max())
