"""GPU parity of mesh set-up, quadrature tables and operator assembly against
the FP64 oracle (all calls go through the C ABI of libdfm).

Tolerances: the GPU integrates each direction patch with a fixed Gauss rule
(order Np + 6 after splitting patches to <= 60 degrees), which the oracle's
order doubling shows to be accurate to ~3e-7 of the block max-norm; FP32
arithmetic adds ~1e-6.  Operator entries must match to 1e-5 relative to the
block max-norm in FP32 (the method's stated entry tolerance) and 2e-6 in FP64.
"""
import numpy as np
import pytest

from gpu_helpers import block_rel_err, need_gpu, to_oracle_layout
from paper_1608_04607_gb300.inputs import kuhn_cube_mesh, workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    need_gpu()
    from paper_1608_04607_gb300 import dfm

    dfm.load()
    return dfm


def test_gauss_legendre_on_device(D):
    for q in (1, 2, 5, 10, 16, 32, 64):
        x, w = D.gauss_legendre(q)
        xr, wr = np.polynomial.legendre.leggauss(q)
        np.testing.assert_allclose(x.cpu().numpy(), xr, atol=2e-15)
        np.testing.assert_allclose(w.cpu().numpy(), wr, atol=2e-15)


def test_mesh_topology_matches_oracle(D, oracle_mod):
    for n, jit in ((1, 0.0), (3, 0.2), (6, 0.2)):
        m = kuhn_cube_mesh(n, jitter=jit, seed=4)
        mesh = D.Mesh(m.verts, m.tets, refl=0.9)
        topo = oracle_mod.topology(m.tets)
        np.testing.assert_array_equal(mesh.recv(), topo.recv)
        info = mesh.info()
        assert info.n_boundary_rows == 12 * n * n
        assert info.total_volume == pytest.approx(1.0, rel=1e-12)


def test_mesh_errors_are_reported(D):
    m = kuhn_cube_mesh(1, jitter=0.0)
    bad = m.tets.copy()
    bad[0, 0] = 99
    with pytest.raises(D.DFMError) as e:
        D.Mesh(m.verts, bad)
    assert e.value.code == D.DFM_ERR_MESH
    # three tets sharing one face
    V = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 1]], float)
    T = np.array([[0, 1, 2, 3], [0, 1, 2, 4], [0, 1, 2, 5]], np.int32)
    with pytest.raises(D.DFMError) as e:
        D.Mesh(V, T)
    assert e.value.code == D.DFM_ERR_MESH
    # flat tet
    V2 = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [1, 1, 0]], float)
    with pytest.raises(D.DFMError) as e:
        D.Mesh(V2, np.array([[0, 1, 2, 3]], np.int32))
    assert e.value.code == D.DFM_ERR_MESH
    with pytest.raises(D.DFMError) as e:
        D.Mesh(m.verts, m.tets, refl=1.5)
    assert e.value.code == D.DFM_ERR_ARG


def _oracle_op(oracle_mod, m, mu, refl, Np, rtol=1e-12):
    return oracle_mod.assemble(m.verts, m.tets, mu, refl, Np, rtol=rtol)


@pytest.mark.parametrize("prec,tol", [(0, 2e-6), (1, 1e-5)])
def test_assembly_single_cube(D, oracle_mod, prec, tol):
    w = workload("kuhn1_np2")
    m = w["mesh"]
    mesh = D.Mesh(m.verts, m.tets, refl=w["refl"])
    op = D.Operator(mesh, w["Np"], mu=0.1, precision=prec)
    got = to_oracle_layout(op.blocks().cpu().numpy(), mesh.recv(), m.n_tets)
    ref = _oracle_op(oracle_mod, m, w["mu"], w["refl"], w["Np"])
    err = block_rel_err(got, ref.blocks)
    assert err.max() <= tol, err.max()


@pytest.mark.parametrize("Np", [0, 1, 3, 4, 6, 8])
def test_assembly_jittered_fp32(D, oracle_mod, Np):
    import torch

    m = kuhn_cube_mesh(2, jitter=0.2, seed=21)
    rng = np.random.default_rng(Np)
    mu = rng.uniform(0.0, 0.4, m.n_tets)
    mesh = D.Mesh(m.verts, m.tets, refl=0.8)
    op = D.Operator(mesh, Np, mu=torch.tensor(mu, device="cuda"), precision=D.F32)
    got = to_oracle_layout(op.blocks().cpu().numpy(), mesh.recv(), m.n_tets)
    topo = oracle_mod.topology(m.tets)
    t, f, fp = oracle_mod.pair_list(m.n_tets)
    sel = np.arange(12 * m.n_tets) if Np <= 4 else rng.choice(12 * m.n_tets, 96, replace=False)
    ref, _, q, _ = oracle_mod.blocks_for_pairs(m.verts, m.tets, topo, mu, 0.8, Np, t[sel], f[sel], fp[sel],
                                               rtol=1e-12)
    err = block_rel_err(got.reshape(-1, got.shape[2], got.shape[3])[sel], ref)
    assert err.max() <= 1e-5, (err.max(), np.argmax(err))


def test_assembly_is_deterministic_and_reassembles(D):
    import torch

    m = kuhn_cube_mesh(3, jitter=0.2, seed=2)
    mesh = D.Mesh(m.verts, m.tets, refl=0.95)
    op = D.Operator(mesh, 4, mu=0.05)
    a = op.blocks().clone()
    op.reassemble(0.3)
    b = op.blocks().clone()
    op.reassemble(0.05)
    c = op.blocks()
    assert torch.equal(a, c)
    assert not torch.equal(a, b)


@pytest.mark.parametrize("Np", range(9))
@pytest.mark.parametrize("quad_order,deg,mu,moment", [(0, 0.0, 0.05, 0), (1, 180.0, 0.0, 0), (7, 10.0, 0.4, 0),
                                                      (32, 60.0, 40.0, 0), (0, 0.0, 0.4, 2)])
def test_tensor_core_blocks_match_the_fp64_rule(D, Np, quad_order, deg, mu, moment):
    """FP32 blocks (FP16 hi + lo products on tensor cores) against FP64 blocks of
    the same rule: one node to 1,024 nodes per patch, subdivision to its deepest
    levels, damping from none to strong, a damping moment; one to three tiles of
    test functions.  Both run the same set-up and subdivision arithmetic, so the
    node counts agree and the entries to the FP32 entry tolerance."""
    m = kuhn_cube_mesh(2, jitter=0.2, seed=5)
    mesh = D.Mesh(m.verts, m.tets, refl=0.8)
    kw = dict(mu=mu, quad_order=quad_order, max_patch_deg=deg, moment=moment)
    a, b = D.Operator(mesh, Np, **kw), D.Operator(mesh, Np, precision=D.F64, **kw)
    assert D.op_nodes(a) == D.op_nodes(b)
    x, y = a.blocks().double(), b.blocks()
    err = (x - y).abs().amax((2, 3)) / y.abs().amax((2, 3))
    assert float(err.max()) <= 1e-5


@pytest.mark.parametrize("Np", [0, 1, 2, 4, 5, 6, 8, 10, 13, 16, 17, 20])
def test_block_entries_have_no_common_loss(D, Np):
    """The tensor cores round towards zero: entries smaller by a common factor
    would be magnified by a solve at little damping.  Mean relative error of the
    entries of the tensor-core kernels (all orders but 9) against FP64 blocks of the
    same rule (the basis is hierarchical), at most the expected loss of one truncation, 2^-24 x 0.72 = 4.3e-8."""
    m = kuhn_cube_mesh(3, jitter=0.2, seed=5)
    mesh = D.Mesh(m.verts, m.tets, refl=1.0)
    kw = dict(mu=0.05, quad_order=14, max_patch_deg=60.0)
    a = D.Operator(mesh, Np, **kw).blocks()
    b = D.Operator(mesh, min(Np, 8), precision=D.F64, **kw).blocks()
    n = b.shape[2]
    d = a[..., :n, :n].double() - b
    assert abs(float((d * b.sign()).sum() / b.abs().sum())) <= 4.3e-8
    assert abs(float(d[..., 0, 0].sum() / b[..., 0, 0].sum())) <= 4.3e-8


@pytest.mark.parametrize("quad_order", [7, 14])
@pytest.mark.parametrize("Np", [2, 4, 5, 6, 7, 8])
def test_isotropic_entries_do_not_depend_on_the_order(D, Np, quad_order):
    """The entry (0, 0) is the sum of the node weights, whatever the order: with
    the tensor cores' sums exact, every order adds the same numbers in the same
    sequence.  The entries' means differ by nothing, or by the mean of FP32
    roundings (at most 1e-7 each) over the 4,608 pairs where a compiler fuses a
    multiplication differently: 1.5e-9, times 3."""
    m = kuhn_cube_mesh(4, jitter=0.2, seed=7)
    mesh = D.Mesh(m.verts, m.tets, refl=1.0)
    kw = dict(mu=0.3, quad_order=quad_order, max_patch_deg=60.0)
    a = D.Operator(mesh, Np, **kw).blocks()[..., 0, 0].double()
    b = D.Operator(mesh, 0, **kw).blocks()[..., 0, 0].double()
    assert abs(float((a - b).sum() / b.sum())) <= 4.5e-9


@pytest.mark.parametrize("Np,quad_order", [(Np, Np + 6) for Np in (2, 3, 4, 5, 6, 7, 8, 10, 12)]
                         + [(0, 9), (4, 14)])
def test_energy_is_conserved_on_average(D, Np, quad_order):
    """Without damping, and with fully reflecting walls, the uniform isotropic
    density is stationary (Sec. 2): its total energy after one application is what
    it was, to the mean relative error of the entries (0, 0).  That is the effect of the
    Gauss nodes' rounding to FP32, common to all pairs (at most 1.1e-8 at these
    orders by a CPU evaluation of the rule in 64 bits with the nodes rounded), and the
    mean of the pairs' own roundings (root mean square 2e-7 at most), three
    standard deviations of it.  The rule's own error is below 6e-10."""
    n = 4 if Np <= 8 else 3
    m = kuhn_cube_mesh(n, jitter=0.2, seed=3)
    P = m.verts[np.stack([np.roll(m.tets, -(f + 1), axis=1)[:, :3] for f in range(4)], 1)]  # [tets, 4, 3, xyz]
    area = 0.5 * np.linalg.norm(np.cross(P[:, :, 1] - P[:, :, 0], P[:, :, 2] - P[:, :, 0]), axis=-1).reshape(-1)
    mesh = D.Mesh(m.verts, m.tets, refl=1.0)
    op = D.Operator(mesh, Np, mu=0.0, quad_order=quad_order, max_patch_deg=60.0)
    import torch

    s = torch.as_tensor(np.sqrt(area), device="cuda")
    x = torch.zeros((1, op.n_rows, op.nb), dtype=torch.float64, device="cuda")
    x[0, :, 0] = s
    got = float((s * op.apply(x)[0, :, 0]).sum())
    assert abs(got / area.sum() - 1.0) <= 1.1e-8 + 6e-10 + 3 * 2e-7 / np.sqrt(12 * m.n_tets)
