"""The one-launch Neumann series and the streamed application of the wide bases
against the general paths."""
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


def operator(D, n, Np, **kw):
    m = kuhn_cube_mesh(n, jitter=0.2 if n > 1 else 0.0, seed=4)
    return D.Operator(D.Mesh(m.verts, m.tets, refl=0.8), Np, mu=0.5, **kw)


# one block; several with a barrier; rows that do not divide among the blocks;
# every block of the chip; too large for shared memory (the general loop)
@pytest.mark.parametrize("n,Np", [(1, 0), (1, 2), (1, 8), (2, 4), (3, 3), (5, 3), (5, 5), (8, 4)])
def test_neumann_series_in_one_launch(D, n, Np):
    """x <- b + B x by the library's application until the increment meets the
    tolerance: the same terms, the same iterate to rounding."""
    import torch

    op = operator(D, n, Np, precision=D.F64)
    b = D.source(op.mesh, Np, [0, 4 * op.mesh.n_tets - 1])
    rho, info = op.solve(b, method=D.NEUMANN, tol=1e-9)
    iters = 0
    for r in range(2):
        x = torch.zeros_like(b[r])
        while True:
            new = op.apply(x, x0=b[r])
            iters += 1
            done = float((new - x).norm()) <= 1e-9 * float(new.norm())
            x = new
            if done:
                break
        assert float((rho[r] - x).abs().max()) <= 1e-14 * float(x.abs().max())
    assert info.iters == iters
    # an initial guess is taken up, the cap is kept, a bad right-hand side is seen
    assert op.solve(b, method=D.NEUMANN, tol=1e-9, x0=rho)[1].iters == 2
    with pytest.raises(D.DFMError) as e:
        op.solve(b, method=D.NEUMANN, tol=1e-14, max_iter=3)
    assert e.value.code == D.DFM_ERR_NOT_CONVERGED
    b[0, 0, 0] = float("nan")
    with pytest.raises(D.DFMError) as e:
        op.solve(b, method=D.NEUMANN, tol=1e-9)
    assert e.value.code == D.DFM_ERR_NONFINITE
    op.check_error()


# chunks that end with and without a remainder, every alignment of the three
# blocks' starts (odd and even sizes), several launches of right-hand sides
@pytest.mark.parametrize("Np,R", [(9, 1), (10, 3), (11, 8), (12, 9), (15, 2), (16, 1), (20, 2)])
def test_streamed_wide_application(D, Np, R):
    """FP32 against FP64 vectors on the same blocks (another kernel): sums of up
    to 693 products in FP32, error below 32 * 2^-24 of the terms' size."""
    import torch

    op = operator(D, 2, Np)
    g = torch.Generator(device="cuda").manual_seed(1)
    x, x0 = (torch.randn((R, op.n_rows, op.nb), generator=g, device="cuda") for _ in range(2))
    for kw, kw64 in (({}, {}), (dict(x0=x0, alpha=-0.5), dict(x0=x0.double(), alpha=-0.5))):
        y, ref = op.apply(x, **kw), op.apply(x.double(), **kw64)
        assert float((y - ref).abs().max()) <= 4e-6 * float(ref.abs().max())
    op.check_error()


def test_neumann_series_is_accounted_for(D):
    """The one launch of a series is in the statistics of the applications it stands
    for: every term takes over a microsecond, the residual after them some 6."""
    op = operator(D, 1, 2, precision=D.F64)
    b = D.source(op.mesh, 2, [0])
    op.solve(b, method=D.NEUMANN, tol=1e-12)
    D.stats_reset()
    D.stats_enable(1)
    try:
        _, info = op.solve(b, method=D.NEUMANN, tol=1e-12)
    finally:
        D.stats_enable(0)
    launches, ms = D.kernel_stats(5)  # DFM_KERNEL_SPMV64
    D.stats_reset()
    assert info.iters > 20 and launches >= 2 and ms > 1e-3 * info.iters


REFUSED = """
// stands in for the CUDA runtime's call in a child process: a launch that does not fit
extern "C" int cudaLaunchCooperativeKernel(const void*, ...) { return 720; }  // cudaErrorCooperativeLaunchTooLarge
"""


def test_neumann_series_where_the_launch_is_refused(D, tmp_path):
    """A device that does not take all blocks at once (here a stand-in for the
    runtime call that says so): the general loop solves the same system."""
    import os
    import shutil
    import subprocess
    import sys

    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, lib = tmp_path / "refused.cpp", tmp_path / "librefused.so"
    src.write_text(REFUSED)
    subprocess.run([cxx, "-shared", "-fPIC", str(src), "-o", str(lib)], check=True)
    prog = """
import torch
from paper_1608_04607_gb300 import dfm as D
from paper_1608_04607_gb300.inputs import kuhn_cube_mesh
out = []
for n in (1, 3):
    m = kuhn_cube_mesh(n, jitter=0.2 if n > 1 else 0.0, seed=8)
    op = D.Operator(D.Mesh(m.verts, m.tets, refl=0.9), 3, mu=0.1, precision=D.F64)
    b = D.source(op.mesh, 3, [0])
    rho, info = op.solve(b, method=D.NEUMANN, tol=1e-10)
    r = rho[0] - op.apply(rho[0], x0=b[0])
    out.append((info.iters, float(r.norm() / rho.norm())))
print(out)
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    got = []
    for preload in ("", str(lib)):
        env = dict(os.environ, LD_PRELOAD=preload, PYTHONPATH=root)
        p = subprocess.run([sys.executable, "-c", prog], capture_output=True, text=True, env=env, cwd=root, timeout=300)
        assert p.returncode == 0, p.stderr[-2000:]
        got.append(eval(p.stdout.strip().splitlines()[-1]))
    for (it, res), (it0, res0) in zip(*got):
        assert it == it0 and res <= 1e-9 and res0 <= 1e-9
