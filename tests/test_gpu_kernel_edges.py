"""Kernels at the sizes where their tiling, remainders and dispatch rules can go wrong."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1603_09493_gb300 import api
    with api.Context(0) as c:
        yield c


@pytest.mark.parametrize("rings,hard,soft", [(1, 3, 1), (1, 2, 1), (2, 3, 2), (3, 5, 4)])
def test_operators_of_small_meshes(ctx, rings, hard, soft):
    """Meshes of 35, 28, 114 and 370 nodes (all or almost all on the boundary, partial 32-row slices, odd column
    counts): the FP64 demag matrix against the oracle's dense one, and lambda_max against its eigenvalues.  CG stops
    below a residual of 1e-12; the Laplacians' condition numbers here are below 1e3."""
    from oracle import fem
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    mesh = synth.layered_island_mesh(8.0, 7.0, 3.0, rings=rings, hard_slabs=hard, soft_slabs=soft, seed=rings + hard)
    mats = synth.ecc_materials()
    ops = fem.MeshOperators(mesh.xyz_nm, mesh.tets, mesh.tet_region, mats)
    mid = ctx.mesh_upload(mesh, mats, keep_f64=True)
    info = ctx.mesh_info(mid)
    assert info["n_nodes"] == ops.n and info["cg_residual_neumann"] < 1e-12
    N = ctx.get_operator(mid, L.OP_DEMAG_F64)
    assert np.abs(N - ops.demag).max() <= 1e-9 * np.abs(ops.demag).max()
    assert abs(info["exchange_lambda_max_T"] - ops.exchange_lambda_max()) <= 1e-9 * ops.exchange_lambda_max()
    ctx.mesh_release(mid)
