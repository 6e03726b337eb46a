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


@pytest.mark.parametrize("B", [1, 15, 17, 127, 128, 129, 145, 257])
@pytest.mark.parametrize("nodes", ["209", "481"])
def test_demag_product_tile_and_slice_edges(ctx, B, nodes):
    """Island counts around the GEMM's tile steps (16 islands, 128 where K is no longer sliced, 256) on two operators
    whose row count is (1536) and is not (704) a multiple of the 128-row tile: the demag field of the split product
    against the CUDA-core evaluation of the same products, within one rounding of 2^-23 of the field scale per MMA."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    mesh = synth.small_island_mesh() if nodes == "209" else \
        synth.layered_island_mesh(12.0, 6.0, 6.0, rings=3, hard_slabs=6, soft_slabs=6, seed=7)
    mid = ctx.mesh_upload(mesh, synth.ecc_materials())
    K = ctx.mesh_info(mid)["k_pad"]
    isl = synth.jittered_islands(B, seed=B, mesh_id=mid)
    p = synth.RunParams(dt_ps=0.1, substeps=1, term_mask=L.TERM_DEMAG)
    rng = np.random.default_rng(B)
    m = rng.standard_normal((B, 3, mesh.n_nodes)) * 0.3
    m[:, 2] += 1.0
    m = (m / np.linalg.norm(m, axis=1, keepdims=True)).astype(np.float32)
    out = []
    for prec in (L.PREC_BF16X3_REF, L.PREC_BF16X3):
        with ctx.batch(isl, p, precision=prec) as bt:
            bt.set_state(m, 0.0)
            out.append(bt.field(0.0, L.TERM_DEMAG))
    ctx.mesh_release(mid)
    assert np.abs(out[1] - out[0]).max() <= (3 * K / 16) * 2.0 ** -23 * np.abs(out[0]).max()


@pytest.mark.parametrize("sizes", [(129,), (300,), (40, 130), (1, 64, 200), (900,), (331, 400), (20, 130)])
def test_few_island_stages_match_the_two_island_stages(ctx, sizes):
    """Batches on the stage kernels of few islands (one and several mesh groups, 256 and 512 threads a CTA; two
    islands a CTA beyond one an SM) against the same run on the CTA-pair GEMM, which takes the two-island stage kernels.  A group of more than 128 islands has
    the same products in the same order on both sides: m and the switch data are bitwise equal, <m_z> up to the order
    of its sum.  Smaller groups slice K on one side: within the drift of the GEMM's rounding (2^-23 of the field per
    MMA, 1e-4 over the run as in the pair GEMM's own run test)."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    meshes = [synth.layered_island_mesh(12.0, 6.0, 6.0, rings=3, hard_slabs=6, soft_slabs=6, seed=7),
              synth.small_island_mesh(), synth.layered_island_mesh(7.0, 6.0, 4.0, rings=2, hard_slabs=9, soft_slabs=6)]
    mids = [ctx.mesh_upload(meshes[-1 - k], synth.ecc_materials()) for k in range(len(sizes))]
    hid = ctx.headmap_upload(synth.synthetic_head_map())
    isl = synth.Islands.concat([synth.jittered_islands(b, seed=b, mesh_id=m) for b, m in zip(sizes, mids)])
    p = synth.RunParams(dt_ps=0.1, alpha=0.1, rise_ps=2.0, use_map=True, x0_nm=-2.0, substeps=0,
                        uniform_T=synth.uniform_field(0.9, 170.0))
    out = []
    for pair in (0, 1):
        with ctx.batch(isl, p, precision=L.PREC_BF16X3, map_id=hid) as bt:
            bt.set_tuning(256, 256, L.RASTER_AUTO, 2, 32, gemm_pair=pair)
            bt.advance(40)
            out.append(bt.read())
    few, two = out
    assert np.all(few["status"] == 0) and np.abs(few["mz"] - 1.0).max() > 0.02      # the islands have moved
    for b, m in zip(sizes, mids):
        r = np.asarray(isl.mesh_id) == m
        if b > 128:
            assert np.array_equal(few["m"][r], two["m"][r]) and np.array_equal(few["t_sw"][r], two["t_sw"][r])
            assert np.abs(few["mz"][r] - two["mz"][r]).max() <= 1e-6
        else:
            assert np.abs(few["m"][r] - two["m"][r]).max() <= 1e-4
    for m in mids:
        ctx.mesh_release(m)
    ctx.headmap_release(hid)


@pytest.mark.parametrize("B", [1, 16, 31, 32, 33, 64, 65, 130])
def test_fp32_product_tile_edges(ctx, B):
    """Row counts around the FP32 GEMM's tiles (16 rows up to 32, 64 beyond) on an operator whose columns (704) end
    inside a 64-column tile: against the FP64 product of the exported FP32 operator and the same FP32 sources.  A sum
    of K products in FP32 with four partial sums: K/4 * 2^-24 of the sum of magnitudes, K = 704."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    mesh = synth.small_island_mesh()
    mid = ctx.mesh_upload(mesh, synth.ecc_materials())
    n = mesh.n_nodes
    isl = synth.jittered_islands(B, seed=B, mesh_id=mid)
    rng = np.random.default_rng(B)
    m = rng.standard_normal((B, 3, n)).astype(np.float32)
    m /= np.linalg.norm(m, axis=1, keepdims=True)
    with ctx.batch(isl, synth.RunParams(dt_ps=0.1, substeps=1, term_mask=L.TERM_DEMAG), precision=L.PREC_FP32) as bt:
        bt.set_state(m, 0.0)
        got = bt.field(0.0, L.TERM_DEMAG).reshape(B, 3 * n)
    Ms = (ctx.get_operator(mid, L.OP_NODAL_MS_F64) * 1e-6).astype(np.float32)
    src = ((Ms[None] * isl.Ms_scale[:, None])[:, None] * m).astype(np.float64).reshape(B, 3 * n)
    W = ctx.get_operator(mid, L.OP_DEMAG_F32).astype(np.float64)
    ctx.mesh_release(mid)
    bound = (176 * 2.0 ** -24 + 2.0 ** -22) * (np.abs(src) @ np.abs(W).T)      # + the sources' own FP32 rounding
    assert np.all(np.abs(got - src @ W.T) <= bound)


@pytest.mark.parametrize("shape", [(16, 256, 4, 2), (3, 100, 1, 5), (70, 130, 2, 17), (200, 256, 6, 128)])
def test_one_kernel_forward_matches_the_layers(ctx, shape):
    """The forward pass in one kernel at its edges (one input k-block to four, padded and whole widths, depths 1 and 6,
    one to eight output groups of 16; one sample, a full tile, two and more tiles of an SM) against the layer-by-layer
    forward pass of the gradient call: the loss of both must agree.  Probabilities and logits go through FP32 once
    more (a sigmoid and its inverse): 1e-5 of the loss."""
    from paper_1603_09493_gb300 import synth
    n_in, width, depth, n_out = shape
    sizes = [n_in] + [width] * depth + [n_out]
    sur = ctx.surrogate(shape, synth.mlp_init_params(sizes, seed=sum(shape)))
    rng = np.random.default_rng(n_in)
    X = rng.uniform(-1, 1, (152 * 128 * 3 + 77, n_in)).astype(np.float32)
    P = sur.infer(X)
    for N in (1, 127, 128, 129, 152 * 128 + 1):
        assert np.array_equal(sur.infer(X[:N]), P[:N])
    for lo, N in ((0, 1), (100, 300), (152 * 128 - 60, 500), (152 * 128 * 3 - 50, 127)):
        x, y = X[lo:lo + N], (rng.random((N, n_out)) < 0.5).astype(np.float32)
        p = P[lo:lo + N].astype(np.float64)
        loss = -np.mean(y * np.log(p) + (1 - y) * np.log1p(-p))
        assert abs(sur.grad(x, y)[1] - loss) <= 1e-5 * max(1.0, loss)
    sur.destroy()


@pytest.mark.parametrize("n", [31, 32, 33, 62, 63, 64, 65, 160, 240])
def test_blocked_kriging_factors(ctx, n):
    """Design counts around the factorisation's 32-column blocks (one CTA to seven below a block; the rows of y and 1
    in the last block, in one of their own or on both sides of an edge): likelihoods, the fit and the predictor against
    the FP64 oracle.  Condition numbers up to 1.4e6, so the bars of well-conditioned models hold: 1e-9 for likelihood,
    mean and variance, 1e-8 of the data scale for predictions."""
    from oracle import ego as oego
    from paper_1603_09493_gb300 import ego, synth
    X = synth.unit_points(n, 4, 12, 0)
    y = np.sin(3.0 * X).sum(1)
    th = 10.0 ** (0.5 + 1.5 * synth.theta_unit_draws(24, 4, 12, 0))
    got = ego.nll(ctx, X, y, th)
    assert np.allclose(got, [oego.nll(X, y, t) for t in th], rtol=1e-9, atol=1e-9)
    gp = oego.fit(X, y, th[0])
    C = synth.unit_points(333, 4, 9, 1)
    ry, rs, rei = oego.predict(gp, C, float(y.min()))
    with ego.Kriging(ctx, X, y, th[0]) as k:
        assert abs(k.mu - gp["mu"]) <= 1e-9 * np.abs(y).max() and abs(k.sigma2 - gp["sigma2"]) <= 1e-9 * gp["sigma2"]
        gy, gs, gei = k.predict(C, float(y.min()))
    scale = np.abs(y).max()
    assert max(np.abs(gy - ry).max(), np.abs(gs - rs).max(), np.abs(gei - rei).max()) <= 1e-8 * scale


@pytest.mark.parametrize("n,T", [(240, 256), (160, 600), (512, 150)])
def test_more_kriging_factors_than_the_gpu_holds(ctx, n, T):
    """Batches whose panel launches have more CTAs than are resident at once (1792, 3000 and 2400; eight an SM), so
    that CTAs of one matrix start after others of it have finished: every likelihood against the FP64 oracle, and
    bitwise equal to that of the vector in a small batch and of a second call."""
    from oracle import ego as oego
    from paper_1603_09493_gb300 import ego, synth
    X = synth.unit_points(n, 12, 12, 0)
    y = np.sin(3.0 * X).sum(1)
    th = 10.0 ** (0.5 + synth.theta_unit_draws(T, 12, 12, 0))
    got = ego.nll(ctx, X, y, th)
    assert np.array_equal(got, ego.nll(ctx, X, y, th))
    assert np.array_equal(got, np.concatenate([ego.nll(ctx, X, y, th[q:q + 50]) for q in range(0, T, 50)]))
    assert np.allclose(got, [oego.nll(X, y, t) for t in th], rtol=1e-9, atol=1e-9)


def test_kriging_pivot_failing_in_a_later_block(ctx):
    """A matrix whose first 70 pivots are those of the unit matrix and whose pivot 70 is 1 - e^2 (a negative
    correlation parameter in a direction in which only two designs differ), between good ones: infinity for it alone,
    as the oracle has it."""
    from oracle import ego as oego
    from paper_1603_09493_gb300 import ego
    n = 100
    X = np.zeros((n, 2))
    X[:, 0] = np.arange(n) / n
    X[70] = [X[45, 0], 1.0]
    y = np.sin(7.0 * X[:, 0]) + X[:, 1]
    th = np.array([[1e6, 1.0], [1e6, -1.0], [1e5, 0.5]])
    got = ego.nll(ctx, X, y, th)
    ref = [oego.nll(X, y, t) for t in th]
    assert np.isinf(ref[1]) and np.isfinite(ref[0]) and np.isfinite(ref[2])
    assert np.isinf(got[1]) and np.allclose(got[[0, 2]], [ref[0], ref[2]], rtol=1e-9, atol=1e-9)


@pytest.mark.parametrize("parts", [2, 3])
def test_operators_of_meshes_of_several_bodies(ctx, parts):
    """A hard and a soft prism across a gap and, with three, a single tetrahedron beside them, nodes numbered
    alternately over the bodies: the Laplacian has a null vector per body, so the nodal sources of the Neumann
    problem have to sum to zero over each.  FP64 demag matrix against the oracle's, as for one body."""
    from oracle import fem
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    a = synth.layered_island_mesh(8.0, 5.0, 3.0, rings=2, hard_slabs=3, soft_slabs=2, seed=1)
    b = synth.layered_island_mesh(9.0, 4.0, 4.0, rings=1, hard_slabs=2, soft_slabs=2, seed=2)
    xyz, tets, reg = [a.xyz_nm, b.xyz_nm + [0.0, 0.0, 9.0]], [a.tets, b.tets + a.n_nodes], [a.tet_region, b.tet_region]
    if parts == 3:
        tets.append(np.arange(4).reshape(1, 4) + a.n_nodes + b.n_nodes)
        xyz.append(np.array([[14.0, 0, 0], [16.0, 0, 0], [14.0, 2.0, 0], [14.0, 0, 2.0]]))
        reg.append(np.zeros(1, reg[0].dtype))
    xyz, tets, reg = np.concatenate(xyz), np.concatenate(tets), np.concatenate(reg)
    new = np.random.default_rng(parts).permutation(len(xyz))              # node i gets number new[i]
    mesh = synth.IslandMesh(xyz[np.argsort(new)], new[tets].astype(np.int32), reg.astype(np.int32), 5.0, 17.0)
    mats = synth.ecc_materials()
    ops = fem.MeshOperators(mesh.xyz_nm, mesh.tets, mesh.tet_region, mats)
    mid = ctx.mesh_upload(mesh, mats, keep_f64=True)
    info = ctx.mesh_info(mid)
    assert info["cg_residual_neumann"] < 1e-12 and info["cg_residual_dirichlet"] < 1e-12
    N = ctx.get_operator(mid, L.OP_DEMAG_F64)
    assert np.abs(N - ops.demag).max() <= 1e-9 * np.abs(ops.demag).max()
    ctx.mesh_release(mid)


def test_mesh_without_a_boundary_is_refused(ctx):
    """Two tetrahedra on the same four nodes: every face belongs to both, none is on the boundary.  An error from the
    library's own check of the faces, before the row count of the boundary's weights divides by their number."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    mesh = synth.IslandMesh(np.array([[0.0, 0, 0], [2, 0, 0], [0, 2, 0], [0, 0, 2]]),
                            np.array([[0, 1, 2, 3], [1, 2, 0, 3]], np.int32), np.zeros(2, np.int32), 1.0, 2.0)
    with pytest.raises(L.BpmError, match="boundary"):
        ctx.mesh_upload(mesh, synth.ecc_materials())


@pytest.mark.parametrize("nodes", ["209", "481", "1547"])
def test_an_island_has_the_same_bits_in_every_batch(ctx, nodes):
    """The demag product's slices of K come from K alone, and their sum has one order: the field and the states of an
    island are bitwise the same in a batch of 300, in parts of it on either side of the 128 islands from which on a
    slice is no longer an item of its own, and on the CTA-pair product; with the split and the single product."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    mesh = {"209": synth.small_island_mesh, "1547": synth.census_island_mesh}.get(
        nodes, lambda: synth.layered_island_mesh(12.0, 6.0, 6.0, rings=3, hard_slabs=6, soft_slabs=6, seed=7))()
    mid = ctx.mesh_upload(mesh, synth.ecc_materials())
    B = 300
    isl = synth.jittered_islands(B, seed=4, mesh_id=mid)
    p = synth.RunParams(dt_ps=0.1, alpha=0.1, rise_ps=1.0, substeps=4, uniform_T=synth.uniform_field(0.9, 170.0))
    rng = np.random.default_rng(5)
    m = rng.standard_normal((B, 3, mesh.n_nodes)) * 0.3
    m[:, 2] += 1.0
    m = (m / np.linalg.norm(m, axis=1, keepdims=True)).astype(np.float32)

    def run(rows, prec, pair=0):
        with ctx.batch(isl.subset(rows), p, precision=prec) as bt:
            if pair:
                bt.set_tuning(256, 256, L.RASTER_AUTO, 2, 32, gemm_pair=1)
            bt.set_state(m[rows], 0.0)
            field = bt.field(0.0, L.TERM_DEMAG)
            bt.advance(2)
            return field, bt.read()["m"]

    for prec in (L.PREC_BF16X3, L.PREC_BF16):
        field, state = run(np.arange(B), prec)
        assert np.abs(state - m).max() > 1e-3                             # the islands have moved
        for rows in (np.arange(1), np.arange(17, 34), np.arange(B - 128, B), np.arange(100, 229)):
            for pair in (0, 1):
                f, s = run(rows, prec, pair)
                assert np.array_equal(f, field[rows]) and np.array_equal(s, state[rows])
    ctx.mesh_release(mid)


@pytest.mark.parametrize("nodes,B", [("209", 40), ("209", 600), ("481", 300)])
def test_autotuned_few_islands_keep_their_intervals(ctx, nodes, B):
    """The autotuner times what a batch of few islands runs, overlapping launches in whole intervals: its choice is no
    slower than a new batch's default, within what two timings of one batch differ by (best of seven each, 15 %)."""
    import time
    from paper_1603_09493_gb300 import synth
    mesh = synth.small_island_mesh() if nodes == "209" else \
        synth.layered_island_mesh(12.0, 6.0, 6.0, rings=3, hard_slabs=6, soft_slabs=6, seed=7)
    mid = ctx.mesh_upload(mesh, synth.ecc_materials())
    isl = synth.jittered_islands(B, seed=4, mesh_id=mid)
    p = synth.RunParams(dt_ps=0.1, alpha=0.1, substeps=8, uniform_T=synth.uniform_field(0.9, 170.0))

    def interval(bt):
        best = 1e9
        for _ in range(8):
            t = time.perf_counter()
            bt.advance(20)
            bt.read()
            best = min(best, time.perf_counter() - t)
        return best

    with ctx.batch(isl, p) as default, ctx.batch(isl, p) as tuned:
        t = tuned.autotune(reps=3)
        assert t["gemm_ms"] > 0 and t["stage_ms"] > 0
        assert interval(tuned) <= 1.15 * interval(default)
    ctx.mesh_release(mid)


def test_chains_of_islands_beyond_the_few(ctx):
    """Tuning streams on batches that are not of few islands (over three pairs an SM; 152 SMs): 1100 and 1300 islands
    of 209 nodes in chunks of a multiple of 128 (two of 640 or three of 384, two of 768, three of 512 or four of 384,
    the last one ragged), and three groups dealt to chains.  A chain has its own kernels of the interval graph; every island sees the same ones, so all results are
    bitwise those of one chain.  A GEMM wait that runs out inside a several-chain graph reports the timeout."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    meshes = [synth.small_island_mesh(), synth.layered_island_mesh(7.0, 6.0, 4.0, rings=2, hard_slabs=9, soft_slabs=6, seed=5),
              synth.layered_island_mesh(6.0, 5.0, 3.0, rings=2, hard_slabs=7, soft_slabs=4, seed=6)]
    mids = [ctx.mesh_upload(m, synth.ecc_materials()) for m in meshes]
    hid = ctx.headmap_upload(synth.synthetic_head_map())
    p = synth.RunParams(dt_ps=0.1, substeps=4, alpha=0.1, rise_ps=10.0, use_map=True, x0_nm=-3.0,
                        uniform_T=synth.uniform_field(0.7, 170.0))
    one = synth.jittered_islands(1100, seed=1, mesh_id=mids[0])
    three = synth.Islands.concat([synth.jittered_islands(b, seed=b, mesh_id=m) for b, m in zip((501, 600, 257), mids)])
    for isl, chains in ((one, (1, 2, 3, 3)), (synth.jittered_islands(1300, seed=2, mesh_id=mids[0]), (1, 2, 3, 4)),
                        (three, None)):
        outs = []
        for streams in (1, 2, 3, 4):
            with ctx.batch(isl, p, precision=L.PREC_BF16X3, map_id=hid) as bt:
                bt.set_tuning(256, 256, L.RASTER_AUTO, 2, 32, streams=streams)
                bt.advance(20)
                outs.append((bt.read(), bt.graph_kernels()))
        if chains:
            assert [k for _, k in outs] == [1 + 16 * c for c in chains]   # four kernels a step and chain, and the clock
        for o, _ in outs:
            for key in ("m", "switched", "t_sw", "mz", "status"):
                assert np.array_equal(o[key], outs[0][0][key]), key
            assert np.all(o["status"] == 0) and np.abs(o["m"][:, :2]).max() > 1e-2     # the islands have moved
    with ctx.batch(one, p, precision=L.PREC_BF16X3, map_id=hid) as bt:
        bt.set_tuning(256, 256, L.RASTER_AUTO, 2, 32, streams=3)
        L.check(ctx.lib.bpm_debug_set_gemm_wait(bt.h, 1000.0))        # 1 us
        bt.advance(2)
        with pytest.raises(L.BpmError) as e:
            bt.read()
        assert e.value.code == L.BPM_ERR_TIMEOUT
    for m in mids:
        ctx.mesh_release(m)
    ctx.headmap_release(hid)


@pytest.mark.parametrize("sizes", [(20,), (120, 120), (300, 200), (40, 150, 90)])
def test_few_islands_of_larger_meshes(ctx, sizes):
    """The stage kernels of few islands on meshes of over 512 nodes (1024 threads a CTA, or 512 where SMs hold several
    islands; several groups at one island a CTA), against the same run on the two-island stage kernels behind the
    CTA-pair product, whose sums are the same: m bitwise, <m_z> up to the order of its sum."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    variants = synth.design_variants()[:4:2] + [dict(mesh=synth.layered_island_mesh(7.0, 6.0, 4.0, rings=3, hard_slabs=9,
                                                                                    soft_slabs=6))]
    meshes = [v["mesh"] for v in variants][:len(sizes)]
    assert all(m.n_nodes > 512 for m in meshes)
    mids = [ctx.mesh_upload(m, synth.ecc_materials()) for m in meshes]
    hid = ctx.headmap_upload(synth.synthetic_head_map())
    isl = synth.Islands.concat([synth.jittered_islands(b, seed=b, mesh_id=m) for b, m in zip(sizes, mids)])
    p = synth.RunParams(dt_ps=0.1, alpha=0.1, rise_ps=2.0, use_map=True, x0_nm=-2.0, substeps=8,
                        uniform_T=synth.uniform_field(0.9, 170.0))
    out = []
    for pair in (0, 1):
        with ctx.batch(isl, p, precision=L.PREC_BF16X3, map_id=hid) as bt:
            bt.set_tuning(256, 256, L.RASTER_AUTO, 2, 32, gemm_pair=pair)
            bt.advance(20)
            out.append(bt.read())
    few, two = out
    assert np.all(few["status"] == 0) and np.abs(few["m"][:, :2]).max() > 1e-2         # the islands have moved
    assert np.array_equal(few["m"], two["m"]) and np.abs(few["mz"] - two["mz"]).max() <= 1e-6
    for m in mids:
        ctx.mesh_release(m)
    ctx.headmap_release(hid)


@pytest.mark.parametrize("B", [33, 64, 65, 130])
def test_fp32_product_column_remainder(ctx, B):
    """The FP32 GEMM's 128-column tiles on an operator of 1472 columns, the last tile half empty: as in
    test_fp32_product_tile_edges, K/4 * 2^-24 of the sum of magnitudes, K = 1472, and the sources' own rounding."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    mesh = synth.layered_island_mesh(12.0, 6.0, 6.0, rings=3, hard_slabs=6, soft_slabs=6, seed=7)
    mid = ctx.mesh_upload(mesh, synth.ecc_materials())
    n = mesh.n_nodes
    assert ctx.mesh_info(mid)["k_pad"] % 128 == 64
    isl = synth.jittered_islands(B, seed=B, mesh_id=mid)
    rng = np.random.default_rng(B)
    m = rng.standard_normal((B, 3, n)).astype(np.float32)
    m /= np.linalg.norm(m, axis=1, keepdims=True)
    with ctx.batch(isl, synth.RunParams(dt_ps=0.1, substeps=1, term_mask=L.TERM_DEMAG), precision=L.PREC_FP32) as bt:
        bt.set_state(m, 0.0)
        got = bt.field(0.0, L.TERM_DEMAG).reshape(B, 3 * n)
    Ms = (ctx.get_operator(mid, L.OP_NODAL_MS_F64) * 1e-6).astype(np.float32)
    src = ((Ms[None] * isl.Ms_scale[:, None])[:, None] * m).astype(np.float64).reshape(B, 3 * n)
    W = ctx.get_operator(mid, L.OP_DEMAG_F32).astype(np.float64)
    ctx.mesh_release(mid)
    bound = (368 * 2.0 ** -24 + 2.0 ** -22) * (np.abs(src) @ np.abs(W).T)
    assert np.all(np.abs(got - src @ W.T) <= bound)


@pytest.mark.parametrize("sizes", [(12, 9, 30, 5, 14, 120), (80, 90, 100, 110), (300, 20, 1, 40, 17)])
def test_groups_of_whole_tiles_have_the_bits_of_their_own_batches(ctx, sizes):
    """Batches of several large meshes, whose tiles fill the SMs without a plane per slice of K (six and five meshes by
    their tiles alone, four by the planes' traffic): field and states of each group bitwise those of a batch of its
    own, which takes the planes where it has up to 128 islands."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    meshes = [v["mesh"] for v in synth.design_variants()[:2 * len(sizes):2]]
    mids = [ctx.mesh_upload(m, synth.ecc_materials()) for m in meshes]
    parts = [synth.jittered_islands(b, seed=b, mesh_id=m) for b, m in zip(sizes, mids)]
    p = synth.RunParams(dt_ps=0.1, alpha=0.1, rise_ps=1.0, substeps=3, uniform_T=synth.uniform_field(0.9, 170.0))
    n_max = max(m.n_nodes for m in meshes)
    rng = np.random.default_rng(5)
    state = []
    for b, mesh in zip(sizes, meshes):
        m = rng.standard_normal((b, 3, mesh.n_nodes)) * 0.3
        m[:, 2] += 1.0
        state.append((m / np.linalg.norm(m, axis=1, keepdims=True)).astype(np.float32))

    def run(isl, m):
        with ctx.batch(isl, p) as bt:
            bt.set_state(m, 0.0)
            field = bt.field(0.0, L.TERM_DEMAG)
            bt.advance(1)
            return field, bt.read()["m"]

    whole = np.concatenate([np.pad(m, ((0, 0), (0, 0), (0, n_max - m.shape[2]))) for m in state])
    field, out = run(synth.Islands.concat(parts), whole)
    at = 0
    for isl, m in zip(parts, state):
        f, s = run(isl, m)
        rows = slice(at, at + len(m))
        at += len(m)
        assert np.array_equal(field[rows, :, :m.shape[2]], f) and np.array_equal(out[rows, :, :m.shape[2]], s)
        assert np.abs(s - m).max() > 1e-3                                 # the islands have moved
    for mid in mids:
        ctx.mesh_release(mid)


@pytest.mark.parametrize("sizes", [(900, 700, 60), (1500, 1, 400), (1200,)])
def test_stages_of_one_plane_and_of_several(ctx, sizes):
    """Batches beyond the few islands on the two-island stage kernels, with a group of at most 128 islands (whose field
    comes in a plane per slice of K, in every stage launch that holds one) and without: states of each group bitwise
    those of parts of 100 islands in batches of their own, which are of few islands."""
    from paper_1603_09493_gb300 import _lib as L
    from paper_1603_09493_gb300 import synth
    meshes = [synth.small_island_mesh(), synth.layered_island_mesh(7.0, 6.0, 4.0, rings=2, hard_slabs=9, soft_slabs=6, seed=5),
              synth.layered_island_mesh(6.0, 5.0, 3.0, rings=2, hard_slabs=7, soft_slabs=4, seed=6)]
    mids = [ctx.mesh_upload(m, synth.ecc_materials()) for m in meshes[:len(sizes)]]
    parts = [synth.jittered_islands(b, seed=b, mesh_id=m) for b, m in zip(sizes, mids)]
    p = synth.RunParams(dt_ps=0.1, alpha=0.1, rise_ps=1.0, substeps=4, uniform_T=synth.uniform_field(0.9, 170.0))

    def run(isl):
        with ctx.batch(isl, p, precision=L.PREC_BF16X3) as bt:
            bt.advance(10)
            return bt.read()["m"]

    out, at = run(synth.Islands.concat(parts)), 0
    assert np.abs(out[:, :2]).max() > 1e-2                                # the islands have moved
    for isl, mesh in zip(parts, meshes):
        n = mesh.n_nodes
        for q in range(0, len(isl), 100):
            rows = np.arange(q, min(q + 100, len(isl)))
            assert np.array_equal(run(isl.subset(rows))[:, :, :n], out[at + rows][:, :, :n])
        at += len(isl)
    for m in mids:
        ctx.mesh_release(m)
