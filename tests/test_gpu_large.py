"""Problems whose size passes a limit of the launches or of the memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1302_4018_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hp():
    from paper_1302_4018_gb300 import build as b

    b.build()
    from paper_1302_4018_gb300 import hprobe

    return hprobe


@pytest.fixture()
def ctx(hp):   # a context of its own: the workspace goes with the test
    torch.cuda.empty_cache()
    c = hp.Context(0)
    yield c
    c.close()
    torch.cuda.empty_cache()


# More tiles of 128 sites than a grid has rows (65535), full lattice and even-odd pair kernels.  The links repeat those of a small
# lattice and probe 0 is constant, so the solution repeats too: q per site and the iterations are those of the small
# lattice (1e-9: both residuals are 1e-10, as in the parity tests).
@pytest.mark.parametrize("dims,eo", [((64, 64, 64, 34), 0), ((64, 64, 64, 66), 1)])
def test_wilson_lattice_of_more_tiles_than_grid_rows(ctx, hp, dims, eo):
    small = (8, 8, 8, 2)
    U = synth.gauge_links(small, 0.3, 61)
    u = torch.from_numpy(U.view(np.float64).reshape(*small[::-1], 72)).to("cuda:0")
    opts = dict(z0_seed=0, even_odd=eo, rhs_block=4, eo_kernel=4)
    ref, _, st0 = ctx.trace_inv(ctx.make_operator(hp.OP_WILSON, 0.05, 0.11, u.reshape(-1)), small, 1, 1e-10,
                                ctx.make_opts("fp64", **opts))
    big = u.repeat(*(a // b for a, b in zip(dims[::-1], small[::-1])), 1).reshape(-1)
    T, _, st = ctx.trace_inv(ctx.make_operator(hp.OP_WILSON, 0.05, 0.11, big), dims, 1, 1e-10,
                             ctx.make_opts("fp16", maxiter=2 * st0["iterations_max"] + 20, **opts))
    assert st["max_true_residual"] <= 1e-10
    scale = np.prod(dims) / np.prod(small)
    assert np.all(np.abs(T - scale * ref) <= 1e-9 * np.abs(T))


# A solve per cluster keeps every resident right-hand side's vectors: 304 of 128^3 would hold 20 GB where the slot engine
# takes 0.8, and 76 of 64^3 find no room (0.64 GB) on a device with 0.4 GB left, where the slot engine (0.13) still does.
# 1e-7: q = z^T x to |r| / lambda_min with residuals of 1e-9 |b|, against the slot engine with its own.
@pytest.mark.parametrize("dims,s,leave,most", [((128, 128, 128), 304, None, 9.4e9), ((64, 64, 64), 76, 0.4e9, 0.4e9)])
def test_laplacian_workspace_is_bounded(ctx, hp, dims, s, leave, most):
    op = ctx.make_operator(hp.OP_LAPLACIAN, 0.3)
    opts = dict(z0_seed=4, probe_kind="z2")
    ref, _, _ = ctx.trace_inv(op, dims, 2, 1e-9, ctx.make_opts("fp64", rhs_block=2, **opts))
    free = torch.cuda.mem_get_info()[0]
    filler = None if leave is None else torch.empty(int(free - leave), dtype=torch.uint8, device="cuda:0")
    before = torch.cuda.mem_get_info()[0]
    T, _, st = ctx.trace_inv(op, dims, s, 1e-9, ctx.make_opts("fp64", **opts))
    used = before - torch.cuda.mem_get_info()[0]
    del filler
    assert st["rhs_solved"] == s and st["max_true_residual"] <= 1e-9
    assert used <= most
    assert np.all(np.abs(T[:2] - ref) <= 1e-7 * np.abs(ref))


# The Laplacian's route for a batch: a solve per cluster (a few launches) where the lattices are alike, but not where one
# solve of the largest on one block outlasts all the others (the slot engine launches four kernels an iteration).
@pytest.mark.parametrize("batch,clusters", [([((8, 8, 8, 8), 64), ((64, 64, 64), 1)], False),
                                            ([((8, 8, 8, 8), 64), ((16, 16, 16), 64)], True),
                                            ([((12, 12, 12), 20), ((16, 16, 16), 20), ((24, 24, 24), 20)], True)])
def test_laplacian_batch_route_and_values(ctx, hp, batch, clusters):
    dims, s = zip(*batch)
    ops = [ctx.make_operator(hp.OP_LAPLACIAN, 0.3)] * len(batch)
    opts = dict(z0_seed=4, probe_kind="z2")
    n0 = ctx.launch_count()
    T, st = ctx.trace_inv_batch(ops, dims, s, 1e-10, ctx.make_opts("fp64", **opts))
    launches = ctx.launch_count() - n0
    assert st["max_true_residual"] <= 1e-10 and (launches < 4 * st["iterations_max"]) == clusters
    ref, _ = ctx.trace_inv_batch(ops, dims, s, 1e-10, ctx.make_opts("fp64", rhs_block=16, **opts))
    for a, b in zip(T, ref):
        assert np.all(np.abs(a - b) <= 1e-8 * np.abs(b))


# More than 96 right-hand sides in FP32 run in a block of 128 (1.6 GB here) where that finds room, else in the block of
# 64 (0.8 GB) they always had.  Both blocks iterate to 1e-9 |b|; 1e-7 as above.
def test_sparse_block_width_falls_back_to_the_room_there_is(ctx):
    rp, ci, val = synth.grid_matrix((80, 80, 80), 5, shift=0.3)
    rp, ci, val = (torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0") for a in (rp, ci, val))
    paths = torch.zeros((1, 80 ** 3), dtype=torch.int32, device="cuda:0")
    opts = dict(z0_seed=4, probe_kind="z2")
    ref, _, _ = ctx.trace_inv_sparse(rp, ci, val, paths, [1], 2, 1e-9, ctx.make_opts("fp32", rhs_block=32, **opts))
    filler = torch.empty(int(torch.cuda.mem_get_info()[0] - 0.7e9), dtype=torch.uint8, device="cuda:0")
    T, _, st = ctx.trace_inv_sparse(rp, ci, val, paths, [1], 100, 1e-9, ctx.make_opts("fp32", **opts))
    del filler
    assert st["rhs_solved"] == 100 and st["max_true_residual"] <= 1e-9
    assert np.all(np.abs(T[:2] - ref) <= 1e-7 * np.abs(ref))
