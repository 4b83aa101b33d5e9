"""Edges of the sweep and network kernels against the FP64 oracle: every row layout of the general
sweeps, chain lengths around the place where the two chains meet, batches of unlike replicas, and
ragged blocks of the network's mma.sync kernels.  Tolerances as in test_gpu_parity.py (FP64 1e-12,
FP32 1e-5 of the largest value) and test_gpu_net_exact.py (exact, or the FP32 accumulation bound)."""
import itertools
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1204_2088_gb300 import build, dscf, inputs
from test_gpu_net_exact import B, bf16, emulate_forward, exact_problem, flat, paired_integers
from test_gpu_parity import melt, ncomp_shape, random_state, rel, run_gpu, solution, t2n

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    dscf.load()


def check_densities(cfg, precision, seed, tuning=None):
    U = inputs.random_field(ncomp_shape(cfg), seed=seed, scale=0.5)
    ref, _, _ = oracle.densities(cfg, U)
    ctx = dscf.Context(cfg, precision, tuning=tuning)
    for _ in range(2):      # twice: the counters carry over between launches
        got = t2n(ctx.densities(torch.from_numpy(U)))
        ctx.status()
        assert rel(got, ref) < (1e-12 if precision == dscf.FP64 else 1e-5)


@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("nx", [1, 2, 31, 32, 33, 45, 53, 66, 96, 97, 100, 128, 131, 160, 163, 192, 200, 211, 224, 255,
                                256, 257, 300, 511])
def test_general_sweeps_row_layouts(nx, precision):
    check_densities(melt((nx, 3, 5), 5, 2), precision, 20, tuning=(8, 1))


@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("nx", [259, 260, 264, 380, 381, 382, 480, 484, 570, 573, 764, 1000, 1021])
def test_general_sweeps_tiles_of_long_rows(nx, precision):
    """Two to nine tiles a row, of equal and of unequal length, either kind; more planes than one."""
    check_densities(melt((nx, 2, 6), 5, 3), precision, 25, tuning=(8, 1))


@pytest.mark.parametrize("nx,ny,nz", [(2, 1025, 256), (6, 307, 301), (8, 257, 256), (12, 211, 210), (20, 173, 155), (22, 161, 151),
                                      (24, 149, 151), (30, 125, 141), (32, 130, 127),
                                      (32, 61, 68), (16, 99, 83)])
def test_general_sweeps_groups_of_short_rows(nx, ny, nz):
    """Several rows a warp, the last group of fewer; also in a batch beside another layout, bit for bit."""
    cfg = melt((nx, ny, nz), 5, 3)
    assert nx * ny * nz >= 1 << 17 and ny % (32 // (nx // (4 if nx % 4 == 0 else 2)))
    U = inputs.random_field(ncomp_shape(cfg), seed=26, scale=0.5)
    ref, _, _ = oracle.densities(cfg, U)
    other = melt((33, 5, 4), 7, 2)
    V = inputs.random_field(ncomp_shape(other), seed=27, scale=0.5)
    solo = dscf.Context(cfg, dscf.FP32, tuning=(8, 1)).densities(torch.from_numpy(U))
    assert rel(t2n(solo), ref) < 1e-5
    ctx = dscf.Context([cfg, other], dscf.FP32)
    both = ctx.densities(torch.from_numpy(np.concatenate([U.ravel(), V.ravel()])))
    ctx.status()
    assert torch.equal(both[:U.size], solo.reshape(-1))


@pytest.mark.parametrize("N", [2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
def test_general_sweeps_where_the_chains_meet(N, precision):
    for nA in range(1, N):
        check_densities(melt((34, 7, 6), N, nA), precision, 30 + N, tuning=(8, 1))


@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("tile,reps", [((32, 16, 8), (8, 16, 16)),      # even cut of strips of 8 rows
                                       ((32, 16, 8), (8, 8, 32)),       # wide field, one run per warp
                                       ((8, 10, 3), (1, 200, 1)),       # more rows than warps: even cut
                                       ((9, 7, 37), (1, 1, 1))],        # one row plane per warp, uneven CTAs
                         ids=["strips", "runs-wide", "even", "runs-small"])
def test_general_sweeps_cuts(tile, reps, precision):
    """A periodic field of any period has the densities of one period."""
    cfg, big = (melt(g, 4, 1) for g in (tile, tuple(t * r for t, r in zip(tile, reps))))
    U = inputs.random_field(ncomp_shape(cfg), seed=60, scale=0.5)
    ref, _, _ = oracle.densities(cfg, U)
    up = lambda a: np.tile(a, (1,) + reps[::-1])
    ctx = dscf.Context(big, precision, tuning=(8, 1))
    got = t2n(ctx.densities(torch.from_numpy(up(U))))
    ctx.status()
    ctx.close()
    assert rel(got, up(ref)) < (1e-12 if precision == dscf.FP64 else 1e-5)


@pytest.mark.parametrize("N", [2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("grid,zc", [((128, 16, 16), 16), ((64, 8, 8), 8), ((48, 16, 32), 16)])
def test_brick_sweeps_where_the_chains_meet(N, grid, zc):
    for nA in range(1, N):
        check_densities(melt(grid, N, nA), dscf.FP32, 40 + N, tuning=(zc, 0))


@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
def test_general_sweeps_of_unlike_replicas_equal_solo_runs(precision):
    """Row layouts, chain lengths (the cut of the work changes as chains end) and species mixed."""
    cfgs = [melt((33, 9, 10), 9, 4, hydro=1, ncg_iters=2, cn_sweeps=4),
            solution((100, 4, 6), 6, 3, hydro=1, ncg_iters=2, cn_sweeps=4),
            melt((12, 10, 8), 2, 1, hydro=1, ncg_iters=2, cn_sweeps=4),
            melt((300, 3, 4), 5, 3, hydro=1, ncg_iters=2, cn_sweeps=4)]
    states = [random_state(c, 80 + 3 * i) for i, c in enumerate(cfgs)]
    ctx = dscf.Context(cfgs, precision)
    dt = ctx.dtype
    for which, k in ((dscf.PHI, 0), (dscf.U, 1), (dscf.POP, 2)):
        ctx.set(which, torch.from_numpy(np.concatenate([s[k].ravel() for s in states])).to(dt).cuda())
    ctx.step(2)
    ctx.status()
    phi = t2n(ctx.get(dscf.PHI))
    off = 0
    for c, (p, U, dn) in zip(cfgs, states):
        solo = run_gpu(c, precision, p, U, dn, 2)
        assert np.array_equal(phi[off:off + p.size], solo["phi"].ravel())
        off += p.size


def test_static_density_map_at_its_scratch_limit():
    """A small grid with the longest chain that fits: few warps, an even cut."""
    grid = (16, 8, 16)
    cfg = melt(grid, 64 * 1024 * 1024 // (2048 * 8) - 7, 1000)   # 2048 sites of 8 bytes: N + 6 fields and tables
    U = inputs.random_field(ncomp_shape(cfg), seed=70, scale=0.01)
    ref, _, _ = oracle.densities(cfg, U)
    U = torch.from_numpy(U).cuda()
    got = t2n(dscf.densities_static(cfg, U, torch.empty_like(U)))
    assert rel(got, ref) < 1e-10      # the bound of a coupled FP64 step: 4089 contour steps


def test_bricks_that_do_not_run_together_take_the_general_sweeps():
    """256 shallow bricks: the tuning stays valid, the densities are those of the deep bricks."""
    cfg = melt((128, 128, 128), 3, 2)
    U = torch.from_numpy(inputs.random_field(ncomp_shape(cfg), seed=50, scale=0.5)).float().cuda()
    out = []
    for zc in (8, 16):
        ctx = dscf.Context(cfg, dscf.FP32, tuning=(zc, 0))
        assert ctx.diagnostics()["kfuse"] == 0 and ctx.diagnostics()["zc"] == zc
        out.append(t2n(ctx.densities(U)))
        ctx.status()
        ctx.close()
    assert rel(out[0], out[1]) < 1e-5


@pytest.mark.parametrize("grid", [(16, 3, 2), (48, 5, 3), (32, 1, 4), (112, 9, 1), (96, 4, 5)], ids=lambda g: "x".join(map(str, g)))
def test_mma_forward_on_ragged_blocks(grid):
    """Every convolution sum is exact; the means (sums / V, V not a power of two) are not: the kernel
    rounds phibar - <y> and its sum with y to FP32."""
    U, params = exact_problem(grid)
    ref, (_, _, _, y) = emulate_forward(params, U, [0.5, 0.5], grid)
    net = dscf.Net(grid, B, seed=1)
    net.set_params(torch.from_numpy(flat(params)).float())
    got = net.forward(torch.from_numpy(U).float(), [0.5, 0.5]).cpu().numpy().astype(np.float64)
    shift = np.abs(0.5 - y.mean(axis=(2, 3, 4), keepdims=True))
    assert np.all(np.abs(got - ref) <= 2.0 ** -24 * (shift + np.abs(ref)) * (1 + 2.0 ** -20))


@pytest.mark.parametrize("grid", [(16, 4, 2), (32, 16, 8), (64, 2, 16), (16, 1, 64)], ids=lambda g: "x".join(map(str, g)))
def test_weight_gradients_on_ragged_tiles(grid):
    U, params = exact_problem(grid)
    (W1, b1), (W2, b2), (W3, b3) = params
    phi, (x, h1, h2, y) = emulate_forward(params, U, [0.5, 0.5], grid)
    nx, ny, nz = grid
    V = nx * ny * nz
    t = np.stack([np.stack([paired_integers(V, 1, 7, 700 + 10 * b + c).reshape(nz, ny, nx) for c in range(2)])
                  for b in range(B)])
    t = (2 * t - np.sign(t)) / 16.0
    n = phi.size                              # a power of two: dy is exact in BF16
    dy = bf16(t / n)
    dW3, _, dh2 = oracle.conv3d_bwd(grid, B, W3, h2, dy)
    dz2 = bf16(dh2 * (1.0 - h2 * h2))
    dW2, _, dh1 = oracle.conv3d_bwd(grid, B, W2, h1, dz2)
    dz1 = bf16(dh1 * (1.0 - h1 * h1))
    dW1, _, _ = oracle.conv3d_bwd(grid, B, W1, x, dz1, want_din=False)
    aW2 = oracle.conv3d_bwd(grid, B, np.abs(W2), np.abs(h1), np.abs(dz2), want_din=False)[0]
    aW1 = oracle.conv3d_bwd(grid, B, np.abs(W1), np.abs(x), np.abs(dz1), want_din=False)[0]
    net = dscf.Net(grid, B, seed=1)
    net.set_params(torch.from_numpy(flat(params)).float())
    _, g = net.gradient(torch.from_numpy(U).float(), torch.from_numpy(phi - t).float(), [0.5, 0.5])
    (gW1, _), (gW2, _), (gW3, _) = dscf.net_params_split(g.cpu().numpy())
    assert np.array_equal(gW3, dW3) and np.abs(dW3).max() > 0
    for got, ref, a in ((gW2, dW2, aW2), (gW1, dW1, aW1)):
        assert np.all(np.abs(got - ref) <= B * V * 2.0 ** -22 * a)
        assert np.abs(ref).max() > 0


@pytest.mark.parametrize("shift", [1, 2, 3])
def test_potentials_at_any_element_of_an_allocation(shift):
    """A contiguous view may begin 4, 8 or 12 bytes into its allocation: same densities, bit for bit
    (a melt: per-site factors, no sum that the order of the threads' sites could change)."""
    cfg = melt((36, 6, 5), 5, 2)
    U = torch.from_numpy(inputs.random_field(ncomp_shape(cfg), seed=90, scale=0.5)).float().cuda()
    view = torch.empty(U.numel() + shift, device="cuda")[shift:].view(U.shape).copy_(U)
    assert view.is_contiguous() and view.data_ptr() % 16 == 4 * shift
    ctx = dscf.Context(cfg, dscf.FP32)
    assert torch.equal(ctx.densities(view), ctx.densities(U))
    ctx.status()
    out = [dscf.densities_static(cfg, u, torch.empty_like(U), dscf.FP32) for u in (view, U)]
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("a", [0.6, 1.1543, 1.5, 1.68])
@pytest.mark.parametrize("grid,ns", [((32, 32, 32), 2), ((30, 31, 33), 2), ((36, 28, 32), 3)], ids=["32", "odd", "solution"])
def test_densities_keep_their_means(grid, ns, a, precision):
    """The densities of a chain sum to phi_p whatever the Boltzmann factors.  Per site the sweeps' and the
    factor's roundings add up to some ulps of either sign, whose mean over 3e4 sites is below a tenth of an
    ulp; the bound, half an ulp of 1, leaves no room for a factor that is itself off by a rounding."""
    cfg = dict(melt(grid, 16, 7) if ns == 2 else solution(grid, 16, 7), a=a)
    U = torch.from_numpy(inputs.random_field(ncomp_shape(cfg), seed=95, scale=0.1))
    ctx = dscf.Context(cfg, precision, tuning=(8, 1))
    phi = t2n(ctx.densities(U))
    ctx.status()
    ctx.close()
    V = grid[0] * grid[1] * grid[2]
    ulp = 2.0 ** (-53 if precision == dscf.FP64 else -24)
    off = lambda f, mean: math.fsum(itertools.chain(f.ravel(), itertools.repeat(-mean, V))) / V   # one rounding
    assert abs(off(phi[:2], cfg["phi_p"])) < 0.5 * ulp
    if ns == 3:
        assert abs(off(phi[2], 1.0 - cfg["phi_p"])) < 0.5 * ulp


@pytest.mark.parametrize("grid", [(127, 127, 127), (33, 17, 9)], ids=["14 a thread", "1 a thread"])
def test_solvent_sum_keeps_every_term(grid):
    """Site counts that no vector access divides are summed in FP64, term by term: the mean of V equal
    FP32 factors is that factor."""
    cfg = solution(grid, 2, 1)
    ctx = dscf.Context(cfg, dscf.FP32, tuning=(8, 1))
    ctx.set(dscf.U, torch.full(ncomp_shape(cfg), 0.37))
    ctx.observables()               # evaluates the densities at U
    qs = ctx.diagnostics()["QS"]
    assert abs(qs - math.exp(-0.37)) < 1e-6
    assert abs(qs - float(np.float32(qs))) < 1e-12 * qs


@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("batch", [False, True], ids=["solo", "batch"])
@pytest.mark.parametrize("chain", [0, 1])
def test_general_sweeps_timeout_is_reported_and_the_context_recovers(chain, batch, precision):
    """Failure detection without a GPU fault: a chain's barrier counter is set far behind (host side), so
    no CTA ever sees the barrier complete; the bounded waits run out, the launch finishes, the host reads
    DSCF_ERR_TIMEOUT, and the counters are as before the launch."""
    cfgs = [melt((40, 30, 20), 9, 4), solution((33, 12, 10), 6, 3)] if batch else [melt((40, 30, 20), 9, 4)]
    U = np.concatenate([inputs.random_field(ncomp_shape(c), seed=97 + i, scale=0.5).ravel() for i, c in enumerate(cfgs)])
    ctx = dscf.Context(cfgs, precision, tuning=(8, 1))
    U = torch.from_numpy(U).to(ctx.dtype).cuda()
    good = ctx.densities(U)
    ctx.status()
    ctx.set_wait_limit(2000)
    ctx.inject_lag(chain)
    ctx.densities(U)
    with pytest.raises(dscf.DSCFError) as err:
        ctx.status()
    assert err.value.code == -4
    ctx.status()                    # re-armed by the call that reported the timeout
    for _ in range(2):
        assert torch.equal(ctx.densities(U), good)
    ctx.status()
    with pytest.raises(dscf.DSCFError):
        ctx.inject_lag(2)


@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
def test_general_sweeps_of_more_replicas_than_the_shared_table(precision):
    """130 replicas: the kernel reads its table from global memory.  Equal chains and two row layouts."""
    cfgs = [melt((6 + 27 * (i % 2), 5, 4), 3 + i % 3, 1 + i % 2) for i in range(130)]
    U = [inputs.random_field(ncomp_shape(c), seed=200 + i, scale=0.5) for i, c in enumerate(cfgs)]
    ref = np.concatenate([oracle.densities(c, u)[0].ravel() for c, u in zip(cfgs, U)])
    ctx = dscf.Context(cfgs, precision)
    for _ in range(2):
        got = t2n(ctx.densities(torch.from_numpy(np.concatenate([u.ravel() for u in U]))))
        ctx.status()
        assert rel(got, ref) < (1e-12 if precision == dscf.FP64 else 1e-5)


@pytest.mark.parametrize("grid", [(32, 256, 120), (64, 256, 136), (128, 128, 136), (96, 128, 120), (48, 128, 168), (64, 72, 136)],
                         ids=lambda g: "x".join(map(str, g)))
def test_bricks_of_eight_planes_beyond_the_sms(grid):
    """More bricks of 8 planes than SMs and nz an odd multiple of 8: bricks of 16, the uppermost of 8; the
    halo rows of every brick against the oracle, and the same bits every time."""
    for N, nA in ((2, 1), (5, 3)):
        cfg = melt(grid, N, nA)
        U = inputs.random_field(ncomp_shape(cfg), seed=98, scale=0.5)
        ref, _, _ = oracle.densities(cfg, U)
        ctx = dscf.Context(cfg, dscf.FP32, tuning=(8, 0))
        U = torch.from_numpy(U).float().cuda()
        first = ctx.densities(U)
        ctx.status()
        assert rel(t2n(first), ref) < 1e-5
        for _ in range(10):
            assert torch.equal(ctx.densities(U), first)
        ctx.status()
        ctx.close()


def test_bricks_of_eight_planes_beyond_the_sms_in_a_batch():
    """Replicas of several widths, heights and depths: each as alone."""
    cfgs = [melt((64, 256, 136), 4, 2), melt((48, 128, 24), 5, 2), melt((64, 64, 40), 4, 1), solution((128, 16, 16), 6, 3)]
    U = [torch.from_numpy(inputs.random_field(ncomp_shape(c), seed=300 + i, scale=0.5)).float().cuda() for i, c in enumerate(cfgs)]
    ctx = dscf.Context(cfgs, dscf.FP32, tuning=(8, 0))
    got = t2n(ctx.densities(torch.cat([u.reshape(-1) for u in U])))
    ctx.status()
    off = 0
    for c, u in zip(cfgs, U):
        solo = dscf.Context(c, dscf.FP32, tuning=(8, 0))
        assert rel(got[off:off + u.numel()], t2n(solo.densities(u)).ravel()) < 1e-6
        off += u.numel()
        solo.close()


@pytest.mark.parametrize("short", [1e-15, 1e-13, 1e-11, 1e-8, 1e-4])
@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
def test_segments_up_to_the_longest(short, precision):
    """alpha = a^2 / 6 just below 1/2, where the stencil's centre weight vanishes."""
    a = math.sqrt(3.0) * (1.0 - short)
    for cfg, tunings in ((melt((34, 7, 6), 6, 2), [(8, 1)]), (melt((32, 16, 16), 70, 30), [(8, 1), (16, 0)])):
        for tuning in tunings[:1 if precision == dscf.FP64 else 2]:
            check_densities(dict(cfg, a=a), precision, 99, tuning=tuning)


@pytest.mark.parametrize("precision", [dscf.FP64, dscf.FP32], ids=["fp64", "fp32"])
def test_general_sweeps_of_hundreds_of_replicas(precision):
    """Chains of five lengths: the CTAs' parts of the table move as chains end.  Sampled replicas bit for bit as
    alone."""
    cfgs = [melt((3 + 7 * (i % 5), 2 + i % 3, 3 + i % 4), 2 + i % 5, 1 + i % 2 * (i % 5 > 0)) for i in range(330)]
    U = [inputs.random_field(ncomp_shape(c), seed=400 + i, scale=0.5) for i, c in enumerate(cfgs)]
    ref = np.concatenate([oracle.densities(c, u)[0].ravel() for c, u in zip(cfgs, U)])
    ctx = dscf.Context(cfgs, precision)
    flat = torch.from_numpy(np.concatenate([u.ravel() for u in U])).to(ctx.dtype).cuda()
    got = ctx.densities(flat)
    ctx.status()
    assert rel(t2n(got), ref) < (1e-12 if precision == dscf.FP64 else 1e-5)
    at = np.cumsum([0] + [u.size for u in U])
    for i in (0, 1, 4, 127, 128, 200, 329):
        solo = dscf.Context(cfgs[i], precision).densities(torch.from_numpy(U[i]))
        assert torch.equal(got[at[i]:at[i + 1]], solo.reshape(-1))


@pytest.mark.parametrize("a", [0.6, 1.0, 1.1543, 1.5])
@pytest.mark.parametrize("N", [8, 20, 64])
@pytest.mark.parametrize("total", [-78.0, 78.0])
def test_fp32_potentials_of_any_gauge(total, N, a):
    """A constant added to both potentials does not change the densities, also where exp(-N U) comes within a few
    units of FP32's limits: the sweeps' own scale takes little of the range.  The bound allows for the rounding
    of the shifted potentials: N half ulps of |total| / N + |U|."""
    cfg = dict(melt((34, 10, 9), N, N // 3), a=a)
    U = inputs.random_field(ncomp_shape(cfg), seed=96, scale=0.5 / N)
    ref, _, _ = oracle.densities(cfg, U)
    ctx = dscf.Context(cfg, dscf.FP32, tuning=(8, 1))
    got = t2n(ctx.densities(torch.from_numpy(U + total / N)))
    ctx.status()
    assert rel(got, ref) < 1e-5 + abs(total) * 2.0 ** -23
