"""Device paths at the sizes where they can go wrong: tails of buffers, edges
of tiles and of the division of the work, odd and smallest grids."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
SEED = 2110144940


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_14494_gb300 import build
    build.build()


def _dirty(value):
    """Leaves value in the allocator's free blocks, which the next workspace takes."""
    x = [torch.full((1 << 20,), value, dtype=torch.float32, device="cuda") for _ in range(16)]
    torch.cuda.synchronize()
    del x


@pytest.mark.parametrize("shape", [(21, 19, 23), (16, 12, 20), (7, 5, 9)])
def test_coupled_start_does_not_depend_on_memory(shape):
    """The low halves of the float-pair potential start at zero over their whole
    length, also where the cell count leaves them off the end of ncell doubles."""
    from paper_2110_14494_gb300 import PicContext
    grid = W.grid_spec(*shape, 5e-5)
    n = shape[0] * shape[1] * shape[2]
    phis = []
    for value in (0.0, 1.0e3):
        _dirty(value)
        ctx = PicContext(W.synthetic_air(), grid, precision=32, capacity=1024, seed=SEED, dt=1e-12, coupled=True,
                         v_lo=0.0, v_hi=2000.0, v_mask=0.0, poisson_rtol=1e-6, poisson_max_cycles=1000)
        ctx.step(1)
        blob = ctx.save()
        phis.append(np.frombuffer(blob, np.float64, count=n, offset=len(blob) - 8 * n))
    assert np.array_equal(phis[0], phis[1])


def _solve_noalloc(P, pc, rho, phi, mask, rtol, cycles):
    import ctypes as C
    st = P.poisson_stats()
    s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = P.lib().poisson_solve_noalloc(C.byref(pc), C.c_void_p(rho.data_ptr()), C.c_void_p(mask.data_ptr()),
                                       C.c_void_p(phi.data_ptr()), None, None, None, rtol, cycles, C.byref(st), s)
    torch.cuda.synchronize()
    return rc, st


@pytest.mark.parametrize("shape", [(2, 2, 2), (3, 7, 5), (4, 6, 10), (33, 6, 10), (16, 16, 16), (20, 20, 20),
                                   (26, 28, 8), (16, 16, 32), (4, 64, 32), (36, 48, 40), (64, 32, 6)])
def test_float64_solve_at_block_and_level_edges(shape):
    """Float64 CG and the one-block small levels: grids below and beside the
    blocks' 32 x 4 x 4 cells, one to four cells of a colour a thread, single
    levels, scattered electrode cells.  The fixed-scratch solve forms A z anew
    and takes the plain kernel for the small levels, operation by operation the
    same, so its bits are equal; against the oracle both residuals are below
    1e-11, times a condition number below 1e3 for these grids."""
    from paper_2110_14494_gb300 import picmcc as P
    grid = W.grid_spec(*shape, 4e-5)
    nz, ny, nx = shape[2], shape[1], shape[0]
    rng = np.random.default_rng(nx * 10007 + ny * 101 + nz)
    mask = (rng.random((nz, ny, nx)) < 0.04).astype(np.uint8)
    rho = rng.uniform(-5e-2, 5e-2, (nz, ny, nx))
    ref, _, _ = O.poisson(grid, rho, mask, 700.0, -100.0, 1500.0, rtol=1e-12)
    drho, dmask = torch.as_tensor(rho).cuda(), torch.as_tensor(mask).cuda()
    phi, phi2 = torch.zeros_like(drho), torch.zeros_like(drho)
    cyc, rel = P.poisson_solve(grid, drho, phi, mask=dmask, v_lo=-100.0, v_hi=1500.0, v_mask=700.0, rtol=1e-11,
                               max_cycles=500, precision=64)
    assert rel <= 1e-11
    pc = P.poisson_config(nx, ny, nz, 4e-5, -100.0, 1500.0, 700.0, 64)
    rc, st = _solve_noalloc(P, pc, drho, phi2, dmask, 1e-11, 500)
    assert rc == P.PIC_OK and st.cycles == cyc and torch.equal(phi, phi2)
    assert np.linalg.norm(phi.cpu().numpy() - ref) <= 1e-8 * np.linalg.norm(ref)


@pytest.mark.parametrize("n0,launch", [(1, 0), (33, 1), (33, 2), (700, 0), (700, 1), (700, 2)])
def test_batched_products_through_warp_and_global_queues(n0, launch):
    """Many ionizations a step (2.6 electrons for one after 2 ps at 900 Td): products wait in the
    warp's queue, what it cannot hold goes to the global one.  Each swarm is the
    oracle's run: counts equal, moments to 1e-9 as elsewhere for float64."""
    from paper_2110_14494_gb300 import swarm_run
    gas, seed, ENs = W.synthetic_air(), 31, [900.0, 600.0]
    res, mom, cnt = swarm_run(gas, ENs, precision=64, n0=n0, n_steps=6, dt=2e-12, seed=seed, n_lo=1, n_hi=100000,
                              want_moments=True, batched=True, block=128, blocks_per_sm=1, use_graph=launch)
    for s, EN in enumerate(ENs):
        omom, ocnt, _, _ = O.swarm(gas, EN, n0, 6, 2e-12, seed + s, n_lo=1, n_hi=100000)
        assert np.array_equal(cnt[s], ocnt), s
        scale = np.abs(omom).max(axis=0) + 1e-300
        assert np.all(np.abs(mom[s] - omom) <= 1e-9 * scale), s


@pytest.mark.parametrize("n", [64, 128, 192, 256, 512, 2304])
def test_training_pass_by_cluster_size(n):
    """One to four blocks a cluster, one and several clusters: the gradient
    against FP64 within the bound of BF16 products, and three steps in one call
    equal, bit by bit, to three calls of one step."""
    from paper_2110_14494_gb300 import mlp_loss_grad, mlp_train
    from tests import test_gpu_mlp as G
    th, x, t = G._problem(n, seed=n)
    p0, xd, td = G._dev(th), G._dev(x), G._dev(t)
    loss, g = mlp_loss_grad(p0, xd, td)
    th2 = G._w2_as_multiplied(th)
    lref, gref = G.M.loss_grad(th2, x, t)
    assert abs(loss.item() - lref) <= 1e-2 * lref
    assert np.all(np.abs(g.cpu().numpy().astype(np.float64) - gref) <= G._grad_bound(th2, x, t))
    runs = []
    for calls in ([(0, 3)], [(0, 1), (1, 1), (2, 1)]):
        p, m, v = p0.clone(), torch.zeros_like(p0), torch.zeros_like(p0)
        for step0, k in calls:
            l = mlp_train(p, m, v, step0, xd, td, k)
        runs.append((p, m, v, l))
    assert all(torch.equal(a, b) for a, b in zip(*runs))


@pytest.mark.parametrize("n", [1, 129, 128 * 152 + 1, 4 * 128 * 152 - 1, 4 * 128 * 152 + 129])
def test_queries_do_not_depend_on_their_tile(n):
    """Ragged tiles, idle groups of a block, one and two tiles a group: each
    point's outputs are, bit by bit, those of the same point in calls of 1000."""
    from paper_2110_14494_gb300 import mlp_forward
    from tests import test_gpu_mlp as G
    th, x, _ = G._problem(n, seed=5)
    p, xd = G._dev(th), G._dev(x)
    y = mlp_forward(p, xd)
    assert torch.equal(y, torch.cat([mlp_forward(p, xd[k:k + 1000].contiguous()) for k in range(0, n, 1000)]))


@pytest.mark.parametrize("shape,cycles,pair", [((132, 92, 92), 24, (16, 8.340650992245674e-07)),
                                               ((68, 132, 124), 25, (17, 6.384658163628055e-07)),
                                               ((64, 128, 132), 25, (17, 6.774815300983311e-07)),
                                               ((516, 44, 52), 22, (15, 5.360662387261354e-07))])
def test_large_level_sweeps_on_ragged_tiles(shape, cycles, pair):
    """Levels of 2^20 cells and more (pairs of cells, four planes a thread):
    widths that end inside a warp, rows that end inside a block, scattered
    electrode cells.  The float64 solve's residual, formed here, is what the
    solve reports; the iterations of both solves and the residual of the
    float-pair solve (deterministic sums) are those of sweeps with one thread a
    cell and its six neighbours loaded, recorded once, bit by bit."""
    from paper_2110_14494_gb300 import picmcc as P
    nx, ny, nz = shape
    grid = W.grid_spec(nx, ny, nz, 4e-5)
    rng = np.random.default_rng(nx)
    mask = (rng.random((nz, ny, nx)) < 0.002).astype(np.uint8)
    rho = rng.uniform(-5e-2, 5e-2, (nz, ny, nx))
    vm, lo, hi = 700.0, -100.0, 1500.0
    dphi = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
    cyc, rel = P.poisson_solve(grid, torch.as_tensor(rho).cuda(), dphi, mask=torch.as_tensor(mask).cuda(), v_lo=lo,
                               v_hi=hi, v_mask=vm, rtol=1e-9, max_cycles=40, precision=64)
    f = dphi.cpu().numpy()
    f[mask != 0] = vm
    p = np.pad(f, 1, mode="edge")
    p[0, 1:-1, 1:-1], p[-1, 1:-1, 1:-1] = 2 * lo - f[0], 2 * hi - f[-1]
    nb = (p[1:-1, 1:-1, :-2] + p[1:-1, 1:-1, 2:] + p[1:-1, :-2, 1:-1] + p[1:-1, 2:, 1:-1] + p[:-2, 1:-1, 1:-1]
          + p[2:, 1:-1, 1:-1])
    h2e = 4e-5 ** 2 / 8.8541878128e-12
    q = np.pad(np.where(mask, vm, 0.0), 1)
    b = h2e * rho + (q[1:-1, 1:-1, :-2] + q[1:-1, 1:-1, 2:] + q[1:-1, :-2, 1:-1] + q[1:-1, 2:, 1:-1]
                     + q[:-2, 1:-1, 1:-1] + q[2:, 1:-1, 1:-1])
    b[0] += 2 * lo
    b[-1] += 2 * hi
    free = mask == 0
    r = (h2e * rho + nb - 6.0 * f)[free]
    res = np.linalg.norm(r) / np.linalg.norm(b[free])
    assert rel <= 1e-9 and abs(res - rel) <= 1e-3 * rel + 1e-13
    assert cyc == cycles
    dphi.zero_()
    assert P.poisson_solve(grid, torch.as_tensor(rho).cuda(), dphi, mask=torch.as_tensor(mask).cuda(), v_lo=lo, v_hi=hi,
                           v_mask=vm, rtol=1e-6, max_cycles=40, precision=32) == pair


def _push_case(n, prec, steps):
    """n electrons by the device and by the oracle: (common, only device, only oracle, outside, worst)."""
    from paper_2110_14494_gb300 import PicContext
    from tests import test_gpu_pic as G
    from tests.gpu_common import compare_sets
    gas, F, mk, p0 = G._setup(n, prec, 11)
    dt, cap = 2e-12, 8 * n + 4096
    ctx = PicContext(gas, G.GRID, precision=prec, capacity=cap, seed=SEED, dt=dt, mask=mk)
    ctx.set_field(*G._field_dev(F))
    ctx.set_particles(p0)
    ctx.step(steps)
    m = O.Model(gas, dt, SEED, prec, G.GRID, F, mask=mk)
    P = O.Particles(cap, p0)
    nc = G.GRID["nx"] * G.GRID["ny"] * G.GRID["nz"]
    rq = [np.zeros(nc, np.int64) for _ in range(2)]
    for s in range(1, steps + 1):
        rc, _ = O.step(m, P, s, s == 1, np.zeros(nc, np.int64), *rq)
        assert rc == 0
    return compare_sets(ctx.get_particles(), P.view(), G.GRID["dx"], 1e-12 if prec == 64 else 1e-3, v_floor=1.0)


@pytest.mark.parametrize("n", [2, 31, 32, 64, 65, 32 * 152, 32 * 152 + 1, 8 * 32 * 152 + 77])
def test_pool_of_electrons_at_its_edges(n):
    """Double precision: warps with one electron to a full pool, ranges that end
    inside a warp, items beyond the first ranges; particle by particle to 1e-12,
    as elsewhere for float64."""
    nc, og, orf, bad, worst = _push_case(n, 64, 2)
    assert og == 0 and orf == 0 and bad == 0, (og, orf, worst)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 33, 4096, 24 * 3648 - 1, 24 * 3648 + 1])
def test_electrons_by_place_at_range_edges(n):
    """Single precision: ranges of 8, 16, 24 and 32 electrons and their last
    ones.  Decision flips (gross differences) at most 1e-5 of the particles plus
    two, as elsewhere for float32."""
    nc, og, orf, bad, worst = _push_case(n, 32, 1)
    assert nc >= n * 0.9 and og + orf + worst["gross"] <= 1e-5 * nc + 2, (og, orf, worst)


@pytest.mark.parametrize("shape", [(2, 2, 2), (33, 6, 10), (35, 9, 13), (20, 20, 20), (64, 48, 40), (100, 20, 36)])
def test_pair_solve_and_field_at_block_edges(shape):
    """Float-pair residual and field: grids whose rows end inside a warp, whose
    rows and planes end inside a block, planes at the plates and those between,
    with and without electrode cells.  The potential is the oracle's; the field
    is the centred difference of that potential, whose pair difference and scaling
    round three times (2e-7), the pair itself to 2^-47."""
    from paper_2110_14494_gb300 import picmcc as P
    nx, ny, nz = shape
    h, lo, hi, vm = 4e-5, -100.0, 1500.0, 700.0
    grid = W.grid_spec(nx, ny, nz, h)
    rng = np.random.default_rng(nx + ny)
    rho = rng.uniform(-5e-2, 5e-2, (nz, ny, nx))
    for density in (0.0, 0.03):
        mask = (rng.random((nz, ny, nx)) < density).astype(np.uint8)
        ref, _, _ = O.poisson(grid, rho, mask, vm, lo, hi, rtol=1e-12)
        phi = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
        E = tuple(torch.zeros((nz, ny, nx), dtype=torch.float32, device="cuda") for _ in range(3))
        P.poisson_solve(grid, torch.as_tensor(rho).cuda(), phi, mask=torch.as_tensor(mask).cuda(), E=E, v_lo=lo, v_hi=hi,
                        v_mask=vm, rtol=1e-8, max_cycles=500, precision=32)
        f = phi.cpu().numpy()
        assert np.linalg.norm(f - ref) <= 1e-5 * np.linalg.norm(ref)
        p = np.pad(f, 1, mode="edge")
        p[0, 1:-1, 1:-1], p[-1, 1:-1, 1:-1] = 2 * lo - f[0], 2 * hi - f[-1]
        want = (-(p[1:-1, 1:-1, 2:] - p[1:-1, 1:-1, :-2]) / (2 * h), -(p[1:-1, 2:, 1:-1] - p[1:-1, :-2, 1:-1]) / (2 * h),
                -(p[2:, 1:-1, 1:-1] - p[:-2, 1:-1, 1:-1]) / (2 * h))
        for e, w in zip(E, want):
            assert np.all(np.abs(e.cpu().numpy() - w) <= 5e-7 * np.abs(w) + 2.0 ** -44 * np.abs(f).max() / h)


@pytest.mark.parametrize("shape", [(2, 2, 2), (13, 17, 31), (16, 16, 32), (264, 256, 256)])
def test_weight_update_on_grids_around_the_scan_tiles(shape):
    """The cell scan's tiles of 2048 and its second level's 8192 tiles: fewer
    cells than a thread's eight, a ragged last tile, whole tiles, more than 8192
    tiles; cells with thousands of electrons beside empty ones.  The merged and
    split set is the oracle's, bit for bit."""
    from paper_2110_14494_gb300 import PicContext
    from tests.gpu_common import by_id
    grid = W.grid_spec(*shape, 1e-4)
    p0 = W.random_particles(6000, grid, 51, w_range=(1.0, 3.0))
    for k in ("x", "y", "z"):  # half of them in the first and the last cells
        p0[k][:2000] = np.float32(0.5e-4)
        p0[k][2000:3000] = np.float32((dict(x=shape[0], y=shape[1], z=shape[2])[k] - 0.5) * 1e-4)
    gas = W.synthetic_air()
    ctx = PicContext(gas, grid, precision=32, capacity=40000, seed=SEED, dt=1e-12, n_ppc=10, w_min=1.0, particle_cap=0)
    ctx.set_particles(p0)
    ctx.weight_update()
    gpu = by_id(ctx.get_particles())
    P = O.Particles(40000, p0)
    rc, _ = O.merge_split(O.Model(gas, 1e-12, SEED, 32, grid), P, 0, n_ppc=10, w_min=1.0, cap=0)
    ref = by_id(P.view())
    assert rc == 0 and len(ref["id"]) != len(p0["id"])
    assert np.array_equal(gpu["id"], ref["id"])
    for k in ("x", "y", "z", "vx", "vy", "vz", "w"):
        assert np.array_equal(gpu[k], ref[k]), k


@pytest.mark.parametrize("n", [1, 3, (1 << 18) - 1, 1 << 18, (1 << 18) + 3])
def test_features_of_aligned_and_shifted_arrays(n):
    """Four points a thread, with a remainder, and one a thread (few points, or
    arrays that begin eight bytes off a 16-byte boundary): the same bits; and
    log10 of the float32 value to 2 units in the last place, its stated error."""
    from paper_2110_14494_gb300 import mlp_features
    rng = np.random.default_rng(n)
    en = torch.as_tensor(10 ** rng.uniform(0, 3.5, n + 1)).cuda()
    f = torch.as_tensor(rng.uniform(0, 1, n + 1)).cuda()
    shifted = mlp_features(en[1:], f[1:])
    aligned = mlp_features(en[1:].clone(), f[1:].clone())
    assert torch.equal(shifted, aligned)
    ref = np.log10(en[1:].cpu().numpy().astype(np.float32).astype(np.float64))
    x = aligned.cpu().numpy()
    assert np.all(np.abs(x[:, 0] - ref) <= 2 * np.spacing(np.abs(ref).astype(np.float32)))
    assert np.array_equal(x[:, 1], f[1:].cpu().numpy().astype(np.float32))


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("n_lo,n_hi", [(995, 5000), (10, 1005)])
def test_swarm_resampled_within_a_step(prec, n_lo, n_hi):
    """A single swarm that falls below n_lo (attachment at 25 Td) is doubled and
    one that rises above n_hi (ionization at 400 Td) thinned at the start of a
    step, and the step's electrons are those: float64 counts are the oracle's,
    float32 counts the same but for decision flips (two of a thousand)."""
    from paper_2110_14494_gb300 import swarm_run
    gas, EN = W.synthetic_air(), 25.0 if n_lo > 100 else 400.0
    _, mom, cnt = swarm_run(gas, [EN], precision=prec, n0=1000, n_steps=120, dt=2e-12, seed=77, n_lo=n_lo, n_hi=n_hi,
                            want_moments=True)
    omom, ocnt, _, _ = O.swarm(gas, EN, 1000, 120, 2e-12, 77, n_lo=n_lo, n_hi=n_hi)
    jumps = np.abs(np.diff(ocnt)) > 0.3 * ocnt[:-1]
    assert jumps.any()
    if prec == 64:
        assert np.array_equal(cnt[0], ocnt)
        assert np.all(np.abs(mom[0] - omom) <= 1e-9 * (np.abs(omom).max(axis=0) + 1e-300))
    else:
        k = int(np.argmax(jumps)) + 1
        assert np.all(np.abs(cnt[0][:k + 1] - ocnt[:k + 1]) <= 2e-3 * ocnt[:k + 1] + 2)


@pytest.mark.parametrize("launch", [1, 2])
@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("n_bins", [3, 11, 1001])
def test_batched_tables_of_odd_length(n_bins, prec, launch):
    """Gas tables with an odd number of nodes, three swarms (the second table
    begins 40 n_bins bytes after the first in float32, 8 modulo 16 unless the
    stride is rounded up).  Float64 counts are the oracle's; in float32 a
    rounding turns about 1e-6 of the decisions, some 10 draws a picosecond for
    20 ps: 2e-4 of the electrons; at most two in a thousand and two here."""
    from paper_2110_14494_gb300 import swarm_run
    gas, seed, ENs = W.synthetic_air(n_bins=n_bins), 91, [150.0, 250.0, 120.0]
    _, mom, cnt = swarm_run(gas, ENs, precision=prec, n0=1000, n_steps=20, dt=1e-12, seed=seed, n_lo=10, n_hi=100000,
                            want_moments=True, batched=True, block=128, blocks_per_sm=1, use_graph=launch)
    for s, EN in enumerate(ENs):
        omom, ocnt, _, _ = O.swarm(gas, EN, 1000, 20, 1e-12, seed + s, n_lo=10, n_hi=100000)
        if prec == 64:
            assert np.array_equal(cnt[s], ocnt), s
            assert np.all(np.abs(mom[s] - omom) <= 1e-9 * (np.abs(omom).max(axis=0) + 1e-300)), s
        else:
            assert np.all(np.abs(cnt[s] - ocnt) <= 2e-3 * ocnt + 2), s


def _in_two_threads(jobs, reps):
    """Runs each job reps times on a thread and stream of its own: lists of results, errors raised."""
    import threading
    out, errs = [[] for _ in jobs], []

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(reps):
                try:
                    out[k].append(jobs[k]())
                except Exception as e:  # noqa: BLE001
                    errs.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    return out, errs


@pytest.mark.parametrize("prec", [64, 32])
def test_solves_on_two_threads(prec):
    """Small levels of 91 and 72 KB of shared memory in solves that run side by
    side: the limit that a launch needs is not lowered by the other thread, and
    both get the bits of a solve that runs alone (deterministic sums)."""
    from paper_2110_14494_gb300 import poisson_solve

    def job(nx, ny, nz):
        rho = torch.as_tensor(np.random.default_rng(nx).uniform(-5e-2, 5e-2, (nz, ny, nx))).cuda()
        torch.cuda.synchronize()

        def solve():
            phi = torch.zeros_like(rho)
            poisson_solve(W.grid_spec(nx, ny, nz, 4e-5), rho, phi, v_hi=1500.0, rtol=1e-6, max_cycles=100, precision=prec)
            return phi
        return solve

    jobs = [job(20, 20, 20), job(24, 16, 16)]
    alone = [j() for j in jobs]
    torch.cuda.synchronize()
    out, errs = _in_two_threads(jobs, 200)
    assert not errs, errs[0]
    for got, want in zip(out, alone):
        assert len(got) == 200 and all(torch.equal(g, want) for g in got)


def test_batched_swarms_on_two_threads():
    """Blocks of 256 and of 64 threads (106 and 27 KB of shared memory) side by
    side: counts of every step as of a run alone."""
    from paper_2110_14494_gb300 import swarm_run
    gas = W.synthetic_air()
    jobs = [lambda b=b: swarm_run(gas, [120.0, 200.0], precision=64, n0=300, n_steps=4, dt=1e-12, seed=3, n_lo=10,
                                  n_hi=10000, want_moments=True, batched=True, block=b, blocks_per_sm=1, use_graph=1)[2]
            for b in (256, 64)]
    alone = [j() for j in jobs]
    out, errs = _in_two_threads(jobs, 40)
    assert not errs, errs[0]
    for got, want in zip(out, alone):
        assert len(got) == 40 and all(np.array_equal(g, want) for g in got)


@pytest.mark.parametrize("n,in_stated", [(88, True), (96, False), (100, True)])
def test_float64_solve_uses_the_room_it_is_given(n, in_stated):
    """A z is kept in the last n^3 doubles of a workspace that has room for
    them (which 96^3 is stated without) and formed again in one that has not;
    the fixed scratch has room at 88^3, none at 96^3: the same bits."""
    import ctypes as C
    from paper_2110_14494_gb300 import picmcc as P
    rho = torch.as_tensor(np.random.default_rng(n).uniform(-5e-2, 5e-2, (n, n, n))).cuda()
    pc = P.poisson_config(n, n, n, 4e-5, 0.0, 1500.0, 0.0, 64)
    stated = P.lib().poisson_workspace_bytes(C.byref(pc))
    az = (8 * n ** 3 + 255) // 256 * 256
    full = stated if in_stated else stated + az
    assert P._poisson_bytes(pc) >= full

    def solve(nb):
        ws, ptr = P._workspace(full)
        ws.fill_(0xA5)
        phi, st = torch.zeros_like(rho), P.poisson_stats()
        rc = P.lib().poisson_solve(C.byref(pc), C.c_void_p(rho.data_ptr()), None, C.c_void_p(phi.data_ptr()), None, None,
                                   None, 1e-10, 100, C.c_void_p(ptr), nb, C.byref(st), P._stream())
        torch.cuda.synchronize()
        assert rc == P.PIC_OK
        off = ptr - ws.data_ptr() + full - az
        return phi, bool((ws[off:off + 8 * n ** 3] != 0xA5).any())

    phi, kept = solve(full)
    assert kept
    if not in_stated:
        less, kept = solve(stated)
        assert not kept and torch.equal(less, phi)
    phi2 = torch.zeros_like(rho)
    rc, _ = _solve_noalloc(P, pc, rho, phi2, torch.zeros((n, n, n), dtype=torch.uint8, device="cuda"), 1e-10, 100)
    assert rc == (P.PIC_OK if n <= 96 else P.PIC_ERR_CAPACITY)
    assert n > 96 or torch.equal(phi2, phi)


def _solve_and_residual(shape, rtol):
    """A float64 solve with scattered electrode cells: the relative residual
    that it reports, the one of the potential that it returns, and what the
    rounding of that potential and of this sum can make of it (its differences
    at seven places, 2^-53 each, thrice)."""
    from paper_2110_14494_gb300 import poisson_solve
    nx, ny, nz = shape
    h, lo, hi, vm = 4e-5, -100.0, 1500.0, 700.0
    g = torch.Generator(device="cuda").manual_seed(nx)
    rho = 1e-1 * torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64) - 5e-2
    mask = torch.rand((nz, ny, nx), generator=g, device="cuda") < 0.002
    phi = torch.zeros_like(rho)
    _, rel = poisson_solve(W.grid_spec(nx, ny, nz, h), rho, phi, mask=mask.to(torch.uint8), v_lo=lo, v_hi=hi, v_mask=vm,
                           rtol=rtol, max_cycles=60, precision=64)
    assert torch.equal(phi[mask], torch.full_like(phi[mask], vm))

    def faces(u, low, high):
        """Sum of the values beyond the six faces less six times the cell's, no difference at the mirrors."""
        s = torch.zeros_like(u)
        for d in (2, 1, 0):
            n = u.shape[d]
            step = u.narrow(d, 1, n - 1) - u.narrow(d, 0, n - 1)
            s.narrow(d, 0, n - 1).add_(step)
            s.narrow(d, 1, n - 1).sub_(step)
        s[0] += 2.0 * (low - u[0])
        s[-1] += 2.0 * (high - u[-1])
        return s

    h2r = h * h / 8.8541878128e-12 * rho
    held = torch.where(mask, torch.full_like(phi, vm), torch.zeros_like(phi))
    b = h2r + faces(held, lo, hi)
    norm = b[~mask].norm()
    return rel, ((h2r + faces(phi, lo, hi))[~mask].norm() / norm).item(), 21 * 2.0 ** -53 * (phi.norm() / norm).item()


@pytest.mark.parametrize("shape", [(96, 64, 100), (96, 96, 96), (160, 144, 72), (512, 128, 240)])
def test_float64_solve_with_several_slabs_a_block(shape):
    """Blocks of the CG kernels that walk 2, 3, 3 and 8 slabs of planes, the
    last ones fewer: the residual that the solve reports (its sums over all
    slabs) is the one of the potential it returns."""
    rel, res, noise = _solve_and_residual(shape, 1e-9)
    assert rel <= 1e-9 and abs(res - rel) <= 1e-3 * rel + noise, (rel, res, noise)


@pytest.mark.parametrize("shape", [(16, 16, 16), (33, 6, 10), (64, 48, 80), (128, 64, 96)])
@pytest.mark.parametrize("rtol", [1e-11, 1e-13, 1e-14])
def test_float64_residual_stays_the_true_one(shape, rtol):
    """The CG's residual and q = A p follow from recurrences: they have not
    drifted from the potential's own residual where its rounding leaves one."""
    rel, res, noise = _solve_and_residual(shape, rtol)
    assert rel <= rtol and abs(res - rel) <= 1e-2 * rel + noise, (rel, res, noise)


@pytest.mark.parametrize("prec", [64, 32])
def test_weight_update_around_the_electrons_of_a_warp(prec):
    """Cells of 1 to 300 electrons, 31, 32, 33, 128 and 129 among them (one
    electron a lane, four, and more), beside empty ones: the merged and split
    set is the oracle's, bit for bit."""
    from paper_2110_14494_gb300 import PicContext
    from tests.gpu_common import by_id
    grid = W.grid_spec(9, 7, 8, 1e-4)
    counts = [1, 2, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 161, 256, 257, 300]
    p0 = W.random_particles(sum(counts), grid, 61, w_range=(1.0, 40.0))
    cells = np.repeat(5 + 17 * np.arange(len(counts)), counts)  # every 17th cell
    for k, i in (("x", cells % 9), ("y", cells // 9 % 7), ("z", cells // 63)):
        p0[k][:] = (1e-4 * (i + 0.25 + 0.5 * (p0[k] / (1e-4 * grid["n" + k])))).astype(np.float32)
    gas = W.synthetic_air()
    ctx = PicContext(gas, grid, precision=prec, capacity=20000, seed=SEED, dt=1e-12, n_ppc=40, w_min=1.0, particle_cap=0)
    ctx.set_particles(p0)
    ctx.weight_update()
    gpu = by_id(ctx.get_particles())
    P = O.Particles(20000, p0)
    rc, _ = O.merge_split(O.Model(gas, 1e-12, SEED, prec, grid), P, 0, n_ppc=40, w_min=1.0, cap=0)
    ref = by_id(P.view())
    assert rc == 0 and len(ref["id"]) != len(p0["id"])
    assert np.array_equal(gpu["id"], ref["id"])
    for k in ("x", "y", "z", "vx", "vy", "vz", "w"):
        assert np.array_equal(gpu[k], ref[k]), k
