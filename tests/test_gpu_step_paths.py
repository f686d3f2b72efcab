"""Forward-step kernels at the sizes where their dispatch or tiling changes, against the oracle."""
import numpy as np
import pytest

from paper_2605_27004_gb300 import inputs
from gpu_util import gpu_run, oracle_run, perm_lib_to_oracle, rand_theta, rel_l2

pytestmark = pytest.mark.gpu


# FP64 steps run blocks of one warp (rows of 1, 31, 32, 33, 65 cells: remainders of a warp; 70,001 rows:
# more than such blocks can cover in grid.y), and D2Q9 boxes of up to 4,864 cells four lanes per cell
# (7 and 260 cells: a last warp of seven cells and of four; 97 x 51 is past that size). Per step the collision
# rounds each population to about 10 * 2^-53 of f <= 0.5, so 20 steps stay below 1e-13.
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("q,dims", [(9, (1, 7, 1)), (9, (31, 9, 1)), (9, (65, 4, 1)), (9, (97, 51, 1)), (9, (2, 70001, 1)),
                                    (19, (33, 3, 5)), (19, (32, 4, 2)), (27, (65, 2, 3))])
def test_fp64_step_block_edges(q, dims, scheme):
    d, N = (2 if q == 9 else 3), int(np.prod(dims))
    Th = rand_theta(5, d)
    rho0, u0 = inputs.noise_field(N, d, 0.05, 6, rho_amp=0.02)
    g = gpu_run(q, dims, 0.8, Th, rho0, u0, 20, storage="fp64", scheme=scheme)
    o = oracle_run(q, dims, 0.8, Th, rho0, u0, 20)
    assert np.abs(g["f"] - o["f"][:, perm_lib_to_oracle(q)].T).max() < 1e-13


# FP64 storage conserves mass and momentum over long runs. A step rounds each stored population once, by at
# most 2^-54 of f <= 0.5 with either sign: over 10,000 steps and 19 populations some 1e-15 of the
# mass if no two cells shared their errors, and less once the decaying flow repeats itself. The bound
# of 1e-14 leaves room for that, while an error of one rounding of the density that comes back every step
# (1e-16) reaches 1e-12. D2Q9 with four lanes and one lane per cell, walls, both schemes.
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("q,dims,tau,frac", [(9, (16, 12, 1), 0.6, 0.0), (9, (97, 51, 1), 0.6, 0.0), (9, (33, 20, 1), 0.7, 0.2),
                                             (19, (8, 7, 6), 0.6, 0.0), (19, (33, 6, 5), 0.55, 0.0), (27, (8, 7, 6), 0.7, 0.2)])
def test_fp64_conserves_mass_and_momentum(q, dims, tau, frac, scheme):
    import torch
    from paper_2605_27004_gb300 import lbm
    d, N = (2 if q == 9 else 3), int(np.prod(dims))
    solid = inputs.random_mask(N, frac, 4) if frac else None
    rho0, u0 = inputs.noise_field(N, d, 0.05, 6, rho_amp=0.02)
    if frac:
        u0 = u0 * (1 - solid)
    L = lbm.LBM(q, *dims, tau, rand_theta(5, d), solid=solid, storage="fp64", scheme=scheme)
    L.init(torch.as_tensor(rho0), torch.as_tensor(u0))
    m0, p0 = L.totals()
    L.step(10000)
    m1, p1 = L.totals()
    assert abs(m1 - m0) < 1e-14 * m0
    if not frac:  # walls take momentum
        assert np.abs(p1 - p0).max() < 1e-14 * m0


# Four lanes per cell read a cell's rest population and one of them replaces it, in place in the AA
# pattern: the values that are rounded are those of the pull scheme, so the bits are the same. Boxes of
# one warp, of a last warp with spare lanes, and of the largest size that runs so.
@pytest.mark.parametrize("dims", [(3, 2, 1), (33, 7, 1), (64, 64, 1), (76, 64, 1)])
def test_fp64_lanes_in_place_match_pull(dims):
    Th = rand_theta(5, 2)
    rho0, u0 = inputs.noise_field(int(np.prod(dims)), 2, 0.05, 6, rho_amp=0.02)
    for steps in (200, 201):
        f = [gpu_run(9, dims, 0.8, Th, rho0, u0, steps, storage="fp64", scheme=s)["f"] for s in ("pull", "aa")]
        assert np.array_equal(f[0], f[1])


# D3Q19 FP32 boxes run two steps per launch: the same arithmetic, so the same bits as single steps.
# Tiles of 64 x 9 cells: rows in one, two and three tiles (the last narrower), rows left over in y,
# planes split among blocks in chunks of one tile and in runs over several; odd step counts, and
# stops for a check and for recorded checkpoints inside the run; boxes on both sides of the rule that
# takes them there.
@pytest.mark.parametrize("storage", ["fp32s", "fp32"])
@pytest.mark.parametrize("dims,pays", [((128, 128, 128), True), ((64, 180, 181), True), ((120, 130, 140), True),
                                       ((192, 99, 160), True), ((192, 100, 113), False), ((8, 1, 1), False)])
def test_two_steps_per_launch_match_single_steps(dims, pays, storage):
    import torch
    from paper_2605_27004_gb300 import lbm
    N = int(np.prod(dims))
    Th = rand_theta(3, 3)
    g = torch.Generator(device="cuda").manual_seed(2)
    rho = 1 + 0.02 * torch.randn(N, device="cuda", generator=g)
    u = 0.03 * torch.randn(3, N, device="cuda", generator=g)
    runs = []
    for together, kw in ((True, {}), (False, {}), (True, {"check_every": 5}), (True, {"use_graphs": 1})):
        L = lbm.LBM(19, *dims, 0.62, Th, storage=storage, **kw)
        L.record_checkpoints(7 if kw else 0)
        L.init(rho, u)
        before = L.launches
        for n in [17] if together else [1] * 17:
            L.step(n)
        runs.append((L.launches - before, L.populations()))
    assert runs[1][0] == 17
    assert runs[0][0] == (9 if pays else 17)
    for _, f in runs:
        assert torch.equal(f, runs[1][1])


# A thread of a tile narrower than 64 cells has no second cell, and what it computes in its place says
# nothing about the box: densities that fall from 55 to 0.02 along x at a speed of 0.9 stay positive over four
# steps, while the populations along z of a tile's first cell with the others of its last cells sum to
# less than zero.
def test_two_steps_per_launch_accept_an_uneven_state():
    import torch
    from paper_2605_27004_gb300 import lbm
    dims = (120, 130, 140)  # tiles of 64 and 56 cells
    N = int(np.prod(dims))
    x = torch.arange(N, device="cuda") % dims[0]
    rho = torch.exp(4 * torch.cos(2 * np.pi * (x - 64) / dims[0]))
    u = torch.zeros(3, N, device="cuda")
    u[0] = 0.9
    L = lbm.LBM(19, *dims, 0.8, np.eye(3) / 3, check_every=2, use_graphs=-1)
    L.init(rho, u)
    before = L.launches
    L.step(4)
    assert L.launches - before == 2
    assert L.moments()[0].min() > 0


# The split of a box for two steps per launch tries every split of nz: once per context, not per launch,
# where it cost the host 140 us at nz = 32768 (a launch costs it some 5). Enqueueing single launches takes
# no longer in a tall box than in a flat one of as many cells.
def test_tall_boxes_cost_the_host_no_more():
    import time
    import torch
    from paper_2605_27004_gb300 import lbm
    took = {}
    for dims in ((8, 32768, 8), (8, 8, 32768)):
        L = lbm.LBM(19, *dims, 0.8, np.eye(3) / 3, use_graphs=-1)
        L.init()
        best = 1e9
        for _ in range(10):
            torch.cuda.synchronize()
            t = time.perf_counter()
            L.step(20)
            best = min(best, time.perf_counter() - t)
        took[dims[2]] = best
    assert took[32768] < 3 * took[8]


# FP16 storage in rows of odd length, and AA with walls: two cells per thread. The FP16 form shifted by
# the weights runs one cell per thread, and at Theta = cs2 I its stored values and its arithmetic
# are the same, so the two give the same bits; so do pull and AA, which round the same post-collision
# values. Rows of 3 to 387 cells (halves of one length and of two), boxes of an odd number of cells and
# of a number that is no multiple of a sector's 16, boxes of one row and one plane.
@pytest.mark.parametrize("q,dims,frac", [(9, (387, 391, 1), 0.0), (9, (67, 9, 1), 0.0), (19, (3, 1, 1), 0.0), (19, (35, 4, 3), 0.0),
                                         (27, (31, 3, 2), 0.0), (19, (5, 1, 7), 0.0), (9, (18, 9, 1), 0.2),
                                         (19, (33, 4, 5), 0.2), (19, (7, 5, 3), 0.3), (27, (6, 5, 3), 0.3),
                                         (27, (40, 6, 5), 0.5), (27, (16, 2, 1), 0.1)])
def test_fp16_two_cells_match_one_cell(q, dims, frac):
    import torch
    from paper_2605_27004_gb300 import lbm
    d, N = (2 if q == 9 else 3), int(np.prod(dims))
    solid = inputs.random_mask(N, frac, 4) if frac else None
    g = torch.Generator(device="cuda").manual_seed(7)
    rho = 1 + 0.02 * torch.randn(N, device="cuda", generator=g)
    u = 0.03 * torch.randn(d, N, device="cuda", generator=g)

    def run(storage, scheme, Th, steps):
        L = lbm.LBM(q, *dims, 0.7, Th, storage=storage, scheme=scheme, solid=solid)
        L.init(rho, u)
        L.step(steps)
        return L.populations()

    iso = np.eye(d) / 3
    for steps in (20, 21):
        for scheme in ("pull", "aa"):
            assert torch.equal(run("fp16s", scheme, iso, steps), run("fp16w", scheme, iso, steps))
        Th = rand_theta(8, d)
        assert torch.equal(run("fp16s", "pull", Th, steps), run("fp16s", "aa", Th, steps))


# D2Q9 FP32 runs eight or four steps per launch on tiles of 8 x 8 to 16 x 16 cells with rings of 3 or 7
# cells: boxes smaller than the rings, rows and columns left over, one box for each tile size; the
# step counts leave remainders of 8, 4 and 1, with and without graphs, checks and checkpoints.
@pytest.mark.parametrize("storage", ["fp32s", "fp32"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 3, 1), (96, 80, 1), (37, 400, 1), (130, 129, 1), (301, 200, 1)])
def test_steps_of_a_plane_match_single_steps(dims, storage):
    import torch
    from paper_2605_27004_gb300 import lbm
    N = int(np.prod(dims))
    Th = rand_theta(3, 2)
    g = torch.Generator(device="cuda").manual_seed(2)
    rho = 1 + 0.02 * torch.randn(N, device="cuda", generator=g)
    u = 0.03 * torch.randn(2, N, device="cuda", generator=g)
    runs = []
    for pieces, kw in (([1] * 53, {}), ([16, 24, 13], {}), ([53], {"use_graphs": -1}), ([53], {"check_every": 11}),
                       ([7, 46], {"use_graphs": 1})):
        L = lbm.LBM(9, *dims, 0.62, Th, storage=storage, **kw)
        L.record_checkpoints(19 if "check_every" in kw else 0)
        L.init(rho, u)
        before = L.launches
        for n in pieces:
            L.step(n)
        runs.append((L.launches - before, L.populations(), L.get_state()))
    assert runs[0][0] == 53 and all(r[0] < 30 for r in runs[1:])
    for _, f, s in runs:
        assert torch.equal(f, runs[0][1]) and torch.equal(s, runs[0][2])


# A D3Q27 FP32 box with walls may fill the GPU's memory: beside its two arrays, a link word a cell and a list
# entry per eight cells it takes no more than its block records (64 bytes per 256 cells).
def test_fp32_walls_take_one_link_word_a_cell():
    from paper_2605_27004_gb300 import lbm
    dims = (64, 64, 64)
    N = int(np.prod(dims))
    L = lbm.LBM(27, *dims, 0.7, np.eye(3) / 3, solid=inputs.random_mask(N, 0.2, 4))
    assert L.device_bytes <= N * (2 * 27 * 4 + 4 + 4 / 8 + 64 / 256) + 4096


# The scalar's AA steps run over the grid: making such a context with walls takes no list memory, not even
# for a while (8 bytes a fluid cell). Beside what it keeps there is the byte mask, and blocks are rounded.
def test_scalar_in_place_makes_no_lists():
    import torch
    from paper_2605_27004_gb300 import lbm
    dims = (64, 64, 64)
    N = int(np.prod(dims))
    solid = inputs.random_mask(N, 0.2, 4)
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated()
    A = lbm.ADE(19, *dims, 0.7, np.eye(3) / 3, solid=solid, storage="fp16s", scheme="aa")
    assert torch.cuda.max_memory_allocated() - before <= A.device_bytes + N + 65536


# Every step kernel reports a density that is not positive, in the step that collides it: of the first step
# (a cell made so) and of the next (a cell of density 100 at a speed of 0.9, whose populations across its
# motion are negative, -0.2 w of it, and take its neighbours there). One launch is `steps` steps; the cell
# is the box's last one, so an end of a tile, of a row's second half and of a warp, or one with a fluid
# neighbour in y and z.
@pytest.mark.parametrize("q,dims,storage,scheme,frac,steps", [
    (19, (120, 130, 140), "fp32s", "pull", 0.0, 2), (9, (37, 40, 1), "fp32s", "pull", 0.0, 8),
    (9, (301, 200, 1), "fp32", "pull", 0.0, 4), (9, (33, 7, 1), "fp64", "pull", 0.0, 1), (9, (33, 7, 1), "fp64", "aa", 0.0, 1),
    (19, (35, 5, 4), "fp16s", "pull", 0.0, 1), (19, (35, 5, 4), "fp16s", "aa", 0.0, 1), (27, (34, 5, 4), "fp16s", "aa", 0.2, 1),
    (19, (33, 5, 4), "fp16s", "aa", 0.2, 1), (27, (34, 5, 4), "fp16s", "pull", 0.2, 1), (19, (20, 5, 4), "fp32s", "aa", 0.0, 1)])
def test_divergence_is_reported(q, dims, storage, scheme, frac, steps):
    import torch
    from paper_2605_27004_gb300 import lbm
    d, N = (2 if q == 9 else 3), int(np.prod(dims))
    solid = inputs.random_mask(N, frac, 4) if frac else np.zeros(N, np.uint8)
    m = solid.reshape(dims[2], dims[1], dims[0])
    near = (m == 0) & (np.roll(m, -1, 1) == 0) & (np.roll(m, -1, 0) == 0)  # fluid, as are its neighbours in +y and +z
    cell = int(np.flatnonzero(near.ravel())[-1])
    if not frac:
        assert cell == N - 1
    L = lbm.LBM(q, *dims, 0.8, np.eye(d) / 3, solid=solid if frac else None, storage=storage, scheme=scheme,
                check_every=steps, use_graphs=-1)

    def start(rho, u):
        r, v = torch.ones(N, dtype=L.dtype), torch.zeros(d, N, dtype=L.dtype)
        r[cell], v[0, cell] = rho, u
        L.init(r, v)

    def fails():
        before = L.launches
        with pytest.raises(lbm.LBMError) as e:
            L.step(steps)
        assert e.value.status == -6 and L.launches - before == 1

    start(1.0, 0.05)
    L.step(2 * steps)
    start(-1.0, 0.0)
    fails()
    start(100.0, 0.9)
    if steps == 1:
        L.step(1)
    fails()
    if frac:  # what stands in a solid cell is no state
        r = torch.ones(N, dtype=L.dtype)
        r[torch.as_tensor(solid != 0)] = float("nan")
        L.init(r, None)
        L.step(4)


# A flow step, its moments into the scalar's velocity field and the scalar's step, each set up while the one
# before still runs: against the same calls with a wait after each, bit for bit, and the oracle. The
# launches queue up behind a bounded spin, so that they do overlap. Boxes of one block an SM at most and
# of several; a velocity that changes from step to step.
@pytest.mark.parametrize("storage,scheme", [("fp32s", "pull"), ("fp32s", "aa"), ("fp16s", "pull"), ("fp16s", "aa")])
@pytest.mark.parametrize("q,dims", [(19, (34, 20, 6)), (9, (30, 40, 1)), (27, (33, 10, 8)), (19, (64, 96, 60)),
                                    (27, (64, 64, 48)), (9, (200, 1000, 1))])
def test_coupled_steps_overlap_in_order(q, dims, storage, scheme):
    import oracle
    import torch
    from paper_2605_27004_gb300 import lbm
    d, N, steps = (2 if q == 9 else 3), int(np.prod(dims)), 11
    Th, ThS = rand_theta(3, d), rand_theta(4, d)
    rho0, u0 = inputs.noise_field(N, d, 0.08, 6, rho_amp=0.02)
    phi0 = 1.0 + 0.5 * np.random.default_rng(2).random(N)
    F = lbm.LBM(q, *dims, 0.6, Th, storage=storage, scheme=scheme)
    S = lbm.ADE(q, *dims, 0.7, ThS, storage=storage, scheme=scheme)
    view = S.velocity_view()
    got = []
    for wait in (False, True, False):
        F.init(torch.as_tensor(rho0), torch.as_tensor(u0))
        view.zero_()
        S.init(torch.as_tensor(phi0))
        torch.cuda.synchronize()
        if not wait:
            torch.cuda._sleep(10_000_000)
        for _ in range(steps):
            for call in (lambda: F.step(1), lambda: F.moments_into(u=view), lambda: S.step(1)):
                call()
                if wait:
                    torch.cuda.synchronize()
        got.append((S.scalar(), S.populations(), F.populations()))
    for g in (got[0], got[2]):
        assert all(torch.equal(a, b) for a, b in zip(g, got[1]))
    if N < 10000:
        Pf = oracle.Problem(q, *dims, 0.6, Th)
        f = Pf.init(rho0, u0)
        g = oracle.ADEProblem(q, *dims, 0.7, ThS, np.zeros((d, N))).init_scalar(phi0)
        for _ in range(steps):
            Pf.run(f, 1)
            PS = oracle.ADEProblem(q, *dims, 0.7, ThS, Pf.moments(f)[1])
            PS.run_scalar(g, 1)
        tol = 2e-6 if storage == "fp32s" else 1e-3  # as for each of the two alone (40 steps)
        assert rel_l2(got[0][0].double().cpu().numpy(), PS.scalar(g)) < tol


# A flow and a scalar on streams of their own, joined by events, as the caller runs them and as a graph
# captured over both streams: kernels that may be set up early then have predecessors on two streams.
@pytest.mark.parametrize("storage,scheme", [("fp32s", "pull"), ("fp16s", "aa")])
@pytest.mark.parametrize("q,dims", [(19, (34, 20, 6)), (9, (200, 1000, 1))])
def test_coupled_steps_on_two_streams_and_in_a_graph(q, dims, storage, scheme):
    import torch
    from paper_2605_27004_gb300 import lbm
    d, N, steps = (2 if q == 9 else 3), int(np.prod(dims)), 6
    rho0, u0 = (torch.as_tensor(a, device="cuda", dtype=torch.float32)
                for a in inputs.noise_field(N, d, 0.08, 6, rho_amp=0.02))
    phi0 = 1.0 + 0.5 * torch.as_tensor(np.random.default_rng(2).random(N), device="cuda", dtype=torch.float32)
    torch.cuda.synchronize()
    sf, ss = torch.cuda.Stream(), torch.cuda.Stream()
    F = lbm.LBM(q, *dims, 0.6, rand_theta(3, d), storage=storage, scheme=scheme, stream=sf)
    S = lbm.ADE(q, *dims, 0.7, rand_theta(4, d), storage=storage, scheme=scheme, stream=ss)
    view = S.velocity_view()

    def run(wait):
        F.init(rho0, u0)
        S.init(phi0)
        for _ in range(steps):
            F.step(1)
            sf.wait_stream(ss)  # the scalar has read the last velocity
            F.moments_into(u=view)
            ss.wait_stream(sf)
            S.step(1)
            if wait:
                torch.cuda.synchronize()
        sf.wait_stream(ss)

    def result():
        torch.cuda.synchronize()
        with torch.cuda.stream(ss):
            g = S.populations()
        with torch.cuda.stream(sf):
            f = F.populations()
        torch.cuda.synchronize()
        return g, f

    got = []
    for wait in (True, False):
        with torch.cuda.stream(ss):
            view.zero_()
        torch.cuda.synchronize()
        run(wait)
        got.append(result())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=sf):
        ss.wait_stream(sf)
        with torch.cuda.stream(ss):
            view.zero_()
        run(False)
    for _ in range(2):
        graph.replay()
        got.append(result())
    for g, f in got[1:]:
        assert torch.equal(g, got[0][0]) and torch.equal(f, got[0][1])


# Held segments with walls (the fluid-cell and sector lists, out of place) and with checkpoints in host
# memory, copied back ahead of use (room for six states) and not (five).
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("frac,states", [(0.2, 0), (0.2, 6), (0.0, 6), (0.0, 5)])
def test_gradient_with_held_segment_walls_and_host_checkpoints(scheme, frac, states):
    import torch
    from paper_2605_27004_gb300 import lbm
    dims, n, K = (18, 7, 6), 20, 5
    N = int(np.prod(dims))
    solid = inputs.random_mask(N, frac, 4) if frac else None
    g = torch.Generator(device="cuda").manual_seed(5)
    u = 0.03 * torch.randn(3, N, device="cuda", generator=g)
    w = torch.randn(3, N, device="cuda", generator=g)
    L = lbm.LBM(19, *dims, 0.7, rand_theta(2, 3), solid=solid, storage="fp16s", scheme=scheme, use_graphs=-1,
                adjoint_mem_limit=states * 19 * N * 2)
    L.record_checkpoints(K)
    runs = []
    for _ in range(3):
        L.init(None, u)
        L.step(n)
        before = L.launches
        L.adjoint(w, n, K)
        runs.append((L.launches - before, L.gradients(), L.populations()))
        assert (L.adjoint_info()[1] > 0) == (states == 6)
    for count, (dth, dtau, du0), f in runs[1:]:
        assert count == runs[0][0] - (K - 1)
        assert np.array_equal(dth, runs[0][1][0]) and dtau == runs[0][1][1]
        assert torch.equal(du0, runs[0][1][2]) and torch.equal(f, runs[0][2])


def test_slab_group_waits_for_fields_of_the_callers_stream():
    """SlabGroup reads the slabs' fields on the slabs' streams: the kernels that cut them out of the box on
    the caller's stream (held back here by bounded spins of some 10 ms) have to end first."""
    import torch
    from paper_2605_27004_gb300 import slabs
    dims, N = (12, 5, 8), 12 * 5 * 8
    rho0, u0 = (torch.as_tensor(a, device="cuda") for a in inputs.noise_field(N, 3, 0.05, 3, rho_amp=0.02))
    got = []
    for hold in (True, False):
        G = slabs.SlabGroup(19, *dims, 0.7, rand_theta(1, 3), 4, storage="fp64")
        if hold:
            cut = G._slab_fields

            def late(x, r):
                part = cut(x, r)
                torch.cuda._sleep(20_000_000)
                return part * 1.0

            G._slab_fields = late
        G.init(rho0, u0)
        G.step(2)
        got.append(G.populations())
    assert torch.equal(got[0], got[1])


def test_slab_group_gradients_wait_for_the_callers_stream():
    """The slabs' parts of du0 are written on the slabs' streams: not into memory that the caller's stream,
    held back here by a bounded spin, has yet to write for tensors that are gone."""
    import torch
    from paper_2605_27004_gb300 import slabs
    dims, N = (12, 5, 8), 12 * 5 * 8
    rho0, u0 = (torch.as_tensor(a, device="cuda") for a in inputs.noise_field(N, 3, 0.05, 3, rho_amp=0.02))
    G = slabs.SlabGroup(19, *dims, 0.7, rand_theta(1, 3), 2, storage="fp64")
    G.init(rho0, u0)
    G.step(4)
    G.adjoint(u0.clone(), 4, 2)
    want = G.gradients()[2]
    for spin in (1, 100_000_000):  # the first pass loads the kernels
        torch.cuda.synchronize()
        torch.cuda._sleep(spin)
        gone = [torch.full((3, G.ctx[0].N), 7.0, dtype=torch.float64, device="cuda") for _ in range(4)]
        del gone
        assert torch.equal(G.gradients()[2], want)


# From the second gradient on, the forward run leaves its last segment's states in the adjoint's
# buffers: the same states as recomputed ones, so the same bits as the first gradient. Whole and cut last
# segments, one of a single step, a run shorter than a segment; both schemes and parities; in between
# a run in two pieces (no segment can be held), a second adjoint of the same run, released buffers.
@pytest.mark.parametrize("n,K", [(24, 6), (23, 5), (21, 5), (9, 20), (22, 7)])
@pytest.mark.parametrize("storage,scheme", [("fp32s", "pull"), ("fp16s", "aa"), ("fp64", "aa")])
@pytest.mark.parametrize("graphs", [-1, 1])
def test_gradient_with_held_segment(n, K, storage, scheme, graphs):
    import torch
    from paper_2605_27004_gb300 import lbm
    dims = (18, 7, 6)
    N = int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(5)
    u = (0.03 * torch.randn(3, N, device="cuda", generator=g)).double()
    w = torch.randn(3, N, device="cuda", generator=g).double()
    L = lbm.LBM(19, *dims, 0.7, rand_theta(2, 3), storage=storage, scheme=scheme, use_graphs=graphs)
    L.record_checkpoints(K)

    def gradient(pieces, times=1):
        L.init(None, u)
        for m in pieces:
            L.step(m)
        f = L.populations()
        for _ in range(times):
            before = L.launches
            L.adjoint(w, n, K)
            count = L.launches - before
        dth, dtau, du0 = L.gradients()
        return f, dth, dtau, du0, count

    first = gradient([n])
    for pieces, times, release in (([n], 1, False), ([n - 2, 2], 1, False), ([n], 2, False), ([n], 1, True), ([n], 1, False)):
        if release:
            L.adjoint_release()
        again = gradient(pieces, times)
        assert torch.equal(again[0], first[0]) and torch.equal(again[3], first[3])
        assert np.array_equal(again[1], first[1]) and again[2] == first[2]
    held = n - (n - 1) // K * K - 1 if n >= K else 0  # a run shorter than a segment is run again
    assert again[4] == first[4] - held


# A run whose states no gradient will read is not taken through the adjoint's buffers in single steps: not
# the pieces of a run (D2Q9 FP32 takes 20 steps in 3 launches), not a run of other length than
# the last gradient's, and of those that follow one gradient only the first. Launches per run, and the
# gradient afterwards.
def test_only_runs_before_a_gradient_are_held():
    import torch
    from paper_2605_27004_gb300 import lbm
    dims, n, K = (30, 20, 1), 40, 20
    N = int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(5)
    u = 0.03 * torch.randn(2, N, device="cuda", generator=g)
    w = torch.randn(2, N, device="cuda", generator=g)
    L = lbm.LBM(9, *dims, 0.7, rand_theta(2, 2), use_graphs=-1)
    L.record_checkpoints(K)

    def run(pieces):
        L.init(None, u)
        before = L.launches
        for m in pieces:
            L.step(m)
        return L.launches - before

    several = run([20])  # 8 + 8 + 4 steps
    assert several == 3 and run([n]) == 2 * several
    L.adjoint(w, n, K)
    first = L.gradients()
    assert run([20, 10, 5, 5]) == several + 3 + 2 + 2  # 8 + 2 * 1, 4 + 1, 4 + 1
    assert run([25]) == several + 2
    assert run([n]) == several + K  # held
    assert run([n]) == 2 * several  # its states were not used
    L.adjoint(w, n, K)
    assert run([n]) == several + K
    L.adjoint(w, n, K)
    again = L.gradients()
    assert torch.equal(again[2], first[2]) and np.array_equal(again[0], first[0]) and again[1] == first[1]
    # a run shorter than a segment is no recorded segment of its adjoint, which runs it again
    assert run([9]) == 2
    L.adjoint(w, 9, K)
    assert run([9]) == 2


# The adjoint's steps add to the gradient records of the step before, and are set up while that one
# runs: their sums against those of a process that waits for every launch, bit for bit. Rows that leave
# fewer than the eight threads of a record in the last block of a row (5, 260 and 33 cells).
def _gradients_of_short_rows(path):
    import torch
    from paper_2605_27004_gb300 import lbm
    out = []
    for q, dims in ((19, (5, 6, 4)), (19, (260, 3, 2)), (9, (33, 5, 1))):
        d, N = (2 if q == 9 else 3), int(np.prod(dims))
        rho0, u0 = inputs.noise_field(N, d, 0.05, 6, rho_amp=0.02)
        w = np.random.default_rng(4).standard_normal((d, N))
        for scheme in ("pull", "aa"):
            L = lbm.LBM(q, *dims, 0.7, rand_theta(2, d), scheme=scheme, use_graphs=-1)
            L.init(torch.as_tensor(rho0), torch.as_tensor(u0))
            L.step(40)
            L.adjoint(torch.as_tensor(w), 40, 20)
            dth, dtau, du0 = L.gradients()
            out.append(np.concatenate([dth, [dtau], du0.double().cpu().numpy().ravel()]))
    np.save(path, np.concatenate(out))


def test_gradient_records_match_waited_launches(tmp_path):
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    got = []
    for wait in ("0", "1"):
        path = str(tmp_path / f"{wait}.npy")
        code = (f"import sys; sys.path[:0] = [{os.path.dirname(here)!r}, {here!r}]; import test_gpu_step_paths as t; "
                f"t._gradients_of_short_rows({path!r})")
        subprocess.run([sys.executable, "-c", code], check=True, timeout=300,
                       env=dict(os.environ, CUDA_LAUNCH_BLOCKING=wait))
        got.append(np.load(path))
    assert np.isfinite(got[0]).all() and np.array_equal(got[0], got[1])


# A caller's graph of a recorded run: it keeps no address of the adjoint's buffers, which may be released
# before a replay, and a replay starts another trajectory without a call that says so, so that states held
# by an earlier run must not serve its gradient.
@pytest.mark.parametrize("storage,scheme", [("fp32s", "pull"), ("fp16s", "aa")])
def test_recorded_run_in_a_callers_graph(storage, scheme):
    import torch
    from paper_2605_27004_gb300 import lbm
    dims, n, K = (18, 7, 6), 20, 5
    N = int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(5)
    fields = [0.03 * torch.randn(3, N, device="cuda", generator=g) for _ in range(2)]
    w = torch.randn(3, N, device="cuda", generator=g)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()

    def context():
        L = lbm.LBM(19, *dims, 0.7, rand_theta(2, 3), storage=storage, scheme=scheme, stream=s)
        L.record_checkpoints(K)
        return L

    def gradient(L):
        before = L.launches
        L.adjoint(w, n, K)
        return L.gradients(), L.launches - before

    with torch.cuda.stream(s):
        want = []
        for u in fields:
            L = context()
            L.init(None, u)
            L.step(n)
            want.append((gradient(L), L.populations()))
        L, u = context(), fields[0].clone()
        for _ in range(2):  # the second run holds its last segment
            L.init(None, u)
            L.step(n)
            (_, _, du0), launches = gradient(L)
            assert torch.equal(du0, want[0][0][0][2])
        assert launches == want[0][0][1] - (K - 1)
        graph = torch.cuda.CUDAGraph()
        s.synchronize()
        with torch.cuda.graph(graph, stream=s):
            L.init(None, u)
            L.step(n)
        for other in (False, True):  # without and with a run of the library's own before the replay
            if other:
                L.init(None, fields[0])
                L.step(n)
            u.copy_(fields[1])
            graph.replay()
            ((dth, dtau, du0), _), ref = gradient(L), want[1][0][0]
            assert torch.equal(du0, ref[2]) and np.array_equal(dth, ref[0]) and dtau == ref[1]
        L.adjoint_release()
        u.copy_(fields[0])
        graph.replay()
        assert torch.equal(L.populations(), want[0][1])
