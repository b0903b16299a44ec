"""The particle step's work units, the one-kernel re-sort and the ring form of
the potential update, at the sizes
where they can go wrong: tiles of exactly one, a whole number and one more
than a whole number of units, key counts around the scans' block sizes, the
sparse tiles' kernel beside the units, an empty bunch; against the oracle."""
import ctypes as C
import re
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_1612_03310_gb300 import inputs
from test_parity_gpu import (C1_UND, M, compare_fields, compare_particles,  # noqa: F401
                             oracle_fields, set_state)

pytestmark = pytest.mark.gpu

# tolerances of the parity tests' single steps, for their reasons: sums of a
# few FP32 roundings a step
TOL = {"P64": (1e-10, 1e-10, 1e-9), "P32": (1e-5, 2e-5, 1e-5), "P32_U64": (1e-5, 2e-5, 1e-5)}


def heavy_bunch(seed, g, counts):
    """counts[m] particles in the m-th 8^3-cell tile (clear of the outer
    cells), the rest of the grid empty."""
    rng = np.random.default_rng(seed)
    r = []
    tiles = [(i, j, k) for k in range(g["nz"] // 8) for j in range(g["ny"] // 8)
             for i in range(g["nx"] // 8)]
    for (i, j, k), n in zip(tiles, counts):
        lo = np.array([max(8 * c, 3) for c in (i, j, k)], float)
        hi = np.array([min(8 * c + 8, v - 5) for c, v in zip((i, j, k), (g["nx"], g["ny"], g["nz"]))],
                      float)
        r.append(lo + (hi - lo) * rng.random((n, 3)))
    r = np.concatenate(r)
    u = 0.2 * rng.standard_normal((3, len(r)))
    return dict(x=g["x0"] + r[:, 0] * g["dx"], y=g["y0"] + r[:, 1] * g["dy"],
                z=g["z0"] + r[:, 2] * g["dz"], ux=u[0], uy=u[1], uz=u[2], q_macro=-1e-15)


def check(M, orc, g, und, P, prec, steps, **tuning):  # noqa: F811
    o = orc.OracleSim(g, und, P)
    tf, tc, eps = TOL[prec]
    with M.Simulation(dict(g, boundary=1), und, P, precision=getattr(M, prec)) as sim:
        if tuning:
            sim.set_tuning(**tuning)
        for n in steps:
            o.step(n)
            sim.step(n)
            sim.sync()
            compare_fields(sim, o, tf, names=["Ex", "Ey", "Bz", "phi", "Jx", "Jz", "rho"])
            compare_particles(sim, o, tc, eps)


@pytest.mark.parametrize("prec", ["P64", "P32", "P32_U64"])
@pytest.mark.parametrize("below", [0, 300])
def test_split_tiles(M, orc, prec, below):  # noqa: F811
    # units of 256 slots: one short of, exactly, and one over one and two
    # units, a heavy tile, empty ones between; with below = 300 the light
    # tiles go to the sparse tiles' kernel
    g = inputs.random_grid(41, 32, 24, 24)
    P = heavy_bunch(42, g, [255, 256, 257, 0, 511, 512, 513, 1, 0, 3000])
    check(M, orc, g, dict(C1_UND, z_ent_lab=0.0), P, prec, (1, 4), push_sparse_below=below)


@pytest.mark.parametrize("shape", [(8, 8, 8), (64, 64, 64), (24, 152, 72), (72, 56, 2056),
                                   (128, 128, 128), (136, 128, 128)])
def test_resort_key_counts(M, orc, shape):  # noqa: F811
    # 1, 512 and 513 tiles (one and two keys a thread of the one-kernel
    # re-sort), 16191 (two passes), 4096 (the two-pass limit) and 4352
    g = inputs.random_grid(51, *shape)
    P = inputs.random_particles(52, g, 3000, u_scale=0.2)
    check(M, orc, g, dict(C1_UND, z_ent_lab=0.0), P, "P32_U64", (1, 4))


def test_no_particles_sources_once(M, orc):  # noqa: F811
    # without particles a set source drives one update, and the following
    # updates read none
    g = inputs.random_grid(61, 20, 18, 24)
    src = 1e3 * np.random.default_rng(3).standard_normal((g["nz"], g["ny"], g["nx"]))
    with M.Simulation(dict(g, boundary=1), None, None, precision=M.P64) as sim:
        o = orc.OracleSim(g, None, dict(x=[], y=[], z=[], ux=[], uy=[], uz=[]))
        for _ in range(2):
            s = o.src.copy()
            s[:o.n_cell] = src.ravel()
            o.set_sources(s)
            sim.set_field("Jx", src)
            for n in (1, 6):
                o.step(n)
                sim.step(n)
                sim.sync()
                compare_fields(sim, o, 1e-10, names=["Ax", "Ex", "By", "Jx"])
        assert sim.source_tiles() == (0, False)
        assert sim.time()[0] == 14


@pytest.mark.parametrize("prec", ["P32", "P32_C"])
@pytest.mark.parametrize("boundary", [1, 2])
@pytest.mark.parametrize("shape", [(64, 72, 273), (129, 40, 155), (130, 48, 155), (97, 80, 243),
                                   (127, 57, 155)])
def test_ring_update(M, orc, prec, boundary, shape):  # noqa: F811
    # the ring form of the update (grids of at least two 8-plane column tiles
    # a multiprocessor): odd nx (lo parts by cp.async) and even (by TMA), nx a
    # multiple of 32, one more (the x+ face in the boundary kernel) and one
    # less, last tiles of one row or plane, runs that end in a short one; a
    # level with everything random so that every face is seen
    g = dict(inputs.random_grid(71, *shape), boundary=boundary)
    f = inputs.random_fields(72, g, scale=1e-9)
    f = {k: v.astype(np.float32).astype(np.float64) for k, v in f.items()}
    P = inputs.random_particles(73, g, 500, u_scale=0.2)
    o = orc.OracleSim(g, None, P)
    with M.Simulation(g, None, P, precision=getattr(M, prec)) as sim:
        set_state(sim, o, f)
        o.step(2)
        sim.step(2)
        sim.sync()
        compare_fields(sim, o, 1e-5)
        for nm in ("Ax", "Az", "phi"):  # the largest vertex too, of the largest value
            ref = oracle_fields(o)[nm]
            assert np.abs(sim.copy_field(nm) - ref).max() <= 1e-5 * np.abs(ref).max(), nm


def test_fp64_moves_across_cells(M, orc):  # noqa: F811
    # the FP64 cell carry: fractions 0 and just below 1, steps that end on a
    # face, before it and past it along each axis
    g = inputs.random_grid(81, 24, 24, 24)
    h = np.array([g["dx"], g["dy"], g["dz"]])
    r0 = np.array([g["x0"], g["y0"], g["z0"]])
    frac = [0.0, 1e-18, 0.25, 0.5, 1.0 - 2.0 ** -40]
    pos, mom = [], []
    for f in frac:
        for a in range(3):
            for u in (-3.0, -1e-3, 0.0, 1e-3, 3.0):
                p = np.full(3, 10.5)
                p[a] = 10.0 + f
                v = np.zeros(3)
                v[a] = u
                pos.append(r0 + p * h)
                mom.append(v)
    pos, mom = np.array(pos), np.array(mom)
    P = dict(x=pos[:, 0], y=pos[:, 1], z=pos[:, 2], ux=mom[:, 0], uy=mom[:, 1], uz=mom[:, 2],
             q_macro=-1e-18)
    check(M, orc, g, None, P, "P64", (1, 1, 3))


@pytest.mark.parametrize("fused", [None, True, False])
def test_sparse_threshold_switched_off(M, orc, fused):  # noqa: F811
    # lists built with every tile sparse, then a threshold of none: the step
    # that still runs on those lists pushes their tiles too
    g = inputs.random_grid(91, 32, 24, 24)
    P = inputs.random_particles(92, g, 2000, u_scale=0.2)
    und = dict(C1_UND, z_ent_lab=0.0)
    o = orc.OracleSim(g, und, P)
    with M.Simulation(dict(g, boundary=1), und, P, precision=M.P32_U64) as sim, M.Batch() as b:
        for below, n in ((1 << 30, 4), (0, 4), (1 << 30, 3), (1, 2)):
            sim.set_tuning(push_sparse_below=below)
            if fused is not None:
                b.set_mode(fused)
                b.add(sim)
                b.step(n)
                b.sync()
                b.remove(sim)
            else:
                sim.step(n)
            o.step(n)
            sim.sync()
            compare_fields(sim, o, 1e-5, names=["Ex", "Bz", "phi", "Jx", "rho"])
            compare_particles(sim, o, 2e-5, 1e-5)


@pytest.mark.parametrize("prec", ["P64", "P32", "P32_C"])
@pytest.mark.parametrize("shape", [(4, 4, 4), (5, 4, 7), (33, 6, 9), (32, 8, 4), (34, 9, 16),
                                   (64, 5, 6), (65, 17, 12)])
def test_update_with_its_boundary(M, orc, prec, shape):  # noqa: F811
    # small grids, where the register form updates every boundary vertex
    # itself (nx - 1 a multiple of 32: the boundary kernel's part): corners
    # and edges of grids down to two interior vertices an axis, every vertex
    # compared
    g = dict(inputs.random_grid(95, *shape), boundary=1)
    f = inputs.random_fields(96, g, scale=1e-9)
    if prec != "P64":
        f = {k: v.astype(np.float32).astype(np.float64) for k, v in f.items()}
    o = orc.OracleSim(g, None, dict(x=[], y=[], z=[], ux=[], uy=[], uz=[]))
    with M.Simulation(g, None, None, precision=getattr(M, prec)) as sim:
        set_state(sim, o, f)
        for n in (1, 2):
            o.step(n)
            sim.step(n)
            sim.sync()
            for nm in ("Ax", "Ay", "Az", "phi", "Ax_prev"):
                ref = oracle_fields(o)[nm]
                tol = 1e-12 if prec == "P64" else 1e-5
                assert np.abs(sim.copy_field(nm) - ref).max() <= tol * np.abs(ref).max(), nm


def test_fused_batch_members_without_particles(M):  # noqa: F811
    # members without particles list no units, among more members than one
    # launch of the particle step takes
    pairs = []
    for k in range(33):
        g = dict(inputs.random_grid(100 + k, 16, 16, 16 + k % 5), boundary=1)
        P = inputs.random_particles(200 + k, g, 100 * (k % 3), u_scale=0.2) if k % 3 else None
        pairs.append([M.Simulation(g, None, P, precision=M.P32_U64) for _ in range(2)])
    with M.Batch() as b:
        b.set_mode(True)
        for s, _ in pairs:
            b.add(s)
        b.step(4)
        assert b.fused()
        b.sync()
        for s, alone in pairs:
            alone.step(4)
            for nm in ("Ay", "Ex", "rho"):
                a, c = s.copy_field(nm), alone.copy_field(nm)
                assert np.abs(a - c).max() <= 1e-5 * np.abs(c).max(), nm
    for s, alone in pairs:
        s.close()
        alone.close()


@pytest.mark.parametrize("prec,tol", [("P64", 1e-11), ("P32_U64", 1e-7)])
def test_bunch_record_waits_for_the_sparse_tiles(M, prec, tol):  # noqa: F811
    # every tile sparse, so that all particles are pushed by the kernel beside
    # the tiled one: each step's record holds the state after that step, as
    # bunch_stats gives it.  The two differ by the order of the field's atomics
    # only (weak charges); a step moves the means of these 2e5 particles by
    # some 0.3 c dt / sqrt(2e5), 2e-5 of the spreads
    g = dict(inputs.random_grid(121, 64, 64, 64), boundary=1)
    P = dict(inputs.random_particles(122, g, 200000, u_scale=0.3), q_macro=-1e-18)
    with M.Simulation(g, None, P, precision=getattr(M, prec)) as sim, \
            M.Simulation(g, None, P, precision=getattr(M, prec)) as alone:
        sim.set_tuning(push_sparse_below=1 << 30)
        sim.set_bunch_sampling(1.0e3, 1, 12)
        sim.step(12)
        rec = sim.read_bunch()
        assert list(rec[:, 0]) == list(range(1, 13))
        for r in rec:
            alone.step(1)
            ref = alone.bunch_stats(1.0e3)
            spread = ref[6:12]
            assert (np.abs(r[1:7] - ref[:6]) <= tol * spread).all(), (r[0], r[1:7] - ref[:6])
            assert (np.abs(r[7:13] - spread) <= tol * spread).all(), (r[0], r[7:13] - spread)
            assert r[14] == ref[13]


def test_copy_out_from_several_threads(M):  # noqa: F811
    # calls of several threads on one simulation, each with scratch of its
    # own: fields of 0.25 MB (the kept scratch), particles, samples, and at
    # (40, 40, 400) a field above the kept scratch's 4 MB
    for shape in ((32, 32, 32), (40, 40, 400)):
        g = dict(inputs.random_grid(131, *shape), boundary=1)
        P = inputs.random_particles(132, g, 20000, u_scale=0.2)
        ijk = np.random.default_rng(1).integers(1, 30, (3000, 3))
        with M.Simulation(g, None, P, precision=M.P64) as sim:
            sim.step(6)
            calls = [lambda nm=nm: sim.copy_field(nm) for nm in ("Ex", "phi", "rho")] + [
                lambda: sim.copy_particles()["z"], lambda: sim.copy_particles()["uy"],
                lambda: sim.sample_fields(["Ey", "Az"], ijk)]
            ref = [f() for f in calls]
            with ThreadPoolExecutor(len(calls)) as pool:
                runs = [pool.submit(lambda f=f, r=r: [np.array_equal(f(), r) for _ in range(40)])
                        for f, r in zip(calls, ref)]
                assert all(all(r.result()) for r in runs)


def test_graph_captured_before_the_sparse_threshold(M, orc):  # noqa: F811
    # a caller's own graph of two steps, captured while every tile is staged
    # (no kernel for sparse tiles in it), replayed on lists whose tiles are all
    # sparse: its first step pushes them too
    torch = pytest.importorskip("torch")
    g = inputs.random_grid(141, 32, 24, 24)
    P = inputs.random_particles(142, g, 2000, u_scale=0.2)
    und = dict(C1_UND, z_ent_lab=0.0)
    o = orc.OracleSim(g, und, P)
    q = torch.cuda.Stream()
    with M.Simulation(dict(g, boundary=1), und, P, precision=M.P32_U64, stream=q.cuda_stream) as sim:
        sim.step(2)
        sim.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=q, capture_error_mode="thread_local"):
            sim.step(2)
        sim.set_tuning(push_sparse_below=1 << 30)
        sim.step(2)
        with torch.cuda.stream(q):
            graph.replay()
        sim.step(3)
        o.step(9)
        sim.sync()
        compare_fields(sim, o, 1e-5, names=["Ex", "Bz", "phi", "Jx", "rho"])
        compare_particles(sim, o, 2e-5, 1e-5)


@pytest.mark.parametrize("prec", ["P32", "P32_U64"])
def test_more_planes_than_a_launch_has_runs_of_eight(M, prec):  # noqa: F811
    # above 8 x 65535 planes: two bunches, each in a window of 64 planes whose
    # vertices agree with a grid of those planes alone (3 steps reach 3 planes)
    nz, size = 8 * 65535 + 9, 64
    small = dict(inputs.random_grid(151, 24, 8, size), boundary=1)
    P = inputs.random_particles(152, dict(small, nz=40), 300, u_scale=0.2)
    P = dict(P, z=P["z"] + 12 * small["dz"])
    big = dict(small, nz=nz)
    windows = (nz // 2, nz - size)
    z = np.concatenate([P["z"] + k * small["dz"] for k in windows])
    both = dict({a: np.tile(P[a], 2) for a in ("x", "y", "ux", "uy", "uz")}, z=z, q_macro=P["q_macro"])
    k, j, i = np.meshgrid(range(8, size - 8), range(1, 7), range(1, 23), indexing="ij")
    at = np.stack([i.ravel(), j.ravel(), k.ravel()], 1)
    names = ["Ex", "Bz", "Az", "phi", "Jz", "rho"]
    with M.Simulation(big, None, both, precision=getattr(M, prec)) as sim, \
            M.Simulation(small, None, P, precision=getattr(M, prec)) as ref:
        sim.step(3)
        sim.sync()
        ref.step(3)
        b = ref.sample_fields(names, at)
        for k0 in windows:
            a = sim.sample_fields(names, at + np.array([0, 0, k0]))
            # z of the big grid is rounded to 2^-52 of 31 m, 1e-10 of a cell
            assert (np.abs(a - b).max(0) <= 1e-5 * np.abs(b).max(0)).all()
            assert (np.abs(b).max(0) > 0).all()


def test_tuning_set_again_changes_nothing(M):  # noqa: F811
    # 64 x 64 x 256 cells, where the library's own run is 8 planes alone: the
    # library's choice stays 0, an explicit 8 stays 8, and settings that leave
    # lz out leave it alone
    g = dict(inputs.random_grid(161, 64, 64, 256), boundary=1)
    with M.Simulation(g, None, None, precision=M.P32) as sim:
        assert sim.tuning()["lz"] == 0 and sim.tuning()["stencil_variant"] == 2
        sim.set_tuning(push_sparse_below=1)
        sim.set_tuning(**sim.tuning())
        assert sim.tuning()["lz"] == 0 and sim.tuning()["push_sparse_below"] == 1
        for lz in (8, 16, 1):
            sim.set_tuning(lz=lz)
            sim.set_tuning(push_variant=0)
            assert sim.tuning()["lz"] == lz
        sim.set_tuning(lz=0)
        assert sim.tuning()["lz"] == 0
        sim.set_tuning(stencil_variant=1)
        assert sim.tuning()["lz"] >= 8


@pytest.mark.parametrize("shape,n", [((16, 16, 24), 80659), ((16, 16, 24), 80660),
                                     ((64, 64, 128), 500), ((64, 64, 129), 500)])
def test_copy_out_parts_and_sizes(M, shape, n):  # noqa: F811
    # outputs on both sides of what fits the kept scratch (4 MB: 80659
    # particles, 524288 vertices), in turn on one simulation; any of the
    # particle arrays NULL leaves the others whole and itself untouched
    g = dict(inputs.random_grid(171, *shape), boundary=1)
    P = dict(inputs.random_particles(172, g, n, u_scale=2.0), q_macro=-1e-18)
    names = ("x", "y", "z", "ux", "uy", "uz")
    with M.Simulation(g, None, P, precision=M.P64) as sim:
        sim.step(6)
        whole = sim.copy_particles()
        assert 0 < whole["lost"].sum() == whole["n_lost"] < n
        ex = sim.copy_field("Ex")
        ijk = np.random.default_rng(2).integers(1, 14, (200, 3))
        at = sim.sample_fields(["Ex"], ijk)[:, 0]
        assert np.array_equal(at, ex[ijk[:, 2], ijk[:, 1], ijk[:, 0]])
        for keep in ([], ["x"], ["uz", "lost"], ["lost"], ["y", "ux"]):
            out = {a: np.full(n, -7.0) for a in names}
            lost = np.full(n, -7, np.int32)
            nl = C.c_int64(-1)
            ptr = [M._dp(out[a]) if a in keep else None for a in names]
            lp = lost.ctypes.data_as(C.POINTER(C.c_int32)) if "lost" in keep else None
            assert M.lib().mithra_copy_particles(sim.h, *ptr, lp, C.byref(nl)) == M.OK
            assert nl.value == whole["n_lost"]
            for a in names:
                assert np.array_equal(out[a], whole[a] if a in keep else np.full(n, -7.0)), a
            assert np.array_equal(lost, whole["lost"] if lp else np.full(n, -7, np.int32))
            assert np.array_equal(sim.copy_field("Ex"), ex)
        again = sim.copy_particles()
        assert all(np.array_equal(again[a], whole[a]) for a in names + ("lost",))


def test_resort_of_the_most_keys_of_one_kernel(M, orc):  # noqa: F811
    # 9 x 13 x 35 = 4095 tiles and the lost particles' bucket: eight keys a
    # thread, every one of the 4096 in use; particles in the last tile, and
    # some that leave the grid through it
    g = inputs.random_grid(181, 72, 104, 280)
    P = inputs.random_particles(182, g, 3000, u_scale=0.2)
    rng = np.random.default_rng(183)
    h = np.array([g["dx"], g["dy"], g["dz"]])
    last = np.array([64.0, 96.0, 272.0]) + rng.random((400, 3)) * [4.0, 4.0, 4.5]
    r = np.array([g["x0"], g["y0"], g["z0"]]) + last * h
    u = 0.2 * rng.standard_normal((3, 400))
    u[2, :100] = 3.0
    P = dict(P, **{a: np.concatenate([P[a], v]) for a, v in
                   zip(("x", "y", "z", "ux", "uy", "uz"), (*r.T, *u))})
    check(M, orc, g, dict(C1_UND, z_ent_lab=0.0), P, "P32_U64", (1, 4, 4))
    o = orc.OracleSim(g, dict(C1_UND, z_ent_lab=0.0), P)
    o.step(9)
    assert 50 < o.lost.sum() < 400


def kernels_of_a_step(M, g, P, prec, path, **tuning):  # noqa: F811
    """Names (mangled) of the kernels that one step launches, from a graph
    captured of it and never run."""
    torch = pytest.importorskip("torch")
    q = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with M.Simulation(g, None, P, precision=getattr(M, prec), stream=q.cuda_stream) as sim:
        if tuning:
            sim.set_tuning(**tuning)
        with torch.cuda.graph(graph, stream=q, capture_error_mode="thread_local"):
            sim.step(1)
        dot = C.CDLL("libcuda.so.1").cuGraphDebugDotPrint  # verbose: 1
        assert dot(C.c_void_p(graph.raw_cuda_graph()), str(path).encode(), C.c_uint(1)) == 0
    return path.read_text()


def smooth_levels(g):
    """Two levels of every component: a constant of order 1 with a hundredth
    of smooth variation, the second a little later than the first; none of the
    values are FP32 numbers."""
    k, j, i = np.meshgrid(np.arange(g["nz"]) / 40.0, np.arange(g["ny"]) / 36.0,
                          np.arange(g["nx"]) / 44.0, indexing="ij")
    levels = [np.concatenate([
        (1.0 / (3 + c) + 0.01 * np.sin(2 * np.pi * (i + 0.7 * j - k + 0.1 * c) + late)).ravel()
        for c in range(4)]) for late in (0.0, 0.02)]
    return dict(prev=levels[0], cur=levels[1], src=np.zeros_like(levels[0]))


@pytest.mark.parametrize("boundary", [1, 2])
@pytest.mark.parametrize("shape,lo", [((64, 72, 273), "TMA"), ((129, 40, 155), "cp.async"),
                                      ((130, 48, 155), "TMA"), ((97, 80, 243), "cp.async"),
                                      ((127, 57, 155), "cp.async")])
def test_ring_update_keeps_the_lo_parts(M, orc, boundary, shape, lo, tmp_path):  # noqa: F811
    # levels near 1 whose second differences are some 1e-4: the hi parts alone
    # round each level by up to 2^-25 = 3e-8 of it, a wrong lo part is worth as
    # much, and the right ones (8 more bits) leave 2^-33 = 1.2e-10, a few times
    # that after four steps' sums (measured 2.9e-10).  The bound lies between,
    # and plain FP32 has to miss it.  The second-order faces' own terms read hi
    # parts alone, in every form; what they leave travels a vertex a step, so
    # that with them the five outermost vertices are left out.
    g = dict(inputs.random_grid(191, *shape), boundary=boundary)
    f = smooth_levels(g)
    # RingLo of the kernel's template: 1 by TMA, 2 by cp.async; 0 plain
    names = {"P32_C": "k_potential_ringILi%d" % (1 if lo == "TMA" else 2), "P32": "k_potential_ringILi0"}
    o = orc.OracleSim(g, None, dict(x=[], y=[], z=[], ux=[], uy=[], uz=[]))
    err = {}
    for prec in ("P32_C", "P32"):
        assert names[prec] in kernels_of_a_step(M, g, None, prec, tmp_path / prec)
        with M.Simulation(g, None, None, precision=getattr(M, prec)) as sim:
            set_state(sim, o, f)
            o.step(4)
            sim.step(4)
            sim.sync()
            ref = oracle_fields(o)
            inner = slice(5, -5) if boundary == 2 else slice(None)
            err[prec] = max(np.abs(sim.copy_field(nm) - ref[nm])[inner, inner, inner].max()
                            for nm in ("Ax", "Ay", "Az", "phi"))
    assert err["P32_C"] <= 2e-9 < 3e-8 < err["P32"], err


@pytest.mark.parametrize("prec", ["P32", "P32_U64", "P64"])
def test_fused_batch_of_sparse_and_dense_members(M, prec):  # noqa: F811
    # 67 uneven members, three groups of the particle step: in turn mixed lists
    # (a dense clump in a thin cloud), all sparse, all dense, none sparse with
    # no particles, and a member whose threshold makes one tile of all dense;
    # each as its lone run, and as its lone run with every tile staged
    rng = np.random.default_rng(201)
    trios, kinds = [], []
    for k in range(67):
        kind = k % 5
        shape = [int(v) for v in rng.integers(16, 34, 3)]
        g = dict(inputs.random_grid(300 + k, *shape, n_sub=1 + k % 2), boundary=1)
        n = 0 if kind == 3 else int(rng.integers(200, 900))
        P = inputs.random_particles(400 + k, g, n, u_scale=0.2) if n else None
        if kind == 0:  # a third of the particles within a cell or two of a vertex
            c = {a: P[a][0] + 0.8 * g["d" + a] * rng.random(n // 3) for a in "xyz"}
            P = dict(P, **{a: np.concatenate([P[a][:-(n // 3)], c[a]]) for a in "xyz"})
        sims = [M.Simulation(g, None, P, precision=getattr(M, prec)) for _ in range(3)]
        below = {0: 60, 1: 1 << 30, 2: 1, 3: 60, 4: 25}[kind]
        for s in sims[:2]:
            s.set_tuning(push_sparse_below=below)
        sims[2].set_tuning(push_sparse_below=1)
        trios.append(sims)
        kinds.append(kind)
    tol = 1e-11 if prec == "P64" else 1e-5
    with M.Batch() as b:
        b.set_mode(True)
        for s in trios:
            b.add(s[0])
        b.step(6)
        assert b.fused()
        b.step(3)
        b.step(2)
        b.sync()
        for k, (inb, alone, staged) in enumerate(trios):
            for s in (alone, staged):
                s.step(11)
                for nm in ("Ay", "Ex", "Jz", "rho"):
                    a, c = inb.copy_field(nm), s.copy_field(nm)
                    assert np.linalg.norm(a - c) <= tol * np.linalg.norm(c), (k, kinds[k], nm)
                if kinds[k] != 3:
                    a, c = inb.copy_particles(), s.copy_particles()
                    assert np.array_equal(a["lost"], c["lost"]), k
                    for nm, d in (("x", "dx"), ("y", "dy"), ("z", "dz")):
                        assert np.abs(a[nm] - c[nm]).max() <= tol * inb.grid[d], (k, kinds[k], nm)
                    for nm in ("ux", "uy", "uz"):
                        assert np.abs(a[nm] - c[nm]).max() <= tol * np.abs(c[nm]).max(), (k, nm)
    for sims in trios:
        for s in sims:
            s.close()


@pytest.mark.parametrize("prec,shape,per_tile,there", [
    ("P64", (64, 128, 384), 40, True), ("P64", (64, 128, 376), 40, False),
    ("P64", (64, 128, 272), 100, True), ("P64", (64, 128, 272), 99, False),
    ("P64", (64, 128, 264), 100, False), ("P32_U64", (128, 128, 232), 40, True),
    ("P32_U64", (128, 128, 224), 40, False)])
def test_automatic_sparse_threshold(M, orc, prec, shape, per_tile, there, tmp_path):  # noqa: F811
    # both sides of the lines: in FP64 (one persistent CTA a multiprocessor) 40
    # tiles a CTA, or 28 with 100 particles a tile, in FP32 (three) 16; the
    # sparse tiles in their own kernel, or every tile staged
    torch = pytest.importorskip("torch")
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = shape[0] * shape[1] * shape[2] // 512
    if n_sm != 152:
        pytest.skip("the shapes are chosen for 152 multiprocessors")
    g = dict(inputs.random_grid(211, *shape), boundary=1)
    # four fifths of the particles in the lower half: sparse and dense tiles
    P = dict(inputs.random_particles(212, g, per_tile * tiles, u_scale=0.2), q_macro=-1e-16)
    far = np.random.default_rng(213).random(len(P["z"])) < 0.6
    P["z"] = np.where(far & (P["z"] > g["nz"] / 2 * g["dz"]), P["z"] - (g["nz"] / 2 - 2) * g["dz"], P["z"])
    names = kernels_of_a_step(M, g, P, prec, tmp_path / "step")
    assert ("k_push_sparse" in names) == there
    check(M, orc, g, None, P, prec, (1, 3))


def test_staged_threshold_launches_no_sparse_kernel(M, tmp_path):  # noqa: F811
    g = dict(inputs.random_grid(221, 32, 24, 24), boundary=1)
    P = inputs.random_particles(222, g, 500, u_scale=0.2)
    for below, there in ((0, False), (1, False), (2, True), (1 << 30, True)):
        names = kernels_of_a_step(M, g, P, "P32", tmp_path / str(below), push_sparse_below=below)
        assert "k_push_tiled" in names and ("k_push_sparse" in names) == there, below


@pytest.mark.parametrize("prec", ["P32", "P64"])
def test_timed_steps_with_sparse_tiles(M, prec):  # noqa: F811
    # the particle step's timed scope holds both its kernels side by side:
    # timed steps, with power and bunch records, leave what untimed ones do
    g = dict(inputs.random_grid(231, 40, 40, 48), boundary=1)
    P = dict(inputs.random_particles(232, g, 30000, u_scale=0.3), q_macro=-1e-17)
    tol = 1e-11 if prec == "P64" else 1e-5
    recs = []
    with M.Simulation(g, None, P, precision=getattr(M, prec)) as a, \
            M.Simulation(g, None, P, precision=getattr(M, prec)) as b:
        for s in (a, b):
            s.set_tuning(push_sparse_below=100)
            s.set_power_sampling(40, 20)
            s.set_bunch_sampling(1.0e3, 1, 20)
        a.profile(True)
        a.step(9)
        kt = a.kernel_times()
        assert kt["push"][1] == 9 and kt["push"][0] > 0.0
        b.step(9)
        for s in (a, b):
            recs.append((s.read_power(), s.read_bunch()))
        for x, y in zip(*recs):
            assert x.shape == y.shape and len(x) == 9
            assert (np.abs(x - y) <= tol * np.abs(y).max(0) + 1e-30).all()
        pa, pb = a.copy_particles(), b.copy_particles()
        for nm in ("x", "uz"):
            assert np.abs(pa[nm] - pb[nm]).max() <= tol * np.abs(pb[nm]).max()


@pytest.mark.parametrize("prec", ["P32", "P32_U64", "P64"])
@pytest.mark.parametrize("shape,n,tuning", [
    ((32, 32, 64), 500, {}), ((33, 32, 64), 500, {}), ((64, 64, 320), 2000, {}),
    ((65, 65, 256), 0, {}), ((128, 64, 264), 2000, dict(push_sparse_below=16)),
    ((64, 128, 280), 250000, {}), ((64, 128, 400), 2000, {}), ((128, 128, 240), 2000, {}),
    ((128, 128, 240), 2000, dict(push_ctas_per_sm=1, stencil_variant=0)),
    ((48, 48, 48), 500, dict(push_variant=0))])
def test_kernels_that_the_bench_counts(M, prec, shape, n, tuning, tmp_path):  # noqa: F811
    # bench.kernels_of against the kernels of a captured step: each form of the
    # update, of the particle step and of the re-sort
    from test_replicas_cpu import _bench
    g = dict(inputs.random_grid(241, *shape), boundary=1)
    P = inputs.random_particles(242, g, n, u_scale=0.2) if n else None
    names = kernels_of_a_step(M, g, P, prec, tmp_path / "step", **tuning)
    full = dict(stencil_variant=2, lz=0, push_variant=1, push_ctas_per_sm=0, push_sparse_below=0)
    full.update(tuning)
    scopes = ["potential_step"] + (["push", "scan_counts", "slot_map"] if n else [])
    count = sum(_bench().kernels_of(k, 1, g, n, prec.lower(), full) for k in scopes)
    found = re.findall(r"6mithra\d+(k_[a-z_0-9]+?)(?=[IE])", names)
    # (without particles, the kernel that advances the step counter)
    assert len(found) == count + (0 if n else 1), (count, found)


@pytest.mark.parametrize("prec,nx", [("P32", 64), ("P32_C", 64), ("P32_C", 67)])
def test_ring_runs_agree(M, prec, nx):  # noqa: F811
    # runs from one plane (fewer planes than stages) to more than the grid has:
    # the same arithmetic whatever the run, to the bit
    g = dict(inputs.random_grid(251, nx, 62, 275), boundary=1)
    f = smooth_levels(g)
    n = nx * 62 * 275
    out = {}
    for lz in (0, 1, 2, 3, 16, 300):
        with M.Simulation(g, None, None, precision=getattr(M, prec)) as sim:
            sim.set_tuning(lz=lz)
            for a, nm in enumerate(("Ax", "Ay", "Az", "phi")):
                sim.set_field(nm + "_prev", f["prev"][a * n:(a + 1) * n])
                sim.set_field(nm, f["cur"][a * n:(a + 1) * n])
            sim.step(5)
            out[lz] = [sim.copy_field(nm) for nm in ("Ax", "phi", "Az_prev")]
    for lz, fields in out.items():
        assert all(np.array_equal(a, b) for a, b in zip(fields, out[0])), lz
