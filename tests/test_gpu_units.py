"""Unit tables of every form give a run the same bits: units cut into parts with the
Yee update inside the push (few particles in the batch), and whole units with a Yee
launch of their own (the same run beside a large one); and a sort whose groups hold
more units than its planning kernel stages."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def picrr():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1008_1685_gb300 as m

    return m


def state(b, run):
    out = [b.field(run, c) for c in range(8)]
    for sp in (0, 1):
        q = b.particles(run, sp)
        out += [q[k] for k in ("x", "px", "py", "pz", "flag")]
    return out, b.energy(run)


# foils of 1 to 256 particles per cell: fewer particles than one part, one more than a
# part, several units per tile, a foil at the wall whose hot electrons freeze there
@pytest.mark.parametrize("cells,foil,ppc,interval,steps", [(64, (20, 16), 1, 8, 40), (500, (20, 57), 9, 8, 41),
                                                           (500, (30, 200), 64, 8, 43), (700, (16, 40), 256, 5, 60),
                                                           (520, (12, 500), 33, 16, 150)])
def test_few_and_many_units_give_the_same_bits(picrr, cells, foil, ppc, interval, steps):
    cpl = 100.0
    run = dict(length_lambda=cells / cpl, foil_x0=foil[0] / cpl, foil_thickness=foil[1] / cpl, ne=20.0, a0=80.0,
               polarization=picrr.CP, duration=3.0, steps=10**9, ppc=ppc, seed=5)
    alone = picrr.Batch(cpl, max_runs=1, sort_interval=interval)
    ra = alone.add_run(**run)
    # 5.2M particles: more than 1216 units of 4096
    beside = picrr.Batch(cpl, max_runs=2, sort_interval=interval)
    beside.add_run(length_lambda=20.0, foil_x0=1.0, foil_thickness=10.0, ne=1.0, a0=1.0, polarization=0, duration=3.0,
                   steps=10**9, ppc=2600, seed=6)
    rb = beside.add_run(**run)
    for n in (3, steps - 3):
        assert alone.step(n) == n and beside.step(n) == n
        (a, ea), (b, eb) = state(alone, ra), state(beside, rb)
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
        assert np.array_equal(ea[[0, 1, 2, 4, 5]], eb[[0, 1, 2, 4, 5]])
        assert eb[3] == pytest.approx(ea[3], rel=1e-12, abs=1e-300)
    assert alone.stats()["n_units"] > 0 and beside.stats()["n_units"] > 1216
    alone.close()
    beside.close()


def test_units_cut_to_even_parts_give_the_same_bits(picrr):
    """5.2M particles beside, units of 16384, 2 particles per thread: parts of 4096 (and whole units again with 4)."""
    cpl, run = 100.0, dict(length_lambda=6.0, foil_x0=0.3, foil_thickness=4.0, ne=20.0, a0=80.0, polarization=picrr.CP,
                           duration=3.0, steps=10**9, ppc=300, seed=5)
    alone = picrr.Batch(cpl, max_runs=1, sort_interval=8)
    ra = alone.add_run(**run)
    alone.set_shapes(16384, 8, 2)
    beside = picrr.Batch(cpl, max_runs=2, sort_interval=8)
    beside.add_run(length_lambda=20.0, foil_x0=1.0, foil_thickness=10.0, ne=1.0, a0=1.0, polarization=0, duration=3.0,
                   steps=10**9, ppc=2600, seed=6)
    rb = beside.add_run(**run)
    units = []
    for w in (4, 2):
        beside.set_shapes(16384, 8, w)
        units.append(beside.stats()["n_units"])
    assert units[1] > 1.8 * units[0]
    for n in (8, 11):
        assert alone.step(n) == n and beside.step(n) == n
        for x, y in zip(state(alone, ra)[0], state(beside, rb)[0]):
            assert np.array_equal(x, y)
    alone.close()
    beside.close()


@pytest.mark.parametrize("first", [1024, 16384])
def test_table_in_use_shrinks_and_grows(picrr, first):
    """Units of 1024, then of 16384 (fewer entries in use), then a run that joins: as that run alone."""
    cpl, run = 100.0, dict(length_lambda=6.0, foil_x0=0.3, foil_thickness=4.0, ne=20.0, a0=80.0, polarization=picrr.CP,
                           duration=3.0, steps=10**9, ppc=300, seed=5)
    alone = picrr.Batch(cpl, max_runs=1, sort_interval=8)
    ra = alone.add_run(**run)
    alone.set_shapes(16384, 8, 4)
    beside = picrr.Batch(cpl, max_runs=2, sort_interval=8)
    beside.add_run(length_lambda=20.0, foil_x0=1.0, foil_thickness=10.0, ne=1.0, a0=1.0, polarization=0, duration=3.0,
                   steps=10**9, ppc=2600, seed=6)
    for unit in (first, 16384):
        beside.set_shapes(unit, 8, 4)
        assert beside.step(8) == 8
    rb = beside.add_run(**run)
    for n in (8, 19):
        assert alone.step(n) == n and beside.step(n) == n
        for x, y in zip(state(alone, ra)[0], state(beside, rb)[0]):
            assert np.array_equal(x, y)
    alone.close()
    beside.close()


def test_more_units_in_a_group_than_are_staged(picrr):
    """1400 units of 1024 particles in 600 cells: the planning kernel reads their bounds from
    the table.  Shapes change the order of single-precision sums only: fields of order 1 after
    17 steps differ by at most 17 x 2^-24 x a few hundred terms, below 1e-4."""
    n, cpl = 700_000, 500.0
    r = np.random.default_rng(3)
    cell = np.sort(r.integers(30, 630, n)).astype(np.int32)
    off = r.random(n, dtype=np.float32)
    p = [(r.normal(size=n) * 0.5).astype(np.float32) for _ in range(3)]
    res = []
    for unit in (1024, 16384):
        g = picrr.Sim(1.4, cpl, sort_interval=8)
        for sp, (q, m) in enumerate(((-1.0, 1.0), (1.0, 1836.15267343))):
            g.load_particles_f32(sp, cell, off, *p, 0.01, q, m)
        g.inject_laser(30.0, picrr.CP, picrr.ENV_SIN2, 2.0)
        g.set_shapes(unit, 8, 2)
        assert g.step(17) == 17
        assert (g.stats()["n_units"] > 1300) == (unit == 1024)
        q = g.particles(0)
        res.append([g.field(c) for c in range(5)] + [q["x"], q["px"]])
        g.close()
    for a, b in zip(*res):
        assert np.max(np.abs(a - b)) <= 1e-4 * max(1.0, np.max(np.abs(b)))


@pytest.mark.parametrize("slots", [2, 4])
@pytest.mark.parametrize("sign,planar", [(1.0, False), (-1.0, False), (1.0, True)])
@pytest.mark.parametrize("n,cells,spread", [(4001, 1, 0.0), (40_003, 5, 0.0), (40_003, 5, 3.0), (9_001, 3, 30.0)])
def test_window_words_wrap(picrr, n, cells, spread, sign, planar, slots):
    """Thousands of particles a cell drifting one way, cold (all lanes in one cell) and hot (anchors change
    from particle to particle): a particle's record is up to 2^22 of the window's units, so the 32-bit words
    wrap many times.  Against the oracle: each value carries a few roundings of 2^-24 (weights, 1/gamma,
    product) and 2^-23 of the record: below 2e-6 also if they all go one way."""
    import oracle

    kw = dict(length_lambda=2, cells_per_lambda=100, cfl=0.95, lambda_um=0.8, source_node=8)
    g, o = picrr.Sim(seed=1, sort_interval=8, **kw), oracle.OracleSim(**kw)
    r = np.random.default_rng(n)
    cell = (100 + r.integers(0, cells, n)).astype(np.int32)
    off = r.random(n)
    p = [sign * d + spread * r.normal(size=n) for d in (1.1, -2.3, 1.7)]
    if planar:  # no Jz, as with linear polarization
        p[2] = 0 * p[2]
    for s in (g, o):
        s.load_particles(0, cell, off, *p, 0.01, -1.0, 1.0)
        s.load_particles(1, cell[:1], off[:1], *(v[:1] * 0 for v in p), 1e-6, 1.0, 1836.0)
    g.set_shapes(4096, 8, slots)
    g.step(1)
    o.step(1)
    for c in (5, 6, 7):
        a, b = g.field(c), o.field(c)
        assert np.linalg.norm(a - b) <= 2e-6 * np.linalg.norm(b), c
    g.close()


@pytest.mark.parametrize("steps", [48, 45])  # (the pulse is in the foil) the last step ends a sort interval, or lies inside one
def test_currents_stay_readable_when_a_large_run_ends(picrr, steps):
    """A run of 488 units ends on the last step of a call, the small run beside it goes on: from
    then on its steps take another form, but its last current is still that of the run alone."""
    cpl, small = 100.0, dict(length_lambda=6.0, foil_x0=0.3, foil_thickness=4.0, ne=20.0, a0=80.0, polarization=picrr.CP,
                             duration=3.0, steps=10**9, ppc=30, seed=5)
    alone, beside = (picrr.Batch(cpl, max_runs=m, sort_interval=8) for m in (1, 2))
    beside.add_run(length_lambda=20.0, foil_x0=1.0, foil_thickness=10.0, ne=1.0, a0=1.0, polarization=0, duration=3.0,
                   steps=steps, ppc=1000, seed=6)
    ra, rb = alone.add_run(**small), beside.add_run(**small)
    for b in (alone, beside):
        assert b.step(steps) == steps
    for n in (0, 1, 9):
        assert alone.step(n) == n and beside.step(n) == n
        for c in range(8):
            f = alone.field(ra, c)
            assert np.array_equal(f, beside.field(rb, c)), (n, c)
            assert c not in (5, 6, 7) or np.any(f)
    alone.close()
    beside.close()


def test_few_runs_in_a_batch_of_many_slots(picrr):
    """Three of 4000 slots, with released ones before and between them, of different lengths."""
    cpl = 100.0
    runs = [dict(length_lambda=l, foil_x0=0.3, foil_thickness=0.7 * l, ne=20.0, a0=80.0, polarization=picrr.CP, duration=3.0,
                 steps=10**9, ppc=20, seed=7 + k) for k, l in enumerate((6.0, 23.0, 2.5))]
    b = picrr.Batch(cpl, max_runs=4000, sort_interval=8)
    ids = []
    for k in range(9):
        r = b.add_run(**runs[k // 3])
        if k % 3 == 2:
            ids.append(r)
        else:
            b.step(0)  # starts it
            b.stop_run(r)
            b.release_run(r)
            b.add_run(**runs[k // 3])  # the slot's next run stays
    b.step(45)
    for r, kw in zip(ids, runs):
        a = picrr.Batch(cpl, max_runs=1, sort_interval=8)
        ra = a.add_run(**kw)
        a.step(45)
        (x, ex), (y, ey) = state(a, ra), state(b, r)
        assert all(np.array_equal(p, q) for p, q in zip(x, y))
        assert ey[3] == pytest.approx(ex[3], rel=1e-12, abs=1e-300)
        a.close()
    b.close()


@pytest.mark.parametrize("cells", [200_003, 17_000_001])  # 782 and 66,408 groups of 512 cells, both species
def test_long_boxes(picrr, cells):
    """Hardly any charge: every particle flies straight on, each step exactly once, through sorts and new
    tables over the whole box.  A step rounds the offset (2^-24) and the velocity (4 x 2^-24, times 0.95): 40
    steps stay below 1.2e-5 cells."""
    n, steps, dx = 60_000, 40, 2 * np.pi / 500.0
    r = np.random.default_rng(cells)
    g = picrr.Sim(cells / 500.0, 500.0, cfl=0.95, sort_interval=8, source_node=8)
    want = []
    for sp, (q, m) in enumerate(((-1.0, 1.0), (1.0, 1836.15267343))):
        cell = np.sort(r.integers(100, cells - 100, n)).astype(np.int32)
        off = r.random(n, dtype=np.float32)
        p = [(3.0 * r.normal(size=n)).astype(np.float32) for _ in range(3)]
        g.load_particles_f32(sp, cell, off, *p, 1e-25, q, m)
        p = [v.astype(float) for v in p]
        want.append(cell + off.astype(float) + steps * 0.95 * p[0] / np.sqrt(1 + p[0] ** 2 + p[1] ** 2 + p[2] ** 2))
    assert g.step(steps) == steps
    assert 2 * n // 512 < g.stats()["n_units"] <= 2 * (n // 512 + (cells + 511) // 512 + 1)
    for sp in (0, 1):
        assert np.max(np.abs(g.particles(sp)["x"] / dx - want[sp])) < 1.2e-5
    g.close()


def test_steps_of_long_boxes_are_not_fused(picrr):
    """Fused, an interval of 8 steps is 8 pushes, one Yee launch and 3 for the sort, else 8 Yee launches; the
    bits are the same in boxes that differ by a cell at the far end."""
    res = []
    for cells, launches in ((194_559, 12), (194_560, 19)):  # 760 and 761 Yee blocks
        g = picrr.Sim(cells / 500.0, 500.0, cfl=0.95, sort_interval=8, source_node=8, seed=3)
        g.load_foil(0.2, 1.0, 20.0, 1, 1.0, 20)
        g.inject_laser(80.0, picrr.CP, picrr.ENV_SIN2, 3.0)
        g.step(8)
        n = g.stats()["kernel_launches"]
        g.step(160)
        assert g.stats()["kernel_launches"] - n == 20 * launches
        q = g.particles(0)
        res.append([g.field(c)[:150_000] for c in range(8)] + [q[k] for k in ("x", "px", "py", "pz")])
        g.close()
    for a, b in zip(*res):
        assert np.any(a) and np.array_equal(a, b)


@pytest.mark.parametrize("npt", [1, 4])  # nodes per thread of the Yee kernel; 2 in the library
def test_other_yee_blocks_give_the_same_bits(picrr, tmp_path, npt):
    """The build option changes which block updates a node, in the kernel of its own and inside the push."""
    code = """
import sys
import numpy as np
from paper_1008_1685_gb300 import binding, build
npt, out = sys.argv[1:]
if npt != "2":
    build.LIB, build.BUILD = out + ".so", out + "_build"
    binding._LIB_PATH = build.build(force=True, extra=["-DPICRR_FIELD_NPT=" + npt])
res = []
for cells, slots in ((500, 2), (1153, 2), (1153, 4)):
    g = binding.Sim(cells / 100.0, 100.0, sort_interval=8, seed=4)
    g.load_foil(0.3, 3.0, 20.0, 1, 1.0, 20)
    g.inject_laser(80.0, binding.CP, binding.ENV_SIN2, 3.0)
    g.set_shapes(4096, 8, slots)
    g.step(150)
    res += [g.field(c) for c in range(8)] + [g.energy()[[0, 1, 2, 4, 5]]]
    g.close()
np.savez(out, *res)
"""
    import os
    import subprocess
    import sys

    root = os.path.dirname(os.path.dirname(os.path.abspath(picrr.__file__)))
    got = []
    for v in ("2", str(npt)):
        out = str(tmp_path / ("npt" + v))
        subprocess.run([sys.executable, "-c", code, v, out], cwd=root, check=True)
        with np.load(out + ".npz") as z:
            got.append([z[k] for k in z.files])
    for a, b in zip(*got):
        assert np.any(a) and np.array_equal(a, b)


@pytest.mark.parametrize("unit", [1024, 4096])
def test_small_units_are_fused_like_the_default_s(picrr, unit):
    g = picrr.Sim(20.0, 500.0, cfl=0.95, sort_interval=8, source_node=8, seed=3)
    g.load_foil(0.2, 1.0, 20.0, 1, 1.0, 600)  # 600,000 particles
    g.set_shapes(unit, 8, 2)
    g.step(8)
    n = g.stats()["kernel_launches"]
    g.step(80)
    assert g.stats()["kernel_launches"] - n == 10 * 12
    g.close()
