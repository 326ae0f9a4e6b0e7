"""The spectrum and kinetic-energy kernels at the sizes and values where they can
go wrong: ragged counts, unaligned arrays, shared and global counters, momenta on
bin edges, zero, subnormal, huge, infinite and NaN.  Bins are decided by the double
evaluation floor((E - e_min) / (e_max - e_min) * nbins), so counts are compared for
equality with numpy's doubles; the energy sum with an extended-precision sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ME_MEV = 0.51099895000


@pytest.fixture(scope="module")
def picrr():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1008_1685_gb300 as m

    return m


def energies(p, mass_me):
    with np.errstate(all="ignore"):
        x, y, z = (v.astype(np.float64) for v in p)
        p2 = x * x + y * y + z * z
        return (mass_me * ME_MEV) * p2 / (np.sqrt(1.0 + p2) + 1.0)


def counts(e, nbins, lo, hi):
    with np.errstate(all="ignore"):
        kf = np.floor((e - lo) / (hi - lo) * nbins)
        k = kf[~(e < lo) & (kf < nbins)].astype(np.int64)
    return np.bincount(k, minlength=nbins).astype(np.float64)


def momenta(n, scale, seed):
    r = np.random.default_rng(seed)
    p = [(r.normal(size=n) * scale * 10.0 ** r.uniform(-3, 0, n)).astype(np.float32) for _ in range(3)]
    odd = np.array([0.0, 1e-42, 1e-20, 1e-13, 1e12, 3e15, 1e19, 1e30, np.inf, -np.inf, np.nan], dtype=np.float32)
    at = r.permutation(n)[: min(n, 4 * len(odd))]
    p[0][at] = np.resize(odd, len(at))
    for q in p[1:]:
        q[at[::2]] = 0.0
    return p


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 4097, 300_001])
@pytest.mark.parametrize("nbins,lo,hi,mass", [(1, 0.0, 5.0, 1.0), (200, 0.0, 60.0, 1.0), (200, -3.0, 7.0, 1.0),
                                              (777, 2.5, 40.0, 1.0), (8190, 0.0, 60.0, 1.0), (8191, 0.0, 60.0, 1.0),
                                              (65536, 0.01, 3e4, 1836.15267343)])
def test_bins_equal_the_double_evaluation(picrr, n, nbins, lo, hi, mass):
    torch = pytest.importorskip("torch")
    from paper_1008_1685_gb300 import binding

    p = momenta(n, 100.0, 1000 + n + nbins)
    e = energies(p, mass)
    mid = np.sort(e[np.isfinite(e) & (e > lo)])
    if lo == 0.0 and len(mid) > 2:  # put one particle's energy on an edge, up to rounding
        hi = float(mid[len(mid) // 2]) * nbins / max(1, nbins // 3)
    for shift in (0, 1):  # 16-byte aligned arrays, and arrays that start one element later
        dev = [torch.cat([torch.zeros(shift), torch.from_numpy(q)]).cuda()[shift:] for q in p]
        out = torch.full((nbins,), -1.0, dtype=torch.float64, device="cuda")
        rc, msg = binding.spectrum_noalloc(*[q.data_ptr() for q in dev], n, mass, 1.0, nbins, lo, hi, out.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream)
        assert rc == 0, msg
        got = np.rint(out.cpu().numpy() * ((hi - lo) / nbins))
        assert np.array_equal(got, counts(e, nbins, lo, hi)), (n, nbins, shift)


@pytest.mark.parametrize("n", [1, 3, 4, 1023, 8193, 300_002])
@pytest.mark.parametrize("kind", ["thermal", "cold", "beam", "tiny", "huge"])
def test_kinetic_sum(picrr, n, kind):
    """At most about 60 double additions lie between a particle and the sum (8 per
    round and thread, 5 + 8 in a block, 1 + 5 + 32 over blocks): 60 x 2^-53 = 7e-15."""
    r = np.random.default_rng(n)
    s = dict(thermal=1.0, cold=0.0, beam=0.0, tiny=1e-16, huge=1e21)[kind]
    p = [(r.normal(size=n) * s).astype(np.float32) for _ in range(3)]
    if kind == "beam":
        p[0][:] = np.float32(0.7310586)
    g = picrr.Sim(4.0, 100.0)
    cell = np.full(n, 100, dtype=np.int32)
    g.load_particles_f32(0, cell, np.zeros(n, dtype=np.float32), *p, 0.5, -1.0, 1.0)
    got = g.energy()[1]
    x, y, z = (v.astype(np.longdouble) for v in p)
    p2 = x * x + y * y + z * z
    want = float(np.sum(p2 / (np.sqrt(1 + p2) + 1)) * np.longdouble(0.5) * np.longdouble(g.dx))
    assert abs(got - want) <= 1e-14 * want, (got, want)
    g.close()
