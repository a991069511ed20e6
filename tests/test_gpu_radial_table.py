"""The radial table of contracted Gaussian shells (double-float projection):
rates of walkers at their start positions, whose electrons sit from 1e-7 bohr
from a nucleus to far beyond the last cell of the tight shells, against the
FP64 oracle. Contractions of 3, 4 and 8 primitives (tabulated; exponents
spanning up to 10^6, s, p and d) beside one of 2 (summed directly), and two
nuclei. The tolerance is the evaluation tests': 1e-10 of each rate's own
floating-point scale, and the exponential's cutoff."""
import numpy as np
import pytest

import lrdmc_synth as S
import _parity_util as U

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1909_01589_gb300 import build

    build.build()
    import paper_1909_01589_gb300 as p

    p.load_library()
    return p


def _system():
    rng = np.random.default_rng(2)

    def gto(c, l, lo, hi, n):
        return S.Shell(c, l, S.GTO, alpha=list(lo * (hi / lo) ** (np.arange(n) / max(n - 1, 1))),
                       coef=list(rng.uniform(0.2, 1.0, n)))

    shells = [gto(0, 0, 0.05, 5e4, 8), gto(0, 1, 0.08, 2.0, 3), gto(0, 0, 3.0, 1e4, 4), gto(0, 2, 0.1, 1.5, 3),
              gto(1, 0, 0.11, 0.9, 2), gto(1, 0, 0.07, 70.0, 5)]
    n_ao = sum(2 * s.l + 1 for s in shells)
    C = rng.normal(size=(n_ao, 2))
    return S.System(name="table", nuc_xyz=np.array([[0.0, 0.0, 0.0], [0.4, 1.3, -0.7]]), Z=np.array([4.0, 1.0]),
                    n_up=2, n_dn=2, shells=shells, C=C, en_b1=np.array([4.0, 1.0]), en_b2=4.0, orbital_shell=[0, 1])


@pytest.mark.parametrize("kind", ["single", "this_work"])
def test_tabulated_rates_match_oracle(pkg, kind):
    import oracle

    system, a, seed = _system(), 0.12, 9
    rng = np.random.default_rng(4)
    r = np.array([1e-7, 1e-4, 0.003, 0.02, 0.11, 0.35, 0.8, 1.7, 2.9, 4.4, 6.1, 8.0, 9.5, 11.0])
    x0 = np.zeros((24, 4, 3))
    for w in range(len(x0)):
        for i in range(4):
            v = rng.normal(size=3)
            x0[w, i] = system.nuc_xyz[(w + i) % 2] + r[(3 * w + 5 * i) % len(r)] * v / np.linalg.norm(v)
    g = pkg.LrdmcSystem(system)
    sp = pkg.Spacing(pkg.SINGLE if kind == "single" else pkg.THIS_WORK)
    g.init_walkers(x0, seed=seed, tau=1e-13, trace_capacity=4)  # no walker jumps within tau
    g.step(1, a, sp)
    got = g.walkers()
    assert np.all(got["jumps_pre"] == 0)
    o = oracle.OracleSystem(system)
    lat = oracle.lattice_for(system, a, oracle.SINGLE if kind == "single" else oracle.THIS_WORK)
    for t in range(len(x0)):
        w = int(got["parent"][t])
        bits = oracle.philox4x64([w, 2 ** 64 - 1, 0, 1], [seed, 0])
        R = oracle.rotation(*[oracle.uniform(b) for b in bits[:3]])
        ref = o.lattice_eval(lat, x0[w], R)
        scale = U.ratio_scale(o, system, lat, x0[w], R, ref["ratio"])
        tol = U.rate_tolerance(lat, ref["w"], scale, w_abs=U.W_ABS)
        assert np.all(np.abs(got["T"][t] - ref["T"]) <= tol), (w, np.max(np.abs(got["T"][t] - ref["T"]) / tol))


def test_table_reaches_a_population_of_another_stream(pkg):
    """A system whose table was made in one stream and that takes a new
    population in another stream: the same walkers bit for bit."""
    rng = np.random.default_rng(2)
    x0 = rng.normal(size=(64, 4, 3))

    def project(g):
        g.init_walkers(x0, seed=3, tau=0.02, trace_capacity=8)
        g.step(2, 0.12, pkg.Spacing(pkg.THIS_WORK))
        return g.walkers()

    want = project(pkg.LrdmcSystem(_system()))
    g = pkg.LrdmcSystem(_system())
    for _ in range(2):
        with torch.cuda.stream(torch.cuda.Stream()):
            got = project(g)
        for key in want:
            assert np.array_equal(np.asarray(got[key]), np.asarray(want[key])), key
