"""The radial table at its first cell: walkers one lattice step from a nucleus
along their own rotated axes, so that the move back lands on it and the squared
distance is a rounding residue of either sign, at most 2^-44 h^2. Without an
e-n Jastrow factor (whose cusp would turn the residue into its square root) the
rate is the radial part's, where a primitive of exponent alpha turns the
residue into a relative error of alpha 2^-44 h^2: rates against the FP64 oracle
within 1e-10 of their scale and this bound for the tightest exponent."""
import numpy as np
import pytest

import lrdmc_synth as S

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


@pytest.mark.parametrize("tight", [3e4, 2e7, 3e9, 2e11])
def test_moves_onto_a_nucleus_from_all_axes(pkg, tight):
    import oracle

    rng = np.random.default_rng(5)
    alpha = 0.06 * (tight / 0.06) ** (np.arange(6) / 5)
    system = S.System(name="tight", nuc_xyz=np.zeros((1, 3)), Z=np.array([2.0]), n_up=1, n_dn=1,
                      shells=[S.Shell(0, 0, S.GTO, alpha=list(alpha), coef=list(rng.uniform(0.2, 1.0, 6)))],
                      C=np.ones((1, 1)), en_b1=np.array([0.0]), orbital_shell=[0])
    W, a, seed = 60, 0.12, 9
    x0, rot = np.zeros((W, 2, 3)), []
    for w in range(W):
        bits = oracle.philox4x64([w, 2 ** 64 - 1, 0, 1], [seed, 0])
        rot.append(oracle.rotation(*[oracle.uniform(b) for b in bits[:3]]))
        x0[w, 0] = (-a if w % 2 else a) * np.asarray(rot[w]).reshape(3, 3)[:, w % 3]
        x0[w, 1] = rng.normal(size=3)
    g = pkg.LrdmcSystem(system)
    g.init_walkers(x0, seed=seed, tau=1e-13, trace_capacity=4)  # no walker jumps within tau
    g.step(1, a, pkg.Spacing(pkg.SINGLE))
    got = g.walkers()
    assert np.all(got["jumps_pre"] == 0)
    o = oracle.OracleSystem(system)
    lat = oracle.lattice_for(system, a, oracle.SINGLE)
    for t in range(W):
        w = int(got["parent"][t])
        ref = o.lattice_eval(lat, x0[w], rot[w])["T"]
        tol = np.full(12, 1e-10)
        tol[2 * (w % 3) + (0 if w % 2 else 1)] += tight * 2.0 ** -44 * a * a
        assert np.all(np.abs(got["T"][t] - ref) <= tol * np.maximum(ref, 0.5 / a ** 2)), w
