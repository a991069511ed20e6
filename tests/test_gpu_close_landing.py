"""FP64 mode: a lattice move that lands close to another electron or on it, from
both spin blocks, against the FP64 oracle. The landing point and the partner
round to 2^-53 of a coordinate each, which the Pade factor's slope of at most
1/2 passes on, so the ratio keeps the digits of any other one: 1e-12 of its own
floating-point scale, a hundred times what the inverses' rounding leaves."""
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


@pytest.mark.parametrize("distance", [0.0, 1e-10, 1e-8, 1e-6, 1e-3])
@pytest.mark.parametrize("name", ["He", "Ne"])
def test_moves_that_land_close_to_an_electron(pkg, name, distance):
    import oracle

    system, a, n = S.make_system(name), 0.2, 6
    x, R = S.initial_positions(system, n, 31), S.random_rotations(n, 32)
    o = oracle.OracleSystem(system)
    lat = oracle.lattice_for(system, a, oracle.PREVIOUS)
    rng = np.random.default_rng(33)
    for c in range(n):
        axis = R[c].reshape(3, 3)[:, c % 3]
        away = rng.normal(size=3)
        h = lat.a if c < 3 else lat.ap
        i, j = (0, system.n_up) if c % 2 else (system.n_up, 0)
        x[c, j] = x[c, i] + (-h if c % 2 else h) * axis + distance * away / np.linalg.norm(away)
    g = pkg.LrdmcSystem(system).set_precision(pkg.PRECISION_FP64)
    ratio = g.evaluate(torch.tensor(x, device="cuda"), torch.tensor(R, device="cuda"), a,
                       pkg.Spacing(pkg.PREVIOUS))[0].cpu().numpy()
    for c in range(n):
        ref = o.lattice_eval(lat, x[c], R[c])["ratio"]
        scale = U.ratio_scale(o, system, lat, x[c], R[c], ref)
        i = system.n_up if c % 2 == 0 else 0
        k = (i * 2 + (0 if c < 3 else 1)) * 6 + 2 * (c % 3) + (1 if c % 2 else 0)
        # the move onto the partner: the pair's own term is exact to its slope
        assert abs(ratio[c, k] - ref[k]) <= 1e-12 * scale[k], (c, ratio[c, k], ref[k])
