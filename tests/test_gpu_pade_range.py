"""The e-e Pade factor at the ends of the range of b that create_system takes:
vanishing, negative and huge ones, with electron pairs from 1e-4 to 10 bohr apart,
against the FP64 oracle. Tolerances are the evaluation tests': 1e-10 of each
ratio's own floating-point scale, 1e-8 of the local energy (or 1e-10 of its
terms' magnitude, where the close pair's repulsion makes them large)."""
import dataclasses

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


def _positions(system):
    x = S.initial_positions(system, 3, 7)
    x[1, system.n_up] = x[1, 0] + np.array([6e-5, -8e-5, 0.0])
    x[2, 1] += np.array([0.0, 6.0, 8.0])
    return x


@pytest.mark.parametrize("b", [1e-300, 1e-40, 1e-20, -1e-19, 1e-16, 1e-9, -1e-3, 1e6, 1e10, 1e20, 1e30])
@pytest.mark.parametrize("name", ["He", "Ne"])
@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32"])
def test_extreme_pade_parameters(pkg, prec, name, b):
    import oracle

    system = dataclasses.replace(S.make_system(name), b_ee=b)
    g = pkg.LrdmcSystem(system).set_precision({"fp64": pkg.PRECISION_FP64, "df64": pkg.PRECISION_DF64,
                                               "fp32": pkg.PRECISION_FP32}[prec])
    o = oracle.OracleSystem(system)
    lat = oracle.lattice_for(system, 0.1, oracle.THIS_WORK)
    x, R = _positions(system), S.random_rotations(3, 12)
    ratio, _, _, el = (q.cpu().numpy() for q in g.evaluate(torch.tensor(x, device="cuda"),
                                                           torch.tensor(R, device="cuda"), 0.1,
                                                           pkg.Spacing(pkg.THIS_WORK)))
    refs = [o.lattice_eval(lat, x[c], R[c]) for c in range(3)]
    scale_el = U.el_scale(system, x, np.array([r["EL"] for r in refs]))
    for c, ref in enumerate(refs):
        assert abs(el[c] - ref["EL"]) <= max(1e-8 * max(abs(ref["EL"]), 1.0), 1e-10 * scale_el[c]), c
        if prec == "fp32":
            # a fraction of sixteen single-precision factors 1 + b r: to b r = 200
            if b <= 100.0:
                assert np.all(np.abs(ratio[c] - ref["ratio"]) <= 2e-4 * np.maximum(np.abs(ref["ratio"]), 1.0)), c
        else:
            scale = U.ratio_scale(o, system, lat, x[c], R[c], ref["ratio"])
            assert np.all(np.abs(ratio[c] - ref["ratio"]) <= 1e-10 * scale), c
