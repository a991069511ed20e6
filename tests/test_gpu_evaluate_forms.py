"""The evaluation kernels' branches against the FP64 oracle: the e-e Pade sum
in the reciprocal form (b >= 1/4), term by term (below) and with b = 0, and the
shapes of an evaluation block (one configuration per block, two, and the full
ones, with a ragged last block). The tolerance is the evaluation tests': 1e-10
of each ratio's own floating-point scale (2e-4 of max(|ratio|, 1) in the mixed
mode)."""
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


def _check(pkg, system, prec, n, a=0.1):
    import oracle

    g = pkg.LrdmcSystem(system).set_precision({"fp64": pkg.PRECISION_FP64, "df64": pkg.PRECISION_DF64,
                                               "fp32": pkg.PRECISION_FP32}[prec])
    o = oracle.OracleSystem(system)
    lat = oracle.lattice_for(system, a, oracle.THIS_WORK)
    x, R = S.initial_positions(system, n, 11), S.random_rotations(n, 12)
    ratio, _, _, el = (q.cpu().numpy() for q in g.evaluate(torch.tensor(x, device="cuda"),
                                                           torch.tensor(R, device="cuda"), a,
                                                           pkg.Spacing(pkg.THIS_WORK)))
    for c in sorted({0, n // 2, n - 2, n - 1} & set(range(n))):
        ref = o.lattice_eval(lat, x[c], R[c])
        if prec == "fp32":
            assert np.all(np.abs(ratio[c] - ref["ratio"]) <= 2e-4 * np.maximum(np.abs(ref["ratio"]), 1.0)), c
        else:
            scale = U.ratio_scale(o, system, lat, x[c], R[c], ref["ratio"])
            assert np.all(np.abs(ratio[c] - ref["ratio"]) <= 1e-10 * scale), c
        assert abs(el[c] - ref["EL"]) <= 1e-8 * max(abs(ref["EL"]), 1.0), c


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("b", [0.0, 0.2499, 0.25, 4.0])
def test_pade_forms(pkg, prec, b):
    _check(pkg, dataclasses.replace(S.make_system("Ne"), b_ee=b), prec, 5)


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("n", [1, 153, 611])
def test_block_shapes(pkg, prec, n):
    _check(pkg, S.make_system("Ne"), prec, n)


def test_block_shapes_of_a_large_system(pkg):
    for n in (3, 305, 461):
        _check(pkg, S.make_system("Kr"), "df64", n, 1.0 / 126.0)
