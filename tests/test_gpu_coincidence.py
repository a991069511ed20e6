"""Electrons on a nucleus or on an electron of the other spin: the local energy
is not finite there (the oracle's is NaN), the projection reports it, and every
other configuration of the call is untouched. The lattice moves out of such a
point are ordinary ones, to the evaluation tests' 1e-10 of each ratio's own
floating-point scale (2e-4 of max(|ratio|, 1) in the mixed mode)."""
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


def _positions(system, where):
    x = S.initial_positions(system, 4, 7)
    if where == "nucleus":
        x[1, 0] = system.nuc_xyz[0]
    else:
        x[1, system.n_up] = x[1, 0]
    return x


def _system(pkg, system, prec):
    return pkg.LrdmcSystem(system).set_precision({"fp64": pkg.PRECISION_FP64, "df64": pkg.PRECISION_DF64,
                                                  "fp32": pkg.PRECISION_FP32}[prec])


@pytest.mark.parametrize("where", ["nucleus", "pair"])
@pytest.mark.parametrize("name", ["He", "Ne", "H2O"])
@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32"])
def test_local_energy_is_not_finite(pkg, prec, name, where):
    import oracle

    system = S.make_system(name)
    x, R = _positions(system, where), S.random_rotations(4, 5)
    o = oracle.OracleSystem(system)
    lat = oracle.lattice_for(system, 0.1, oracle.THIS_WORK)
    sp = pkg.Spacing(pkg.THIS_WORK)
    ratio, _, _, el = (q.cpu().numpy() for q in _system(pkg, system, prec).evaluate(
        torch.tensor(x, device="cuda"), torch.tensor(R, device="cuda"), 0.1, sp))
    for c in range(4):
        ref = o.lattice_eval(lat, x[c], R[c])
        assert np.isfinite(ref["EL"]) == (c != 1)
        if c == 1:
            assert not np.isfinite(el[c])
        else:
            assert abs(el[c] - ref["EL"]) <= 1e-8 * max(abs(ref["EL"]), 1.0)
        if prec == "fp32":
            assert np.all(np.abs(ratio[c] - ref["ratio"]) <= 2e-4 * np.maximum(np.abs(ref["ratio"]), 1.0)), c
        else:
            scale = U.ratio_scale(o, system, lat, x[c], R[c], ref["ratio"])
            assert np.all(np.abs(ratio[c] - ref["ratio"]) <= 1e-10 * scale), c
    g = _system(pkg, system, prec)
    g.init_walkers(x, seed=3, tau=0.01, e_trial=-2.9, trace_capacity=8)
    with pytest.raises(pkg.LrdmcError) as e:
        g.step(1, 0.1, sp)
        g.energy_trace()
    assert e.value.status == pkg.ERR_NONFINITE


@pytest.mark.parametrize("where", ["nucleus", "pair"])
def test_training_terms_are_not_finite(pkg, where):
    """The neural term's own gradient has no direction there: E_L is not a
    number even with base terms that the caller gives as finite."""
    from oracle import neural as onn
    from paper_1909_01589_gb300 import neural

    system = S.make_system("Ne")
    spec = S.default_neural_spec(system)
    params = S.neural_init(spec, 4, out_scale=0.5)
    x = _positions(system, where)
    grad, e = np.zeros((4, system.N, 3)), np.full(4, -128.0)
    el, j = neural.NeuralJastrowTerms.apply(torch.tensor(params, device="cuda"), pkg.LrdmcSystem(system), spec,
                                            torch.tensor(x, device="cuda"), torch.tensor(grad, device="cuda"),
                                            torch.tensor(e, device="cuda"), False)
    ref, refj = onn.energy_terms(params, spec, x, system.n_up, system.nuc_xyz, grad, e, bf16=False)
    assert torch.equal(torch.isfinite(el).cpu(), torch.isfinite(ref))
    assert list(torch.isfinite(ref)) == [True, False, True, True]
    assert torch.isfinite(j).all() and torch.isfinite(refj).all()
