"""Which systems lrdmc_create_system accepts (CPU, host code only): one block
of four walkers with their state, evaluation buffers and scratch side by side
within 227 KB less 2 KB, whatever layout the kernels use. The kernels' layout
overlays buffers and adds tables, and must fit every accepted system."""
import numpy as np
import pytest

import lrdmc_synth as S

LIMIT = 232448 - 2048


def _system(n_up, n_dn, n_s, n_p, n_mo, n_nuc, prims):
    rng = np.random.default_rng(n_up * 1000 + n_s * 10 + n_p)
    shells = []
    for q in range(n_s + n_p):
        l = 0 if q < n_s else 1
        if prims:
            shells.append(S.Shell(q % n_nuc, l, S.GTO, alpha=list(0.3 * 2.5 ** np.arange(prims)), coef=[0.5] * prims))
        else:
            shells.append(S.Shell(q % n_nuc, l, S.STO, 1.0 + l, 1.0 + 0.1 * q))
    n_ao = n_s + 3 * n_p
    return S.System(name="limit", nuc_xyz=rng.normal(size=(n_nuc, 3)) * 3.0, Z=np.full(n_nuc, 4.0), n_up=n_up, n_dn=n_dn,
                    shells=shells, C=rng.normal(size=(n_ao, n_mo)), en_b1=np.full(n_nuc, 0.5), orbital_shell=[0])


def _accepted_bytes(s):
    n, N, nao = s.n_up, s.N, s.n_ao
    scr = max(2 * n * n + n * nao, nao + 3 * n + n * n)
    warp = 3 * N + s.n_up ** 2 + s.n_dn ** 2 + 12 + 12 * N + N * nao + N + 3 * N + 12 + scr
    nc = nao * s.n_mo
    return 8 * (((2 * nc + (nc + 1) // 2 + 65) & ~1) + 4 * ((warp + 1) & ~1))


def test_acceptance_is_the_documented_limit():
    pkg = pytest.importorskip("paper_1909_01589_gb300")
    rng = np.random.default_rng(3)
    seen = {True: 0, False: 0}
    for _ in range(400):
        n_up = int(rng.integers(8, 33))
        n_dn = int(rng.integers(0, n_up + 1))
        n_p = int(rng.integers(0, 17))
        n_s = int(rng.integers(1, 33 - n_p))
        if n_s + 3 * n_p > 64:
            continue
        n_mo = int(rng.integers(n_up, 33))
        s = _system(n_up, n_dn, n_s, n_p, n_mo, int(rng.integers(1, 9)), int(rng.choice([0, 1, 8])))
        fits = _accepted_bytes(s) <= LIMIT
        seen[fits] += 1
        if fits:
            pkg.LrdmcSystem(s)
        else:
            with pytest.raises(pkg.LrdmcError, match="shared memory"):
                pkg.LrdmcSystem(s)
    assert seen[True] > 50 and seen[False] > 10
