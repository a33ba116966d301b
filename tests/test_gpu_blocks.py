"""The kernels that rank by blocks of kets, at the sizes where their routes change.

A space's route depends on its modes, its couplings and its size: sectors resident in shared
memory, one cooperative launch, direct stage launches (four records in flight or one), or
factored couplings in an annihilation and a creation pass.  Each case below lies on one
route or next to the line between two; the comparison is with the CPU oracle, and where two
routes share their arithmetic, with the other one bit for bit.

Tolerances, set before the first run:
  * H psi in FP64 of up to some 200 terms a row: 1e-13 relative (the summation order differs);
  * 3 RK4 steps whose stages hold 48-bit pairs: each of 12 stage vectors is off by at most
    some 2^-44 of a step's increment, itself below the state's norm: 1e-11 is above their sum;
  * first and second moments, FP64 sums over double-float products: 1e-11 of the particle number.
"""
import threading

import numpy as np
import pytest

import oracle as orc
import workloads as wl
from helpers import random_state, rel_err, to_dev, to_host

pytestmark = pytest.mark.gpu


def _hermitian(M, seed, scale):
    rng = np.random.default_rng(seed)
    L = (rng.standard_normal((M,) * 4) + 1j * rng.standard_normal((M,) * 4)) * scale * wl._conserving(M)
    return 0.5 * (L + np.conj(L.transpose(2, 3, 0, 1)))


def _coupling(kind, M, exact):
    if kind == "contact":
        return wl.contact_coupling(M, -0.02, exact=exact)
    if kind == "long":
        return wl.long_range_coupling(M, 0.02, exact=exact)
    return _hermitian(M, M, 0.01)


# M, n_min, n_max, momenta, coupling, exact, kets
CASES = {
    "one_ket": (5, 0, 0, None, "contact", False, 1),
    "resident_m5": (5, 0, 10, None, "contact", False, 3003),
    "grid_m5_one_sector": (5, 22, 22, [0], "contact", False, None),
    "grid_m5_last": (5, 0, 20, None, "long", False, 53130),
    "direct_m5_first": (5, 0, 21, None, "contact", False, 65780),
    "grid_m7": (7, 3, 10, None, "long", False, 19448 - 36),
    "grid_m7_last": (7, 0, 11, None, "contact", False, 31824),
    "direct_m7": (7, 0, 12, None, "long", False, 50388),
    "factored_m7": (7, 0, 12, None, "contact", False, 50388),
    "factored_m7_n_min": (7, 4, 12, None, "contact", False, 50388 - 120),
    "factored_m7_lower_not_held": (7, 14, 14, None, "contact", False, 38760),
    "factored_m7_two_momenta": (7, 18, 18, [0, 3], "contact", False, None),
    "factored_m7_exact": (7, 0, 12, None, "contact", True, 50388),
    "direct_m7_exact": (7, 0, 9, None, "long", True, 11440),
    "factored_m9": (9, 0, 8, None, "contact", False, 24310),
    "direct_m9_small": (9, 0, 7, None, "contact", False, 11440),
    "factored_m11": (11, 7, 7, None, "contact", False, 19448),
    "direct_m11": (11, 6, 6, None, "long", False, 8008),
    "direct_m4": (4, 0, 20, None, "hermitian", False, 10626),
    "direct_m6": (6, 0, 9, None, "hermitian", False, 5005),
    "direct_m7_complex": (7, 0, 8, None, "hermitian", False, 6435),
    "direct_m8": (8, 0, 7, None, "hermitian", False, 6435),
    "direct_m5_exact": (5, 0, 14, None, "long", True, 11628),
    "factored_m8_exact": (8, 0, 10, None, "contact", True, 43758),
    "factored_m6": (6, 0, 14, None, "contact", False, 38760),
    "factored_m8": (8, 0, 10, None, "contact", False, 43758),
}


@pytest.mark.parametrize("name", CASES)
def test_routes_against_the_oracle(name):
    """Basis (the set-up by blocks), H psi, three steps, and the moments of the result."""
    import paper_2111_00050_gb300 as qb

    M, lo, hi, momenta, kind, exact, kets = CASES[name]
    w, L = wl.dispersion_quadratic(M) * 0.3, _coupling(kind, M, exact)
    qs = qb.Space(M, w, L, lo, hi, momenta, exact=exact)
    assert kets is None or qs.total == kets
    os_ = orc.Space(M, qs.sectors, exact=exact)
    np.testing.assert_array_equal(qs.basis().cpu().numpy(), os_.basis)
    x = random_state(qs.total, 3)
    y = qs.empty_state()
    qs.hpsi(to_dev(x), y)
    ref = orc.apply_h(os_, w, L, x)
    assert rel_err(to_host(y), ref) <= 1e-13 or np.linalg.norm(ref) == 0.0
    dt = 0.2 / max(1.0, np.linalg.norm(ref))
    psi = to_dev(x)
    qs.evolve(psi, dt, 3)
    end = orc.rk4(os_, w, L, x, dt, 3)
    assert rel_err(to_host(psi), end) <= 1e-11
    end /= np.linalg.norm(end)
    got, want = qs.observables(to_dev(end)), orc.moments(os_, end)
    scale = max(1.0, float(hi))
    for k in ("a", "Mij", "aa"):
        assert np.abs(np.asarray(got[k]) - np.asarray(want[k])).max() <= 1e-11 * scale, k


@pytest.mark.parametrize("name", [n for n in CASES if n.startswith(("grid", "resident", "one_ket"))])
@pytest.mark.parametrize("steps", [1, 33])
def test_one_launch_routes_equal_stage_launches(name, steps):
    """Resident sectors and the cooperative launch against one launch a stage, bit for bit."""
    import paper_2111_00050_gb300 as qb

    M, lo, hi, momenta, kind, exact, _ = CASES[name]
    qs = qb.Space(M, wl.dispersion_quadratic(M) * 0.3, _coupling(kind, M, exact), lo, hi, momenta, exact=exact)
    a = to_dev(random_state(qs.total, 5))
    b = a.clone()
    qs.evolve(a, 1e-3, steps)
    qs.set_resident_max(0)
    qs.evolve(b, 1e-3, steps)
    assert bool((a == b).all())


def test_cooperative_launches_on_several_streams():
    """Three spaces advanced at once by a thread and a stream each: the states of one after
    the other."""
    import torch

    import paper_2111_00050_gb300 as qb

    spaces = [qb.Space(M, wl.dispersion_quadratic(M) * 0.3, _coupling("contact", M, False), 0, hi)
              for M, hi in ((5, 18), (7, 9), (5, 20))]
    want = []
    for k, qs in enumerate(spaces):
        want.append(to_dev(random_state(qs.total, k)))
        qs.evolve(want[-1], 1e-3, 50)
    got = [to_dev(random_state(qs.total, k)) for k, qs in enumerate(spaces)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in spaces]

    def run(k):
        with torch.cuda.stream(streams[k]):
            for _ in range(5):
                spaces[k].evolve(got[k], 1e-3, 10)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(len(spaces))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert all(bool((g == e).all()) for g, e in zip(got, want))


@pytest.mark.parametrize("M,hi,kind,exact", [(1, 9, "contact", False), (2, 9, "contact", False), (3, 9, "long", False),
                                             (5, 9, "long", False), (5, 9, "contact", True), (7, 7, "long", False),
                                             (8, 5, "hermitian", False), (9, 5, "long", False),
                                             (11, 4, "contact", False), (7, 12, "contact", False)])
def test_coupling_gradient_by_blocks(M, hi, kind, exact):
    """The derivative along the space's own coupling equals grad_scale (two different sums of
    the same products, FP64 over double-float: 1e-10), for every record width, pairs without a
    partner, and a factored space, which keeps the moments kernel."""
    import paper_2111_00050_gb300 as qb

    rng = np.random.default_rng(M)
    L = _coupling(kind, M, exact) * 10
    z = (rng.standard_normal(M) + 1j * rng.standard_normal(M)) * 0.8
    qs = qb.Space(M, wl.dispersion_quadratic(M) * 0.3, L, 0, hi, exact=exact)
    got = qs.adjoint(z, -0.3, 2e-3, 6, ckpt_every=0, loss="Q", coupling_grad=True)
    along = float(np.sum((np.conj(got["grad_L"]) * L).real))
    assert abs(along - got["grad_scale"]) <= 1e-10 * abs(got["grad_scale"]) + 1e-16
