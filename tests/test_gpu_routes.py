"""Calls that meet on one space or one device, and the routes' limits and refusals.

Where two runs take the same arithmetic they are compared bit for bit; against the oracle the
tolerances are those of test_gpu_blocks.py.
"""
import ctypes
import math
import threading

import numpy as np
import pytest

import oracle as orc
import workloads as wl
from helpers import random_state, rel_err, to_dev, to_host
from test_gpu_blocks import CASES, _coupling

pytestmark = pytest.mark.gpu


def _space(M, hi, lo=0, kind="contact", **kw):
    import paper_2111_00050_gb300 as qb

    L = wl.long_range_coupling(M, 0.02) if kind == "long" else wl.contact_coupling(M, -0.02)
    return qb.Space(M, wl.dispersion_quadratic(M) * 0.3, L, lo, hi, **kw)


def _rk4(qs, x, dt, steps):
    """The Horner steps by FP64 H psi (qb_hpsi, compared with the oracle by itself)."""
    out = qs.empty_state()
    for _ in range(steps):
        v = x
        for d in (4, 3, 2, 1):
            qs.hpsi(v, out)
            v = x - (1j * dt / d) * out
        x = v
    return x


@pytest.mark.parametrize("threads", [2, 4])
def test_threads_evolve_states_of_one_space(threads):
    """A thread, a stream, a state and a workspace each on one space of the cooperative launch
    (33,649 kets): the states of one call after the other, bit for bit."""
    import torch

    qs = _space(5, 18)
    assert qs.total == 33649
    want = [to_dev(random_state(qs.total, k)) for k in range(threads)]
    got = [x.clone() for x in want]
    for x in want:
        for steps in (1, 20, 70, 3):
            qs.evolve(x, 1e-3, steps)
    work = [qs.workspace() for _ in range(threads)]
    streams = [torch.cuda.Stream() for _ in range(threads)]
    torch.cuda.synchronize()
    errors = []

    def run(k):
        try:
            with torch.cuda.stream(streams[k]):
                for steps in (1, 20, 70, 3):
                    qs.evolve(got[k], 1e-3, steps, work[k])
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    pool = [threading.Thread(target=run, args=(k,)) for k in range(threads)]
    for t in pool:
        t.start()
    for t in pool:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    assert all(bool((g == e).all()) for g, e in zip(got, want))


def test_a_call_under_capture_leaves_nothing_behind():
    """A call on a stream that its caller captures ends in an error (its status is read by the
    host); the next call, on any stream, is as if it had not been."""
    import torch

    import paper_2111_00050_gb300 as qb

    rt = ctypes.CDLL("libcudart.so.13")
    qs = _space(5, 18)
    x = to_dev(random_state(qs.total, 1))
    want = x.clone()
    qs.set_resident_max(0)  # stage by stage
    qs.evolve(want, 1e-3, 5)
    qs.set_resident_max(1024)
    work = qs.workspace()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, 1) == 0  # thread-local mode
    with torch.cuda.stream(stream), pytest.raises(qb.QbError):
        qs.evolve(x, 1e-3, 5, work)
    rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
    if graph.value:
        rt.cudaGraphDestroy(graph)
    rt.cudaGetLastError()
    qs.evolve(x, 1e-3, 5, work)
    assert bool((x == want).all())


@pytest.mark.parametrize("M,hi", [(5, 18), (7, 10)])
def test_a_wait_that_runs_out_is_reported(M, hi):
    """With no polls every thread block gives up at the first barrier and leaves: QB_ETIMEOUT, for
    this call alone; the calls after it, with the limit back, are as if it had not been."""
    import paper_2111_00050_gb300 as qb

    qs = _space(M, hi)
    x = to_dev(random_state(qs.total, 2))
    want = x.clone()
    qs.evolve(want, 1e-3, 5)
    y = x.clone()
    qs.set_wait_polls(0)
    for steps in (1, 40):
        with pytest.raises(qb.QbError) as e:
            qs.evolve(y, 1e-3, steps)
        assert e.value.code == qb._lib.QB_ETIMEOUT
    assert qs.status() == 0
    qs.observables(x)
    qs.set_wait_polls(1 << 27)
    y.copy_(x)
    qs.evolve(y, 1e-3, 5)
    assert bool((y == want).all())


@pytest.mark.parametrize("kind", ["long", "contact"])
def test_a_workspace_that_is_too_small_is_refused(kind):
    """Two spaces over the same kets can differ in what they take (a contact coupling adds the
    annihilated vectors): a workspace of the smaller one is refused, not written past its end."""
    import torch

    qs = _space(7, 12, kind=kind)
    base = torch.empty(3 * qs.total, dtype=torch.complex128, device="cuda")
    x = to_dev(random_state(qs.total, 1))
    want = x.clone()
    qs.evolve(want, 1e-3, 2)
    calls = {
        "evolve": lambda y, work: qs.evolve(y, 1e-3, 2, work),
        "evolve_plain": lambda y, work: qs.evolve_plain(y, 1e-3, 2, work),
        "evolve_observe": lambda y, work: qs.evolve_observe(y, 1e-3, 2, 1, work),
        "evolve_batch": lambda y, work: qs.evolve_batch(y, [1.0], 1e-3, 2, work),
    }
    work = qs.workspace()
    assert (work.numel() > base.numel()) == (kind == "contact")
    for name, call in calls.items():
        for w in (base, work[1:]):
            y = x.clone()
            if w is base and kind == "long":
                call(y, w)
                assert bool((y == want).all()), name
            else:
                with pytest.raises(ValueError):
                    call(y, w)
                assert bool((y == x).all()), name
    qs.evolve(x, 1e-3, 0, work[1:])  # no steps take no workspace
    with pytest.raises(ValueError):
        qs.autotune(1e-3, x, steps=1, work=work[1:])
    with pytest.raises(ValueError):
        qs.evolve_batch(torch.stack([x, x]), [1.0, 2.0], 1e-3, 2, work)


@pytest.mark.parametrize("M,hi", [(5, 3), (5, 4), (7, 3), (9, 3)])
def test_moments_of_few_kets_lose_nothing_between_the_lanes(M, hi):
    """Up to 56 kets of fewer than n_max particles are one or two rounds of a warp: every lane has
    one product, and a moment's error is that of the products and of the sum over the lanes.  With
    a positive state nothing cancels.  32 double-float products of double-float factors, drawn at
    random and added without loss, are off by 7e-16 (rms, relative to their sum); added in
    double-float pair by pair, by 1.9e-15.  The bound lies between."""
    import paper_2111_00050_gb300 as qb

    qs = _space(M, hi, kind="long")
    occ = qs.basis().cpu().numpy()
    at = {tuple(o): k for k, o in enumerate(occ.tolist())}
    rng = np.random.default_rng(M + hi)
    err = []
    for _ in range(8):
        x = rng.random(qs.total) + 0.1
        x /= np.linalg.norm(x)
        got = qs.observables(to_dev(x))
        norm = math.fsum(v * v for v in x)

        def below(o, *modes):
            """sqrt(n_i ...) and the ket below o by a particle of each mode, or None."""
            o, c = list(o), 1
            for m in modes:
                c *= o[m]
                o[m] -= 1
            return (c, at[tuple(o)]) if c > 0 else None

        lower = [[below(o, i) for i in range(M)] for o in occ.tolist()]
        raised = {}  # ket -> the kets above it by a particle of mode i
        for k, row in enumerate(lower):
            for i, t in enumerate(row):
                if t:
                    raised.setdefault(t[1], {})[i] = (t[0], k)
        for i in range(M):
            a = math.fsum(math.sqrt(t[0]) * x[t[1]] * x[k] for k, row in enumerate(lower) for t in [row[i]] if t)
            err.append(got["a"][i].real * norm / a - 1.0)
            for j in range(i, M):
                aa = math.fsum(math.sqrt(t[0]) * x[t[1]] * x[k] for k, o in enumerate(occ.tolist())
                               for t in [below(o, i, j)] if t)
                err.append(got["aa"][i, j].real * norm / aa - 1.0)
                if j > i:
                    ad = math.fsum(math.sqrt(up[i][0] * up[j][0]) * x[up[i][1]] * x[up[j][1]] for up in raised.values())
                    err.append(got["Mij"][i, j].real * norm / ad - 1.0)
    assert np.sqrt(np.mean(np.square(err))) <= 1.2e-15
    assert np.abs(err).max() <= 1e-14


@pytest.mark.parametrize("M,hi,kets", [(7, 16, 245157), (7, 12, 50388), (9, 8, 24310)])
def test_energy_of_factored_couplings_takes_the_weights_in_fp64(M, hi, kets):
    """<H> of a contact coupling, sum_k lam_k |B_k psi|^2 over the lower kets, of positive states,
    where nothing cancels and the few values of the ket weights err alike in many kets: products
    of some ten factors in FP64 are off by 2 or 3 in its last place (6e-16), weights of 48 bits by
    twice that.  Against FP64 H psi, summed in more bits."""
    qs = _space(M, hi)
    assert qs.total == kets
    err = []
    for k in range(4):
        rng = np.random.default_rng(k)
        x = rng.random(qs.total) + 0.1
        x /= np.linalg.norm(x)
        psi, out = to_dev(x), qs.empty_state()
        qs.hpsi(psi, out)
        h = to_host(out).real
        x, h = x.astype(np.longdouble), h.astype(np.longdouble)
        err.append(float((qs.observables(psi)["H"] * (x * x).sum() - (x * h).sum()) / np.abs(x * h).sum()))
    assert np.sqrt(np.mean(np.square(err))) <= 7e-16


@pytest.mark.parametrize("M,hi,kets", [(16, 6, 74613), (14, 7, 116280)])
def test_many_modes_against_the_oracle(M, hi, kets):
    """Hundreds of terms a ket, and blocks of more modes than the maps' line asks for: H psi and
    two steps."""
    qs = _space(M, hi, kind="long")
    assert qs.total == kets
    os_ = orc.Space(M, qs.sectors)
    w, L = wl.dispersion_quadratic(M) * 0.3, wl.long_range_coupling(M, 0.02)
    x = random_state(qs.total, M)
    y = qs.empty_state()
    qs.hpsi(to_dev(x), y)
    ref = orc.apply_h(os_, w, L, x)
    assert rel_err(to_host(y), ref) <= 1e-13
    psi = to_dev(x)
    dt = 0.2 / max(1.0, np.linalg.norm(ref))
    qs.evolve(psi, dt, 2)
    assert rel_err(to_host(psi), to_host(_rk4(qs, to_dev(x), dt, 2))) <= 1e-11


def test_tables_of_many_modes_stay_small():
    """14 modes, 4.5M kets: with blocks of three kets, each with a row of 840 bases, the space took
    5 GB.  60 bytes a ket, rows of at most 256 and half a gigabyte of maps and sums are 1.9."""
    import torch

    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    qs = _space(14, 11, kind="long")
    assert qs.total == 4457400
    assert free - torch.cuda.mem_get_info()[0] <= (60 + 256) * qs.total + (1 << 29)


@pytest.mark.parametrize("name", CASES)
def test_norm_particles_and_energy_of_every_route(name):
    """Norm, <N> and <H> (direct rows, or factored couplings' lower kets) against the oracle: FP64
    sums of products of 48 bits, 1e-12 of what they sum."""
    import paper_2111_00050_gb300 as qb

    M, lo, hi, momenta, kind, exact, _ = CASES[name]
    w, L = wl.dispersion_quadratic(M) * 0.3, _coupling(kind, M, exact)
    qs = qb.Space(M, w, L, lo, hi, momenta, exact=exact)
    os_ = orc.Space(M, qs.sectors, exact=exact)
    x = random_state(qs.total, 11) * 1.5
    got, hx = qs.observables(to_dev(x)), orc.apply_h(os_, w, L, x)
    norm, N = np.sum(np.abs(x) ** 2), os_.basis.sum(1)
    assert abs(got["norm"] - norm) <= 1e-12 * norm
    assert abs(got["N"] - np.sum(np.abs(x) ** 2 * N) / norm) <= 1e-12 * max(1, hi)
    assert abs(got["H"] - np.vdot(x, hx).real / norm) <= 1e-12 * np.sum(np.abs(x * hx)) / norm


# M, n_max, coupling, kets: more rounds of 32 kets than 16 warps an SM take at once, so that every
# shape but the first two is a launch of its own, in the direct kernel of two and three partners
# (unrolled) and of four, the generic one, and both passes of factored couplings
SHAPES = [(5, 24, "contact", 118755), (7, 14, "long", 116280), (9, 10, "long", 92378), (4, 40, "contact", 135751),
          (7, 14, "contact", 116280), (8, 12, "contact", 125970)]


@pytest.mark.parametrize("M,hi,kind,kets", SHAPES)
def test_tile_shapes_of_stage_launches_are_bit_identical(M, hi, kind, kets):
    """70 steps (a graph of 32 replayed once, and single launches) under every shape, and one launch
    a sector."""
    import paper_2111_00050_gb300 as qb

    qs = _space(M, hi, kind=kind)
    assert qs.total == kets
    x = to_dev(random_state(qs.total, 4))
    want = x.clone()
    qs.evolve(want, 1e-4, 70)
    for shape in range(1, qb._lib.QB_TILE_SHAPES):
        qs.set_tile_shape(shape)
        y = x.clone()
        qs.evolve(y, 1e-4, 70)
        assert bool((y == want).all()), shape
    qs.set_tile_shape(0)
    qs.evolve_plain(x, 1e-4, 70)
    assert bool((x == want).all())


@pytest.mark.parametrize("B", [2, 4, 8])
@pytest.mark.parametrize("M,lo,hi", [(7, 0, 12), (11, 7, 7)])
def test_sweeps_of_factored_couplings(M, lo, hi, B):
    """The members of a sweep take their passes in turn through one vector: each against the oracle
    under its own coupling (the bound of three steps in test_gpu_blocks.py), and 70 steps against
    a space of that coupling alone (a coupling scaled in the kernel or in the tables: 1e-11)."""
    import torch

    import paper_2111_00050_gb300 as qb

    w, L = wl.dispersion_quadratic(M) * 0.3, wl.contact_coupling(M, -0.02)
    qs = qb.Space(M, w, L, lo, hi)
    os_ = orc.Space(M, qs.sectors)
    scale = [0.25 * (b + 1) * (-1) ** b for b in range(B)]
    x = [random_state(qs.total, 20 + b) for b in range(B)]
    dt = 0.2 / max(1.0, np.linalg.norm(orc.apply_h(os_, w, 2 * L, x[0])))
    psi = torch.stack([to_dev(v) for v in x])
    qs.evolve_batch(psi, scale, dt, 3)
    for b in (0, B - 1):
        assert rel_err(to_host(psi[b]), orc.rk4(os_, w, scale[b] * L, x[b], dt, 3)) <= 1e-11, b
    psi = torch.stack([to_dev(v) for v in x])
    qs.evolve_batch(psi, scale, dt, 70)
    for b in range(B):
        alone = to_dev(x[b])
        qb.Space(M, w, scale[b] * L, lo, hi).evolve(alone, dt, 70)
        assert rel_err(to_host(psi[b]), to_host(alone)) <= 1e-11, b


@pytest.mark.parametrize("M,lo,hi,exact", [(7, 0, 12, False), (7, 14, 14, False), (9, 0, 8, False), (11, 7, 7, False),
                                           (7, 0, 12, True)])
def test_factored_steps_by_graph(M, lo, hi, exact):
    """70 steps of factored couplings (a replayed graph) and the same by one launch a sector, bit for
    bit, and by FP64 H psi: 280 stages, each off by some 2^-44 of its increment, 1e-11."""
    import paper_2111_00050_gb300 as qb

    w, L = wl.dispersion_quadratic(M) * 0.3, wl.contact_coupling(M, -0.02, exact=exact)
    qs = qb.Space(M, w, L, lo, hi, exact=exact)
    x, out = to_dev(random_state(qs.total, 6)), qs.empty_state()
    qs.hpsi(x, out)
    dt = 0.2 / max(1.0, float(out.norm()))
    a, b = x.clone(), x.clone()
    qs.evolve(a, dt, 70)
    qs.evolve_plain(b, dt, 70)
    assert bool((a == b).all())
    assert rel_err(to_host(a), to_host(_rk4(qs, x, dt, 70))) <= 1e-11


# M, n_max, coupling, exact: few particles in many modes, where each lane walks its own ket's
# records, resident (the first row) and stage by stage, and next to the lines between the two
FEW = [(16, 3, "long", False), (12, 3, "hermitian", False), (11, 3, "contact", False), (9, 3, "long", False),
       (8, 4, "contact", True), (6, 4, "long", False),
       (14, 5, "long", False), (12, 5, "hermitian", False), (11, 5, "long", False), (10, 5, "long", True), (9, 5, "long", False)]


@pytest.mark.parametrize("M,hi,kind,exact", FEW)
def test_few_particles_in_many_modes(M, hi, kind, exact):
    """H psi and three steps against the oracle (the bounds of test_gpu_blocks.py); 33 and 70 steps in
    one launch, stage by stage and sector by sector, bit for bit."""
    import paper_2111_00050_gb300 as qb

    w, L = wl.dispersion_quadratic(M) * 0.3, _coupling(kind, M, exact)
    qs = qb.Space(M, w, L, 0, hi, exact=exact)
    os_ = orc.Space(M, qs.sectors, exact=exact)
    x = random_state(qs.total, M)
    y = qs.empty_state()
    qs.hpsi(to_dev(x), y)
    ref = orc.apply_h(os_, w, L, x)
    assert rel_err(to_host(y), ref) <= 1e-13
    dt = 0.2 / max(1.0, np.linalg.norm(ref))
    psi = to_dev(x)
    qs.evolve(psi, dt, 3)
    assert rel_err(to_host(psi), orc.rk4(os_, w, L, x, dt, 3)) <= 1e-11
    for steps in (33, 70):
        runs = [to_dev(x) for _ in range(3)]
        qs.evolve(runs[0], dt, steps)
        qs.set_resident_max(0)
        qs.evolve(runs[1], dt, steps)
        qs.evolve_plain(runs[2], dt, steps)
        qs.set_resident_max(1024)
        assert bool((runs[0] == runs[1]).all()) and bool((runs[0] == runs[2]).all())


@pytest.mark.parametrize("B", [2, 4, 8])
@pytest.mark.parametrize("M,hi,kind", [(4, 9, "long"), (5, 10, "contact"), (6, 9, "long"), (7, 6, "long"), (7, 10, "long"),
                                       (8, 7, "contact"), (9, 6, "long"), (10, 6, "long"), (11, 5, "long"), (12, 4, "long"),
                                       (13, 4, "contact")])
def test_members_of_a_sweep_equal_single_runs(M, hi, kind, B):
    """The number of members decides whether all lanes take every record or each its own ket's: the
    states of the members one by one, bit for bit."""
    import torch

    qs = _space(M, hi, kind=kind)
    x = [to_dev(random_state(qs.total, b)) for b in range(B)]
    scale = [0.3 * (b + 1) * (-1) ** b for b in range(B)]
    psi = torch.stack(x)
    qs.evolve_batch(psi, scale, 1e-3, 5)
    for b in range(B):
        qs.evolve_batch(x[b], [scale[b]], 1e-3, 5)
        assert bool((psi[b] == x[b]).all()), b
