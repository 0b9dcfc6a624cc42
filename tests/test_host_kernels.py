"""The thread-per-cell kernels' device arithmetic on the CPU (tests/host/host_kernels.cpp):
rare states and numerical properties that need no GPU."""
import copy
import os
import subprocess

import numpy as np
import pytest

from paper_2508_16105_gb300 import synth

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2508_16105_gb300", "csrc")


def _build(d, *flags):
    """run(command, mechanism, doubles) -> doubles"""
    exe = str(d / "host_kernels")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-ffp-contract=off", *flags, "-I", CSRC,
                    os.path.join(HERE, "host", "host_kernels.cpp"), os.path.join(CSRC, "mech_host.cpp"), "-o", exe],
                   check=True)

    def run(command, mech, x):
        path = str(d / "mech.txt")
        with open(path, "w") as f:
            f.write(mech.to_text())
        r = subprocess.run([exe, command, path], input=np.ascontiguousarray(x, dtype=np.float64).tobytes(),
                           stdout=subprocess.PIPE, check=True)
        return np.frombuffer(r.stdout)

    return run


@pytest.fixture(scope="session")
def host(tmp_path_factory):
    return _build(tmp_path_factory.mktemp("host"))


@pytest.fixture(scope="session")
def host_checked(tmp_path_factory):
    """The same, ended by undefined integer arithmetic (shift counts, signed overflow)."""
    return _build(tmp_path_factory.mktemp("checked"), "-fsanitize=shift,signed-integer-overflow",
                  "-fsanitize-undefined-trap-on-error")


@pytest.fixture(scope="module")
def no_collider():
    """H2/air whose first three-body reaction takes no part from the species of air."""
    mech = copy.deepcopy(synth.h2_air_mechanism(16105))
    rx = next(r for r in mech.reactions if r.kind == "THREEBODY")
    rx.eff = dict(rx.eff, N2=0.0, O2=0.0)
    return mech


@pytest.mark.parametrize("command", ["hvp", "hvp_fix"])
@pytest.mark.parametrize("gas", ["N2", "air", "field"])
def test_second_derivatives_without_a_third_body(host, no_collider, gas, command):
    """hvp_sum equals the sum of its directions' dual-number evaluations, also where a third
    body's concentration is exactly zero (pure N2 with a zero efficiency)."""
    mech, N = no_collider, no_collider.K + 1
    for seed in range(4):
        if gas == "field":
            c = synth.uniform_cells(mech, 1, seed=seed)
            p, y = c.p[0], np.concatenate([c.Y[:, 0], c.T])
        else:
            p, y = 1e5 * (1 + seed), np.zeros(N)
            y[mech.index("N2")] = 1.0 if gas == "N2" else 0.767
            y[mech.index("O2")] = 1.0 - y[mech.index("N2")]
            y[-1] = 700.0 + 400.0 * seed
        u = synth.normal(seed, "u", 4 * N) * np.tile(np.append(np.full(N - 1, 1e-3), 10.0), 4)
        w = synth.normal(seed, "w", 4 * N) * np.tile(np.append(np.ones(N - 1), 1e-3), 4)
        out = host(command, mech, np.concatenate([[1.0 / p], y, u, w]))
        assert np.isfinite(out).all()
        # the same terms in another order: N + 2 R sums of some 10^3 rounded terms, whose
        # cancellation leaves at least 10^-2 of the largest term: 10^3 2^-53 10^2 < 2e-11
        a, b = out.reshape(2, -1)
        for q in (slice(0, N), slice(N, N + mech.R), slice(N + mech.R, None)):
            assert np.abs(a[q] - b[q]).max() <= 2e-11 * np.abs(b[q]).max()


@pytest.mark.parametrize("command", ["rhs", "rhs_fix"])
def test_integer_arithmetic_is_defined(host_checked, command):
    """The fixed-point logarithms on ordinary states and on a Rosenbrock stage's wild ones:
    |ln k| of 256 and more, temperatures of any finite size, thermo of next to nothing."""
    mech = synth.h2_air_mechanism(16105)
    flat = copy.deepcopy(mech)
    for x in flat.species:
        x.lo = x.hi = [0.5] + [0.0] * 6
    for m in (mech, flat):
        c = synth.uniform_cells(m, 32, seed=44)
        states = [np.concatenate([[1.0 / c.p[i]], c.Y[:, i], [T]]) for i in range(32)
                  for T in (c.T[i], 1e-280, 1e-3, 40.0, 130.0, 8191.0, 8193.0, 1e9, 1e120, 1e300)]
        host_checked(command, m, np.concatenate(states))


def many_efficiencies(n):
    """n copies of a three-body reaction of the 53-species mechanism with seeded efficiencies."""
    mech = copy.deepcopy(synth.large_mechanism(16105))
    rx = next(r for r in mech.reactions if r.kind == "THREEBODY")
    mech.reactions = []
    for i in range(n):
        x = copy.deepcopy(rx)
        x.A = rx.A / n
        a = synth.uniform_range(i, "efficiencies", mech.K, 0.0, 2.0)
        x.eff = {s.name: float(a[k]) for k, s in enumerate(mech.species)}
        mech.reactions.append(x)
    return mech


def expected_plan(mech):
    """(row, column, value index, coefficient) of every term, as test_gather_plan reads them."""
    out = []
    for r, x in enumerate(mech.reactions):
        net = {}
        for sign, side in ((-1.0, x.reac), (1.0, x.prod)):
            for s, n in side:
                net[s] = net.get(s, 0.0) + sign * n
        for s, nu in net.items():
            if nu == 0.0:
                continue
            k = mech.index(s)
            out.append((-1, k, 9 * r + 7, nu))
            for first, side in ((0, x.reac), (3, x.prod)):
                out += [(k, mech.index(t), 9 * r + first + q, nu) for q, (t, _) in enumerate(side)]
            if x.kind != "ELEM":
                out.append((-2, k, 9 * r + 6, nu))
                out += [(k, mech.index(t), 9 * r + 6, nu * (a - 1.0)) for t, a in x.eff.items() if a != 1.0]
    return np.array(sorted(out))


@pytest.mark.parametrize("n", [0, 1300])
def test_gather_plan(host, n):
    """Every term of the CTA-per-cell kernels' sums, also where the mechanism has more
    distinct coefficients than a term's 16 bits count (n three-body reactions, each with its
    own efficiency of every species)."""
    mech = many_efficiencies(n) if n else synth.large_mechanism(16105)
    got = host("plan", mech, np.zeros(0)).reshape(-1, 4)
    want = expected_plan(mech)
    assert n == 0 or len(np.unique(want[:, 3])) > 65536
    assert np.array_equal(np.array(sorted(map(tuple, got))), want)


def fitted(low, high):
    """The H2/air species with fits of the given two ranges, a0 as seeded."""
    mech = copy.deepcopy(synth.h2_air_mechanism(16105))
    for x in mech.species:
        x.lo, x.hi = [x.lo[0]] + low + x.lo[5:], [x.hi[0]] + high + x.hi[5:]
    return mech


@pytest.mark.parametrize("fit", ["seeded", "wide", "narrow"])
def test_fixed_point_thermo_is_no_coarser_than_fp64(host, fit):
    """Cp/R, H/RT and d(Cp/R)/dT in fixed point against 80-bit arithmetic.  Coefficients of
    the size of published fits (wide: those for 1,000 to 3,500 K, narrow: 200 to 1,000 K) have
    too coarse a unit and stay in FP64."""
    wide, narrow = [2.2e-3, -1.6e-7, -1.0e-10, 1.7e-14], [-2.0e-3, 6.5e-6, -5.5e-9, 1.8e-12]
    mech = synth.h2_air_mechanism(16105) if fit == "seeded" else fitted(wide if fit == "wide" else narrow, wide)
    T = synth.uniform_range(54, "T", 4000, 300.0, 3500.0)
    try:
        out = host("thermo", mech, T).reshape(len(T), mech.K, 8).astype(np.longdouble)
    except subprocess.CalledProcessError as e:
        assert e.returncode == 6 and fit != "seeded"      # refused: the kernels use FP64
        return
    x = T.astype(np.longdouble)
    for k, s in enumerate(mech.species):
        # the coefficients as the packed mechanism holds them (doubles)
        rows = [np.array([[a[0], a[1], a[2], a[3], a[4]], [a[0], a[1] / 2, a[2] / 3, a[3] / 4, a[4] / 5],
                          [a[1], 2 * a[2], 3 * a[3], 4 * a[4], 0.0]]).astype(np.longdouble) for a in (s.lo, s.hi)]
        for q, name in enumerate(("Cp/R", "H/RT", "d(Cp/R)/dT")):
            c = np.where((T >= s.Tmid)[:, None], rows[1][q], rows[0][q])
            want = (((c[:, 4] * x + c[:, 3]) * x + c[:, 2]) * x + c[:, 1]) * x + c[:, 0]
            ulp = np.spacing(np.abs(want).astype(np.float64)).astype(np.longdouble)
            err = float((np.abs(out[:, k, q] - want) / ulp).max())
            if name == "d(Cp/R)/dT":
                # a unit is at most 2^-61 of the scheme's bound; three steps lose up to 6.1 units
                bound = max(abs(a[j]) * j * 2.0 ** (14 * (j - 1)) for a in (s.lo, s.hi) for j in (1, 2, 3, 4)) * 2
                assert err <= 0.5 + 6.1 * 2.0 ** -61 * bound / float(ulp.min()), (s.name, name, err)
            else:
                assert err <= 0.71, (s.name, name, err)   # 0.5 + 6.6 units of 2^-56 at Cp/R of 2 to 4


def test_fixed_point_gibbs(host):
    """G/RT as a fixed-point logarithm against 80-bit arithmetic.  Six Horner steps lose at most
    3 units of 2^-51 each, halved by every later step in T (14 units in all, in base 2); ln T
    is good to 2 ulp (2^-49), 1/T and the final product are rounded once."""
    mech = synth.h2_air_mechanism(16105)
    T = synth.uniform_range(55, "T", 4000, 150.0, 8000.0)
    out = host("thermo", mech, T).reshape(len(T), mech.K, 8)
    x = T.astype(np.longdouble)
    for k, s in enumerate(mech.species):
        g = [np.array([a[0] - a[6], -a[0], a[1] / 2 - a[1], a[2] / 3 - a[2] / 2, a[3] / 4 - a[3] / 3,
                       a[4] / 5 - a[4] / 4, a[5]]).astype(np.longdouble) for a in (s.lo, s.hi)]
        c = np.where((T >= s.Tmid)[:, None], g[1], g[0])
        want = c[:, 0] + c[:, 1] * np.log(x) + x * (c[:, 2] + x * (c[:, 3] + x * (c[:, 4] + x * c[:, 5]))) + c[:, 6] / x
        tol = (14 * 2.0 ** -51 * np.log(2.0) + np.abs(c[:, 1]) * 2.0 ** -49 + np.abs(c[:, 6] / x) * 2.0 ** -53 +
               np.abs(want) * 2.0 ** -52)
        err = np.abs(out[:, k, 3] - want)
        assert (err <= tol).all(), (s.name, float((err / tol).max()))
