"""What a tuning leaves behind in a batch context: a failed one its schedule
as it was, a successful one the full range of resident blocks for the next.
Trials are counted and failed on the host (SDEB_FAULT=trial:<k>), each case in
a child process."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = textwrap.dedent("""
    import sys
    import torch
    sys.path.insert(0, {root!r})
    import paper_1908_03869_gb300 as sdeb
    from paper_1908_03869_gb300 import inputs
    from paper_1908_03869_gb300.integrator import BatchIntegrator

    # a few long chains, which few blocks an SM end soonest, and many short tasks
    sizes = [(200, 6000, 30)] + [(40, 300, 4000)] * 8
    pbs = [sdeb.Problem.make("kuramoto", n, orbits, 0.005, steps, steps, 0, "fp32") for n, steps, orbits in sizes]
    data = [inputs.kuramoto(n, orbits, seed=i) for i, (n, _, orbits) in enumerate(sizes)]
    p, x0 = ([torch.tensor(d[i], dtype=torch.float32, device="cuda") for d in data] for i in (0, 1))

    def final(it):
        it.set_params(p, x0)
        it.integrate()
        return torch.cat([it.final(i).flatten() for i in range(len(sizes))])

    with BatchIntegrator(pbs) as it, BatchIntegrator(pbs) as untouched:
        before, failed = it.info(), None
        for k in range(int(sys.argv[1])):
            it.set_params(p, x0)
            try:
                it.autotune()
            except sdeb.SdebError as e:
                failed = k
                print("STATUS", e.status)
                print("SCHEDULE KEPT", it.info() == before)
                print("SAME", torch.equal(final(it), final(untouched)))
                break
            before = it.info()
        print("FAILED", failed)
        if failed is None:  # schedules on the tuner's grid and on the rule's, which differ for some
            for frac in (0.02, 0.125, 0.5, 4.0):
                it.set_params(p, x0)
                untouched.set_params(p, x0)
                it.set_schedule(frac)
                untouched.set_schedule(frac)
                print("GRIDS", it.info()["grid"], untouched.info()["grid"])
                print("BITS", torch.equal(final(it), final(untouched)))
""")


def _child(tunings, fault):
    env = dict(os.environ, SDEB_FAULT=fault)
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT), str(tunings)], env=env, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1908_03869_gb300 import build as sdeb_build
    sdeb_build.build()


@pytest.mark.parametrize("trial", [0, 5])
def test_a_failed_tuning_leaves_the_schedule_as_it_was(trial):
    import paper_1908_03869_gb300 as sdeb
    out = _child(1, "trial:%d" % trial)
    assert "STATUS %d" % sdeb.SDEB_ECUDA in out and "FAILED 0" in out
    assert "SCHEDULE KEPT True" in out and "SAME True" in out


def test_a_second_tuning_tries_as_much_as_the_first():
    trials = next(t for t in range(8, 48, 8) if "FAILED 1" in _child(2, "trial:%d" % t))
    assert "FAILED 2" in _child(3, "trial:%d" % (2 * trials))


def test_the_grid_does_not_change_the_bits():
    out = _child(1, "")
    assert out.count("BITS True") == 4
