"""Contexts on several host threads at once, as the server's slots are: a
launch in one thread must not depend on what another thread sets."""
import threading

import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_00804_gb300 import build
    build.build()


def _together(jobs):
    """Runs the callables on a thread each and raises the first error."""
    errors = []

    def run(f):
        try:
            f()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=run, args=(f,)) for f in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def test_clusters_of_several_sizes_on_several_threads():
    """Single clusters of 44 and 64 waters (mixed path), each in steps of its
    own thread.  The dipole history keeps every step a launch of its own."""
    import torch
    import paper_2201_00804_gb300 as pkg

    def job(n):
        def steps():
            s = synth.make_cluster(n, seed=n)
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                pos = torch.tensor(s.pos.reshape(-1), dtype=torch.float64, device="cuda")
                m = torch.tensor(s.masses().reshape(-1), dtype=torch.float64, device="cuda")
                ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, periodic=False, pcg_tol_D=1e-4,
                                       precision=pkg.PREC_MIXED, warm_start=2)
                try:
                    for _ in range(20):
                        pkg.sibfa_md_steps(ctx, pos.clone(), torch.zeros_like(pos), m, 0.01, 100)
                finally:
                    pkg.sibfa_destroy(ctx)
        return steps

    _together([job(n) for n in (44, 64)])


def test_short_range_caps_on_several_threads():
    """FP64 contexts whose schedule tuning is under way: each tries caps of 3,
    0 and 2 blocks per SM, which reserve different amounts of shared memory."""
    import numpy as np
    import paper_2201_00804_gb300 as pkg

    def job(k):
        def calls():
            s = synth.make_cluster(2, seed=70 + k)
            pos = np.ascontiguousarray(s.pos.reshape(-1))
            for _ in range(120):
                ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, periodic=False, pcg_tol_D=1e-4,
                                       precision=pkg.PREC_FP64, warm_start=False)
                try:
                    for _ in range(12):
                        pkg.sibfa_energy_forces(ctx, pos)
                finally:
                    pkg.sibfa_destroy(ctx)
        return calls

    _together([job(k) for k in range(6)])


FIRST_SOLVES = """
import threading
import numpy as np
import synth
import paper_2201_00804_gb300 as pkg

s = synth.make_cluster(30, seed=80)
pos = np.ascontiguousarray(s.pos.reshape(-1))
ctx = [pkg.sibfa_create(synth.PARAMS, s.mp_local, periodic=False, pcg_tol_D=1e-8, precision=pkg.PREC_FP64,
                        warm_start=False) for _ in range(8)]
start, pol = threading.Barrier(8), []

def first(c):
    start.wait()
    pol.append(pkg.sibfa_energy_forces(c, pos)["pol"])

threads = [threading.Thread(target=first, args=(c,)) for c in ctx]
for t in threads:
    t.start()
for t in threads:
    t.join()
assert len(pol) == 8 and max(pol) - min(pol) <= 1e-9 * abs(pol[0]), pol
"""


def test_first_solves_of_a_process_on_several_threads():
    """The first solves by separate kernels of a process, at the same time:
    each sees the launch shape that the first of them lays down."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FIRST_SOLVES], cwd=root, env=dict(os.environ, SIBFA_PCG_HOST_LOOP="1"),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
