"""GPU: contexts of several threads at once, each on its own stream: the first launches of every kernel
family set launch limits that all threads read."""
import concurrent.futures as cf

import numpy as np
import pytest

import gabp_synth
from gpu_common import ensure_built, solver

pytestmark = pytest.mark.gpu


def _run(job):
    (nx, ny), precision, kernel = job
    p = gabp_synth.make_problem(nx, ny, 0.2, nx, n_uniform=nx * ny // 10)
    with solver(p, precision, kernel=kernel) as s:
        s.iterate(45, 0.4)
        return s.get_messages(), s.residual()


def test_contexts_of_several_threads():
    ensure_built()
    jobs = [(shape, precision, kernel) for shape in ((64, 40), (91, 67), (300, 170))
            for precision, kernel in (("fp32", 0), ("fp32", 1), ("fp32", 4), ("fp64", 0))]
    with cf.ThreadPoolExecutor(8) as ex:
        together = list(ex.map(_run, jobs * 2))
    for job, a, b in zip(jobs, together[:len(jobs)], together[len(jobs):]):
        alone = _run(job)
        for got in (a, b):
            assert np.array_equal(got[0], alone[0]) and got[1] == alone[1], job
