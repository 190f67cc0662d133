"""Far fields of several contexts, each in a thread of its own."""
import threading

import numpy as np
import pytest

from dda_inputs import random_complex

pytestmark = pytest.mark.gpu


def test_farfields_of_lattices_of_many_sizes_at_once():
    """One kernel, whose blocks have 56 to 157 KB of shared memory by the
    lattice's length, launched from eight threads: each call succeeds and
    gives its own result."""
    import paper_1202_3424_gb300 as dda
    theta, phi = np.linspace(0.0, np.pi, 3), np.zeros(3)
    k = np.array([[0.36, 0.48, 0.8]])
    wrong = []

    def work(nx, calls):
        ctx = dda.Context(0)
        ctx.set_target(np.ones((1, 1, nx), np.uint8))
        ctx.set_materials([1.5 + 0.1j])
        ctx.prepare_size_parameter(1.0, dda.Precision.FP64)
        P = random_complex((1, 3, nx), 5)
        try:
            first = ctx.farfield(0, k, P, theta, phi)
            for _ in range(calls):
                if np.abs(ctx.farfield(0, k, P, theta, phi) - first).max() > 1e-12 * np.abs(first).max():
                    wrong.append(nx)
        except dda.DdaError as err:
            wrong.append(err)
        ctx.close()

    threads = [threading.Thread(target=work, args=(nx, 3000)) for nx in (256, 60, 250, 64, 240, 70, 230, 80)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
