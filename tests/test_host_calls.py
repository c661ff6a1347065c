"""Host code of the library's calls on a stand-in for the CUDA runtime (fake_runtime.py; no GPU)."""
import numpy as np
import pytest

import fake_runtime
from oracle import poisson
from paper_1003_4570_gb300 import omen


@pytest.fixture(scope="module")
def watch(tmp_path_factory):
    with fake_runtime.loaded(tmp_path_factory.mktemp("host")) as w:
        yield w


@pytest.fixture
def ctx(watch):
    watch.reset()
    return omen.omen_create(0)


def test_poisson_never_lowers_a_shared_memory_limit(watch, ctx):
    """The limit is the kernel's, shared by every context: a small plane or line after a large one
    must leave it, or a large solve of another thread fails between its setting and its launch."""
    for sizes in [((55, 55, 9), (43, 41, 9)), ((2048, 3, 9), (1600, 3, 9)), ((9, 2048, 9), (9, 1600, 9))]:
        for n in sizes:
            f = np.zeros((n[2] - 1, n[1], n[0]))
            omen.omen_poisson(ctx, poisson.Grid(*n, 1.0, 1.0, 1.0), f, f.copy())
    assert watch.lowered() == 0
