"""The footprint that admits a problem (ps_estimate_bytes) covers what its handle holds (ps_device_bytes): rows
scattered over the whole plane, where every occupied tile of the grid makes a work item of its own, rows on few tiles, many
blocks, no rows."""
import numpy as np
import pytest

from paper_1801_02417_gb300 import binding as B
from paper_1801_02417_gb300.solver import PolarizedSARA

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1801_02417_gb300 import _build
    _build.build_library()
    B.lib()


@pytest.mark.parametrize("n,levels,M,blocks,reach", [(1024, 3, 20001, 1, 0.9999), (2048, 2, 60001, 3, 0.9999),
                                                     (64, 2, 5000, 2047, 0.9999), (32, 2, 2047, 2047, 0.9999),
                                                     (16, 1, 1, 1, 0.9999), (256, 4, 50000, 8, 0.1), (64, 2, 0, 0, 1.0)])
def test_estimate_covers_the_handle(n, levels, M, blocks, reach):
    rng = np.random.default_rng(M)
    uv = rng.uniform(-reach * np.pi, reach * np.pi, size=(M, 2))
    vis = np.ones((M, 4), np.complex64)
    off = np.round(np.linspace(0, M, max(blocks, 1) + 1)).astype(np.int64) if M else np.zeros(1, np.int64)
    with PolarizedSARA(n, levels, gamma=1.0) as s:
        s.set_measurements(uv, vis, None, off, np.ones(blocks))
        held = B.ps_device_bytes(s.h)
    estimate = B.ps_estimate_bytes(n, levels, M)
    assert held <= estimate, (held, estimate)
    assert M == 0 or reach < 0.5 or estimate <= 1.05 * held + 2 ** 20     # and is no more than a full grid takes
