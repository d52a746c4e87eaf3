"""Device paths at the sizes where they can go wrong: tails of buffers, edges
of tiles and of the division of the work, odd and smallest grids."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
SEED = 2110144940


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_14494_gb300 import build
    build.build()


def _dirty(value):
    """Leaves value in the allocator's free blocks, which the next workspace takes."""
    x = [torch.full((1 << 20,), value, dtype=torch.float32, device="cuda") for _ in range(16)]
    torch.cuda.synchronize()
    del x


@pytest.mark.parametrize("shape", [(21, 19, 23), (16, 12, 20), (7, 5, 9)])
def test_coupled_start_does_not_depend_on_memory(shape):
    """The low halves of the float-pair potential start at zero over their whole
    length, also where the cell count leaves them off the end of ncell doubles."""
    from paper_2110_14494_gb300 import PicContext
    grid = W.grid_spec(*shape, 5e-5)
    n = shape[0] * shape[1] * shape[2]
    phis = []
    for value in (0.0, 1.0e3):
        _dirty(value)
        ctx = PicContext(W.synthetic_air(), grid, precision=32, capacity=1024, seed=SEED, dt=1e-12, coupled=True,
                         v_lo=0.0, v_hi=2000.0, v_mask=0.0, poisson_rtol=1e-6, poisson_max_cycles=1000)
        ctx.step(1)
        blob = ctx.save()
        phis.append(np.frombuffer(blob, np.float64, count=n, offset=len(blob) - 8 * n))
    assert np.array_equal(phis[0], phis[1])
