"""Launch rules and kernel variants of the step, at the sizes where they change:
every variant evaluates the per-node arithmetic of the two-pass form, so the
populations agree bit for bit."""
import numpy as np
import pytest
import torch

from paper_2101_04550_gb300 import elbm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    elbm.load()


def populations(lattice, n, storage, kernel, steps, **kw):
    """Populations after the given launches of steps, from a seeded field."""
    if lattice == elbm.D3Q27:
        rho, u = inputs.isotropic_turbulence(n, seed=5, k0=3.0, u_rms=0.05)
    else:
        rho, u = inputs.double_shear_layer(n, U=0.08)
    with elbm.Solver(lattice, n, storage=storage, kernel=kernel, T=0.42, nu=0.02,
                     stream=torch.cuda.current_stream(), **kw) as s:
        s.init(rho, u)
        for k in steps:
            s.step(k)
        return s.get_populations(dtype=np.float32)


# one plane per segment (32 x 16 x 3 is one tile column), a last segment
# shorter than the others (3 planes of 150), whole segments, the deepest ones
@pytest.mark.parametrize("n", [(32, 16, 3), (32, 16, 150), (64, 32, 33), (128, 80, 5), (512, 304, 70)])
@pytest.mark.parametrize("storage", [elbm.F32_SHIFT, elbm.F16_SHIFT])
def test_segment_depths_bitwise(n, storage):
    kw = dict(stretch=(1.0, 1.5, 2.0))
    want = populations(elbm.D3Q27, n, storage, 1, (1, 2), **kw)
    assert np.array_equal(populations(elbm.D3Q27, n, storage, 3, (1, 2), **kw), want)


@pytest.mark.parametrize("n", [(32, 8, 3), (64, 24, 41)])
def test_segment_depths_of_eight_row_tiles_bitwise(n):
    want = populations(elbm.D3Q27, n, elbm.F32, 1, (3,))
    assert np.array_equal(populations(elbm.D3Q27, n, elbm.F32, 3, (3,)), want)
