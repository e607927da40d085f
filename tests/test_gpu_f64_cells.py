"""FP64 phase integration (seeded quotients, cube root and table logarithm)
against the oracle over the whole range of the field and the energy."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_09348_gb300 import binding as B
from paper_2308_09348_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_09348_gb300 import build
    build.build()


# chi from 0 over 1e-9 to 1e6 and far beyond any field
@pytest.mark.parametrize("a0,gamma", [(0.0, 2000.0), (1e-4, 5.0), (1.0, 100.0), (30.0, 4e3),
                                      (300.0, 1e5), (3e3, 1e8), (1.0, 1e14)])
@pytest.mark.parametrize("variant", [0, I.VAR_CELL_FOCUS])
def test_records_match_the_oracle(a0, gamma, variant):
    n, cells = 257, 61
    L = I.Laser(a0=a0, w0_um=3.0, model=I.MODEL_QFP, n_phase=cells, variant=variant,
                delay_fs=10.0, dx_um=0.5)
    Bm = I.Beam(gamma_mean=gamma, rel_spread=0.05, sigma_x_um=2.0, sigma_y_um=2.0,
                sigma_z_um=3.0, div_rad=1e-3)
    xi = I.sample_streams(n, 77, dtype=np.float64)
    rec = B.qs_eval_samples(L, Bm, [torch.from_numpy(a).cuda() for a in xi], precision="f64")
    ref = oracle.evaluate(L, Bm, I.Bins(), xi)
    # mu: 61 cells of a few roundings each (2^-53) in 1/mu, V: the same in a
    # sum whose terms carry mu^4; both with a factor of 10 to spare
    np.testing.assert_allclose(rec["mu"].cpu().numpy(), ref["mu"], rtol=61 * 4 * 1.2e-16 * 10)
    np.testing.assert_allclose(rec["V"].cpu().numpy(), ref["V"], rtol=61 * 20 * 1.2e-16 * 10,
                               atol=1e-300)
