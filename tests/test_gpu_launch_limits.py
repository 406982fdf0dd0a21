"""Launches at the limits of what a kernel gets by default: shared memory (48 KB,
of which a kernel's static part counts too)."""
import numpy as np
import pytest

from gpu_util import aos, f32_exact, soa
from paper_2107_08119_gb300 import inputs

pytestmark = pytest.mark.gpu


def _split_model(n_neu, rng):
    """Hyperparameters and parameters of the split model at another width, the
    input columns scaled to the weighted descriptors."""
    from paper_2107_08119_gb300 import nep
    hyper = nep.Hyper(**dict(inputs.PBTE_HYPER, n_neu=n_neu))
    z = inputs.random_z(hyper.n_par, rng)
    n_r = hyper.n_max_R + 1
    n_des = hyper.n_par // n_neu - 2
    zbar = np.sqrt(inputs.Z_PB * inputs.Z_TE)
    w1 = z[:n_neu * n_des].reshape(n_neu, n_des)
    w1[:, :n_r] /= zbar
    w1[:, n_r:] /= zbar ** 2
    return hyper, z


@pytest.mark.parametrize("n_neu", [49, 50, 51, 52, 64])
@pytest.mark.parametrize("n", [12160, 12161])
def test_split_model_widths(orc, n, n_neu):
    """The site pass of the split model with 16 and 32 atoms per block around the
    width at which the latter needs more than the default shared memory (50 and 51
    only together with the static part): a sample against the oracle, at the bars
    of the force path for wider networks."""
    from paper_2107_08119_gb300 import nep
    rng = np.random.default_rng(n_neu)
    pos, _, box = inputs.rocksalt(12, 12, 11)
    pos = inputs.displace(pos, 0.1, rng)[:n]
    hyper, z = _split_model(n_neu, rng)
    model = nep.NEP(z, hyper)
    out = model.compute(soa(pos), box)
    idx = np.unique(rng.integers(0, n, 60))
    U, F, _ = orc.efv_sample(orc.NepHyper(12, 6, 4, n_neu, 8.0, 4.0), f32_exact(z), pos, box, idx)
    assert np.abs(out["e_atom"].cpu().numpy()[idx] - U).max() <= 1e-6 * n_neu / 30
    assert np.abs(aos(out["force"])[idx] - F).max() <= 1e-4
    model.close()
