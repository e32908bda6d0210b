"""The 128-trial tile (Q_4X4), whose warps share the channels of a call (GB300
only): channel counts around the parts and the batches of eight, trials and
bins around a tile, calls on parts of the bins and trials.

Tolerance: a product carries two hardware-sine phasors (absolute error up to
2^-20.9 each, 1.7e-7 rms) and sums of at most 17 channels a part round to
2^-24 each; random over channels, below 4e-7, and 1e-6 leaves the factor
between rms and a small sample.
"""
import numpy as np
import pytest

import oracle
import paper_2110_03482_gb300 as fdd
from gpu_util import complex_to_device, device_to_complex, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-6
BAND = (1200.0, 1500.0)


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fdd.build()


@pytest.mark.parametrize("n_chan,n_dm,n_series", [
    (1, 1, 1), (2, 127, 1), (3, 128, 2), (4, 129, 1), (5, 17, 1), (8, 256, 1), (9, 100, 3),
    (31, 130, 1), (32, 128, 1), (33, 64, 1), (64, 128, 1), (65, 255, 2), (68, 16, 1),
])
def test_edges_match_oracle(n_chan, n_dm, n_series):
    L, dms = 1 << 12, 3.7 + 0.31 * np.arange(n_dm)
    dnu = (BAND[1] - BAND[0]) / n_chan
    nu = oracle.channel_centres(n_chan, BAND[0] + 0.5 * dnu, dnu)
    rng = np.random.default_rng(100 * n_chan + n_dm)
    b0, nb = 1021, 13
    X = (rng.standard_normal((n_series, n_chan, nb)) +
         1j * rng.standard_normal((n_series, n_chan, nb))).astype(np.complex64)
    with fdd.Plan(n_chan=n_chan, nu_lo_mhz=BAND[0] + 0.5 * dnu, dnu_mhz=dnu, t_samp_s=2e-3, n_t=L,
                  dm_list=dms, in_dtype=fdd.FDD_IN_F32, output=fdd.FDD_OUT_SPECTRA) as plan:
        assert plan.info["mac_variant"] == fdd.FDD_MAC_Q_4X4
        dX = complex_to_device(X, nb + 1)
        dY = torch.full((n_series, n_dm, nb + 3, 2), 7.0, device="cuda")
        plan.dedisperse_spectra_bins(dX, nb + 1, n_series, b0, nb, 0, n_dm, dY, nb + 3)
        assert torch.all(dY[:, :, nb:] == 7.0)  # the pitch's padding is untouched
        # parts of the bins, and whole tiles of the trials, give the same bits
        one = torch.empty((n_dm, 1, 2), device="cuda")
        for k in (0, 6, 12):
            plan.dedisperse_spectra_bins(complex_to_device(X[:1, :, k:k + 1], 1), 1, 1, b0 + k, 1,
                                         0, n_dm, one, 1)
            assert torch.equal(one[:, 0], dY[0, :, k])
        if n_dm > 128:
            rest = torch.empty((n_dm - 128, nb, 2), device="cuda")
            plan.dedisperse_spectra_bins(dX, nb + 1, 1, b0, nb, 128, n_dm - 128, rest, nb)
            assert torch.equal(rest, dY[0, 128:, :nb])
        torch.cuda.synchronize()
        plan.query()
    d = oracle.delays(nu, dms, 2e-3)
    Y = device_to_complex(dY, nb)
    for s in range(n_series):
        ref = oracle.fdd_bins(X[s].astype(np.complex128), np.arange(b0, b0 + nb), L, d)
        assert rel_l2(Y[s], ref) <= TOL, s


@pytest.mark.parametrize("n_chan,n_dm,tol", [
    (128, 5, TOL), (129, 130, TOL), (160, 128, TOL), (161, 40, TOL), (300, 129, TOL),
    (1024, 256, TOL), (11200, 33, 5e-6), (11201, 33, 5e-6), (15, 3, TOL), (16, 200, TOL),
    (17, 200, TOL),
])
def test_long_parts_match_oracle(n_chan, n_dm, tol):
    """A part of more than 32 channels goes round the rings of X and of phase
    constants; up to 16 channels one warp takes them all.  Sums of n terms
    round to 2^-25 sqrt(n / 2) of the result: 3.4e-7 for a quarter of 1024
    channels, 1.1e-6 for one of 11200, 2.2e-6 were they one sum, beside the
    phasors' 2.4e-7."""
    L, dms = 1 << 12, 3.7 + 0.31 * np.arange(n_dm)
    dnu = (BAND[1] - BAND[0]) / n_chan
    nu = oracle.channel_centres(n_chan, BAND[0] + 0.5 * dnu, dnu)
    rng = np.random.default_rng(n_chan)
    b0, nb = 700, 13
    X = (rng.standard_normal((2, n_chan, nb)) +
         1j * rng.standard_normal((2, n_chan, nb))).astype(np.complex64)
    with fdd.Plan(n_chan=n_chan, nu_lo_mhz=BAND[0] + 0.5 * dnu, dnu_mhz=dnu, t_samp_s=2e-3, n_t=L,
                  dm_list=dms, in_dtype=fdd.FDD_IN_F32, output=fdd.FDD_OUT_SPECTRA) as plan:
        assert plan.info["mac_variant"] == fdd.FDD_MAC_Q_4X4
        dX = complex_to_device(X, nb + 2)
        dY = torch.full((2, n_dm, nb + 1, 2), 7.0, device="cuda")
        plan.dedisperse_spectra_bins(dX, nb + 2, 2, b0, nb, 0, n_dm, dY, nb + 1)
        torch.cuda.synchronize()
        plan.query()
    assert torch.all(dY[:, :, nb:] == 7.0)
    Y = device_to_complex(dY, nb)
    d = oracle.delays(nu, dms, 2e-3)
    for s in range(2):
        ref = oracle.fdd_bins(X[s].astype(np.complex128), np.arange(b0, b0 + nb), L, d)
        assert rel_l2(Y[s], ref) <= tol, s
