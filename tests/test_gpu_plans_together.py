"""Plans of different sizes alive at a time (GB300 only): the shared-memory
limit belongs to a kernel, not to a plan, so making or running a small plan
must leave a larger one of the same kernel working, with the bytes it gave
before."""
import numpy as np
import pytest

import paper_2110_03482_gb300 as fdd

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fdd.build()


def _randn(*shape, seed=1):
    return torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(seed),
                       device="cuda")


@pytest.mark.parametrize("variant", range(fdd.FDD_MAC_VARIANTS))
def test_spectra_plans(variant):
    n_dm, nb = 300, 13

    def plan(n_chan):
        return fdd.Plan(n_chan=n_chan, nu_lo_mhz=1200.0, dnu_mhz=300.0 / n_chan, t_samp_s=1e-3,
                        n_t=1 << 10, dm_list=0.1 * np.arange(n_dm), in_dtype=fdd.FDD_IN_F32,
                        output=fdd.FDD_OUT_SPECTRA, mac_variant=1 + variant)

    X = _randn(1, 1024, nb, 2)
    with plan(1024) as large:
        first, again, other = (torch.full((1, n_dm, nb, 2), 7.0, device="cuda") for _ in range(3))
        large.dedisperse_spectra_bins(X, nb, 1, 50, nb, 0, n_dm, first, nb)
        with plan(40) as small:
            large.dedisperse_spectra_bins(X, nb, 1, 50, nb, 0, n_dm, again, nb)
            small.dedisperse_spectra_bins(X, nb, 1, 50, nb, 0, n_dm, other, nb)
        torch.cuda.synchronize()
    assert torch.equal(first, again) and not torch.any(other == 7.0)


@pytest.mark.parametrize("variant", range(fdd.FDD_MAC_VARIANTS))
def test_batches(variant):
    beams = [(1000, 0.0, 0.1, 300), (500, 0.0, 0.1, 40)]

    def batch(n_chan):
        return fdd.Batch(beams, autotune=False, n_chan=n_chan, nu_lo_mhz=1200.0,
                         dnu_mhz=300.0 / n_chan, t_samp_s=1e-3, in_dtype=fdd.FDD_IN_F32,
                         output=fdd.FDD_OUT_POWER, mac_variant=1 + variant)

    x = _randn(1500 * 1024)
    with batch(1024) as large:
        first, again = (torch.full((large.info["out_elems"],), 7.0, device="cuda") for _ in range(2))
        large.execute(x, first)
        with batch(40) as small:
            other = torch.full((small.info["out_elems"],), 7.0, device="cuda")
            small.execute(x, other)
            large.execute(x, again)
        torch.cuda.synchronize()
    assert torch.equal(first, again) and not torch.any(other == 7.0)


@pytest.mark.parametrize("u8", [False, True])
def test_time_domain_plans(u8):
    def plan(ddm):
        return fdd.Plan(n_chan=48, nu_lo_mhz=1200.0, dnu_mhz=6.0, t_samp_s=1e-4, n_t=30000,
                        dm_list=ddm * np.arange(64),
                        in_dtype=fdd.FDD_IN_U8 if u8 else fdd.FDD_IN_F32)

    x = _randn(30000 * 48).abs_().mul_(20.0)
    x = x.to(torch.uint8) if u8 else x
    with plan(1.0) as wide, plan(0.01) as narrow:
        first, again = (torch.full((64, 30000 - wide.info["d_max"]), -7.0, device="cuda")
                        for _ in range(2))
        other = torch.full((64, 30000 - narrow.info["d_max"]), -7.0, device="cuda")
        wide.tdd_execute(x, first)
        narrow.tdd_execute(x, other)
        wide.tdd_execute(x, again)
        torch.cuda.synchronize()
    assert torch.equal(first, again) and torch.all(other >= 0.0)
