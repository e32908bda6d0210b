"""The G12_4X8 tile (split-FP16 operands on the tensor cores) at the sizes
where it can go wrong (GB300 only): channel counts around a K step (16) and a
stage (64), trial counts around an al (256) and the pass capacities (1024,
2048, 4096 trials), bin counts that leave a group of bins partly idle.

Tolerance: a product carries two hardware-sine phasors (absolute error up to
2^-20.9 each, 1.7e-7 rms), table phasors of a few 2^-24 and operands of 22
bits (2^-22 each); random over channels, the sum's relative L2 error stays
below 4e-7, and 1e-6 leaves the factor between rms and a small sample.
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


def _plan(n_chan, L, dms, **kw):
    dnu = (BAND[1] - BAND[0]) / n_chan
    return fdd.Plan(n_chan=n_chan, nu_lo_mhz=BAND[0] + 0.5 * dnu, dnu_mhz=dnu, t_samp_s=2e-3,
                    n_t=L, dm_list=dms, in_dtype=fdd.FDD_IN_F32, output=fdd.FDD_OUT_SPECTRA,
                    mac_variant=1 + fdd.FDD_MAC_G12_4X8, **kw)


def _reference(X, bins, L, n_chan, dms):
    dnu = (BAND[1] - BAND[0]) / n_chan
    nu = oracle.channel_centres(n_chan, BAND[0] + 0.5 * dnu, dnu)
    return oracle.fdd_bins(X, bins, L, oracle.delays(nu, dms, 2e-3))


@pytest.mark.parametrize("n_chan,n_dm,n_series", [
    (1, 1, 1), (15, 255, 1), (16, 256, 2), (17, 257, 1), (48, 512, 1), (63, 513, 1),
    (64, 1024, 1), (65, 1025, 2), (80, 2048, 1), (81, 2049, 1), (129, 2305, 1), (130, 4096, 1),
    (193, 4097, 1), (33, 8449, 1),
])
def test_edges_match_oracle(n_chan, n_dm, n_series):
    L, dms = 1 << 12, 3.7 + 0.31 * np.arange(n_dm)
    K = L // 2 + 1
    rng = np.random.default_rng(100 * n_chan + n_dm)
    for b0, nb in [(0, 1), (1021, 7), (K - 6, 6)]:
        X = (rng.standard_normal((n_series, n_chan, nb)) +
             1j * rng.standard_normal((n_series, n_chan, nb))).astype(np.complex64)
        with _plan(n_chan, L, dms) as plan:
            dX = complex_to_device(X, nb + 1)
            dY = torch.full((n_series, n_dm, nb + 3, 2), 7.0, device="cuda")
            plan.dedisperse_spectra_bins(dX, nb + 1, n_series, b0, nb, 0, n_dm, dY, nb + 3)
            dP = torch.full((n_series, n_dm, nb), 7.0, device="cuda")
            plan.dedisperse_spectra_bins(dX, nb + 1, n_series, b0, nb, 0, n_dm, dP, nb,
                                         fdd.FDD_OUT_POWER)
            torch.cuda.synchronize()
            plan.query()
        assert torch.all(dY[:, :, nb:] == 7.0)  # the pitch's padding is untouched
        for s in range(n_series):
            ref = _reference(X[s].astype(np.complex128), np.arange(b0, b0 + nb), L, n_chan, dms)
            assert rel_l2(device_to_complex(dY, nb)[s], ref) <= TOL, (b0, s)
            assert rel_l2(dP[s].cpu().numpy(), np.abs(ref) ** 2) <= 2 * TOL, (b0, s)


@pytest.mark.parametrize("n_dm", [300, 2048, 3000])
def test_dynamic_range(n_dm):
    """Channels of very different size (the columns share one power-of-two
    scale per 64 channels), the smallest and largest normal magnitudes, zeros,
    and a NaN that stays in its own bin."""
    n_chan, L, nb, b0 = 100, 1 << 12, 8, 333
    dms = 0.5 * np.arange(n_dm)
    rng = np.random.default_rng(n_dm)
    X = rng.standard_normal((1, n_chan, nb)) + 1j * rng.standard_normal((1, n_chan, nb))
    X[0, :, 1] *= 10.0 ** rng.uniform(-6, 6, n_chan)   # spread over twelve decades
    X[0, :, 2] *= 1e-36
    X[0, :, 3] *= 1e35
    X[0, :, 4] = 0.0
    X[0, :70, 5] = 0.0
    X[0, :, 6] = 1e-30 + 0j
    X = X.astype(np.complex64)
    with _plan(n_chan, L, dms) as plan:
        dX = complex_to_device(X, nb)
        dX[0, 40, 7, 0] = float("nan")
        dY = torch.empty((1, n_dm, nb, 2), device="cuda")
        plan.dedisperse_spectra_bins(dX, nb, 1, b0, nb, 0, n_dm, dY, nb)
        torch.cuda.synchronize()
    ref = _reference(X[0].astype(np.complex128), np.arange(b0, b0 + nb), L, n_chan, dms)
    Y = device_to_complex(dY, nb)[0]
    for i in range(7):
        assert rel_l2(Y[:, i], ref[:, i]) <= TOL, i
    assert np.all(Y[:, 4] == 0) and np.all(np.isnan(Y[:, 7]))


@pytest.mark.parametrize("n_dm", [2049, 4096, 5000, 9000])
def test_calls_on_whole_blocks_agree_bit_for_bit(n_dm):
    """Trials are centred in blocks of 2048 from the call's first: a call on
    part of the list that starts at a whole block (as the streamed and batched
    calls do) gives the whole call's bytes."""
    n_chan, nb = 70, 5
    with _plan(n_chan, 1 << 12, 0.25 * np.arange(n_dm)) as plan:
        X = torch.randn((1, n_chan, nb, 2), device="cuda")
        whole = torch.empty((1, n_dm, nb, 2), device="cuda")
        plan.dedisperse_spectra_bins(X, nb, 1, 99, nb, 0, n_dm, whole, nb)
        for j in range(0, n_dm, 2048):
            n = min(2048, n_dm - j)
            part = torch.empty((1, n, nb, 2), device="cuda")
            plan.dedisperse_spectra_bins(X, nb, 1, 99, nb, j, n, part, nb)
            assert torch.equal(part, whole[:, j:j + n]), j


@pytest.mark.parametrize("n_dm", [257, 1024, 1300, 2048, 2304])
@pytest.mark.parametrize("n_series", [2, 3, 5, 7])
def test_series_sharing_passes_equal_each_alone(n_series, n_dm):
    """Two or four series share a pass (up to 1024 trials; two up to 2048):
    the same bits as each series by itself, whatever the others' scale."""
    n_chan, L, nb, b0 = 81, 1 << 12, 9, 1500
    rng = np.random.default_rng(n_series + n_dm)
    X = (rng.standard_normal((n_series, n_chan, nb)) +
         1j * rng.standard_normal((n_series, n_chan, nb)))
    X *= np.array([1.0, 1e-12, 3e9, 1.0, 0.0, 7.0, 1e20])[:n_series, None, None]
    dX = complex_to_device(X.astype(np.complex64), nb)
    with _plan(n_chan, L, 3.7 + 0.31 * np.arange(n_dm)) as plan:
        dY = torch.full((n_series, n_dm, nb, 2), 7.0, device="cuda")
        plan.dedisperse_spectra_bins(dX, nb, n_series, b0, nb, 0, n_dm, dY, nb)
        for s in range(n_series):
            one = torch.full((n_dm, nb, 2), 7.0, device="cuda")
            plan.dedisperse_spectra_bins(dX[s].contiguous(), nb, 1, b0, nb, 0, n_dm, one, nb)
            assert torch.equal(dY[s], one), s
        torch.cuda.synchronize()
        plan.query()


@pytest.mark.parametrize("output", [fdd.FDD_OUT_TIME, fdd.FDD_OUT_SPECTRA, fdd.FDD_OUT_POWER])
@pytest.mark.parametrize("n_beams,n_t,chunk_len,n_dm", [
    (1, 20000, 1 << 12, 600),    # chunks of one beam, an odd number
    (3, 20000, 1 << 13, 1100),   # beams and chunks, two of different beams together
    (2, 4096, 0, 2048),          # whole rows, no chunks
    (1, 9000, 1 << 12, 513),
])
def test_plans_that_take_two_at_a_time_give_the_same_bits(n_beams, n_t, chunk_len, n_dm, output):
    """A plan with room for two (beam, chunk)s a launch against one whose
    limit leaves room for one."""
    kw = dict(n_chan=40, nu_lo_mhz=1200.0, dnu_mhz=7.5, t_samp_s=1e-3, n_t=n_t,
              chunk_len=chunk_len, n_beams=n_beams, in_dtype=fdd.FDD_IN_F32,
              dm_list=1.0 + 0.05 * np.arange(n_dm), output=output)
    g = torch.Generator(device="cuda").manual_seed(n_t + n_dm)
    x = torch.randn(n_beams * n_t * 40, generator=g, device="cuda")
    outs, held = [], []
    limit = 0
    for _ in range(2):
        with fdd.Plan(workspace_limit=limit, **kw) as plan:
            assert plan.info["mac_variant"] == fdd.FDD_MAC_G12_4X8
            out = torch.full((plan.info["out_elems"] * (2 if output == fdd.FDD_OUT_SPECTRA else 1),),
                             7.0, device="cuda")
            plan.execute(x, out)
            torch.cuda.synchronize()
            plan.query()
            outs.append(out)
            held.append(plan.info["workspace_bytes"])
            limit = fdd.fdd_plan_geometry(fdd.Params(**kw))["workspace_bytes"] - 1
    assert held[1] < held[0]
    assert torch.equal(outs[0], outs[1])


def test_batch_beams_have_the_bits_of_their_own_plans():
    """Beams of one batch are launched by the form of their trial counts (up to
    512, 1024, 2048, more): each equals a plan of its own."""
    counts = [300, 4096, 512, 513, 2049, 1024, 1025, 700, 2048, 1]
    kw = dict(n_chan=40, nu_lo_mhz=1200.0, dnu_mhz=7.5, t_samp_s=1e-3, in_dtype=fdd.FDD_IN_F32,
              output=fdd.FDD_OUT_SPECTRA, chunk_len=0, mac_variant=1 + fdd.FDD_MAC_G12_4X8)
    n_t = [2048 if i % 2 else 1024 for i in range(len(counts))]
    g = torch.Generator(device="cuda").manual_seed(5)
    xs = [torch.randn(n * 40, generator=g, device="cuda") for n in n_t]
    with fdd.Batch([(t, 1.0, 0.02, d) for t, d in zip(n_t, counts)], autotune=False, **kw) as batch:
        out = torch.full((batch.info["out_elems"], 2), 7.0, device="cuda")
        batch.execute(torch.cat(xs), out)
        torch.cuda.synchronize()
        for i, d in enumerate(counts):
            with fdd.Plan(n_t=n_t[i], dm_list=1.0 + 0.02 * np.arange(d), **kw) as plan:
                one = torch.full((plan.info["out_elems"], 2), 9.0, device="cuda")
                plan.execute(xs[i], one)
                torch.cuda.synchronize()
            at = batch.out_offsets[i]
            assert torch.equal(out[at:at + one.shape[0]], one), i


@pytest.mark.parametrize("n_chan", [1, 16, 63, 64])
@pytest.mark.parametrize("n_dm,n_series", [(3000, 1), (700, 4), (700, 6), (2000, 2), (2000, 3)])
def test_one_stage_items_match_oracle(n_chan, n_dm, n_series):
    """Up to 64 channels and one bin at a time, an item is one stage; with
    fewer items than CTAs the second of the two warps that make the stages'
    tables has none, and the loads that it starts ahead must be real ones."""
    L, dms = 1 << 12, 3.7 + 0.31 * np.arange(n_dm)
    b0, nb = 1021, 3
    rng = np.random.default_rng(n_chan + n_dm + n_series)
    X = (rng.standard_normal((n_series, n_chan, nb)) +
         1j * rng.standard_normal((n_series, n_chan, nb))).astype(np.complex64)
    with _plan(n_chan, L, dms) as plan:
        dX = complex_to_device(X, nb)
        dY = torch.full((n_series, n_dm, nb, 2), 7.0, device="cuda")
        plan.dedisperse_spectra_bins(dX, nb, n_series, b0, nb, 0, n_dm, dY, nb)
        torch.cuda.synchronize()
        plan.query()
    for s in range(n_series):
        ref = _reference(X[s].astype(np.complex128), np.arange(b0, b0 + nb), L, n_chan, dms)
        assert rel_l2(device_to_complex(dY, nb)[s], ref) <= TOL, s


@pytest.mark.parametrize("n_dm", [300, 700, 2048, 3000])
def test_infinite_samples_stay_in_their_bin(n_dm):
    """An infinity takes every trial of its own bin and series (not a finite
    value anywhere: the split makes NaN of it) and none of another's."""
    n_chan, nb, n_series, b0 = 70, 9, 2, 333
    X = torch.randn((n_series, n_chan, nb, 2), device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(n_dm))
    with _plan(n_chan, 1 << 12, 0.5 * np.arange(n_dm)) as plan:
        clean, dY = (torch.empty((n_series, n_dm, nb, 2), device="cuda") for _ in range(2))
        plan.dedisperse_spectra_bins(X, nb, n_series, b0, nb, 0, n_dm, clean, nb)
        X[0, 3, 1, 0], X[1, 69, 6, 1] = float("inf"), -float("inf")
        plan.dedisperse_spectra_bins(X, nb, n_series, b0, nb, 0, n_dm, dY, nb)
        dP = torch.empty((n_series, n_dm, nb), device="cuda")
        plan.dedisperse_spectra_bins(X, nb, n_series, b0, nb, 0, n_dm, dP, nb, fdd.FDD_OUT_POWER)
        torch.cuda.synchronize()
        plan.query()
    hit = torch.zeros((n_series, nb), dtype=torch.bool, device="cuda")
    hit[0, 1] = hit[1, 6] = True
    hit = hit[:, None].expand(n_series, n_dm, nb)
    assert not torch.any(torch.isfinite(dY[hit])) and not torch.any(torch.isfinite(dP[hit]))
    assert torch.equal(dY[~hit], clean[~hit])


@pytest.mark.parametrize("nb", [5, 260])
@pytest.mark.parametrize("n_dm", [700, 2048, 2049, 5000, 9000])
@pytest.mark.parametrize("n_chan", [32, 33, 64, 65, 128, 129])
def test_forms_by_channel_count_give_the_same_bits(n_chan, n_dm, nb):
    """On both sides of the channel counts at which series begin to share
    passes and passes of 4096 trials begin, in one launch of few bins and in
    several of more: a series among five has the bits it has alone, and blocks
    of 2048 trials those of the whole call."""
    n_series, L = 5, 1 << 12
    dms = 0.25 * np.arange(n_dm)
    rng = np.random.default_rng(n_chan + n_dm)
    X = (rng.standard_normal((n_series, n_chan, nb)) +
         1j * rng.standard_normal((n_series, n_chan, nb))).astype(np.complex64)
    dX = complex_to_device(X, nb)
    with _plan(n_chan, L, dms) as plan:
        whole = torch.full((n_series, n_dm, nb, 2), 7.0, device="cuda")
        plan.dedisperse_spectra_bins(dX, nb, n_series, 999, nb, 0, n_dm, whole, nb)
        for j in range(0, n_dm, 2048):
            n = min(2048, n_dm - j)
            for s in (0, 4):
                part = torch.full((n, nb, 2), 7.0, device="cuda")
                plan.dedisperse_spectra_bins(dX[s].contiguous(), nb, 1, 999, nb, j, n, part, nb)
                assert torch.equal(part, whole[s, j:j + n]), (j, s)
        torch.cuda.synchronize()
        plan.query()
    ref = _reference(X[2, :, :5].astype(np.complex128), np.arange(999, 1004), L, n_chan, dms)
    assert rel_l2(device_to_complex(whole[2, :, :5], 5), ref) <= TOL
