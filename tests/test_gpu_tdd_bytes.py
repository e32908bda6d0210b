"""Time-domain dedispersion of 8-bit samples, added as integers, against the same
samples given as floats (GB300 only).  Every sum is a whole number below 2^24,
exact in FP32 in any order, so the two are equal bit for bit.  Sizes around a
stage (8 channels), the channels whose sums fit 16 bits (256), a CTA's samples
(512) and trials (32), series shorter than a window, shift spans of several
windows, rows at every alignment.
"""
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


@pytest.mark.parametrize("layout", [fdd.FDD_LAYOUT_TIME_MAJOR, fdd.FDD_LAYOUT_CHAN_MAJOR])
@pytest.mark.parametrize("n_chan,n_t,ddm,n_dm,n_beams", [
    (1, 40, 0.0, 1, 1), (7, 513, 0.01, 5, 2), (8, 1025, 0.05, 32, 1), (9, 1531, 0.1, 33, 1),
    (255, 2047, 0.1, 31, 1), (256, 2050, 0.2, 64, 1), (257, 2049, 0.3, 65, 2),
    (264, 1601, 0.3, 32, 1), (520, 9001, 2.0, 40, 1), (40, 30011, 25.0, 70, 1),
])
def test_bytes_equal_floats(n_chan, n_t, ddm, n_dm, n_beams, layout):
    kw = dict(n_chan=n_chan, nu_lo_mhz=1200.0, dnu_mhz=300.0 / n_chan, t_samp_s=1e-3 / 4, n_t=n_t,
              n_beams=n_beams, dm_list=ddm * np.arange(n_dm), in_layout=layout,
              output=fdd.FDD_OUT_TIME)
    rng = np.random.default_rng(n_chan + n_t)
    x = rng.integers(0, 256, size=n_beams * n_t * n_chan, dtype=np.uint8)
    x[: x.size // 3] = 255  # the largest sums
    ys = []
    for dtype, v in ((fdd.FDD_IN_U8, x), (fdd.FDD_IN_F32, x.astype(np.float32))):
        with fdd.Plan(in_dtype=dtype, **kw) as plan:
            y = torch.full((n_beams, n_dm, n_t - plan.info["d_max"]), float("nan"), device="cuda")
            plan.tdd_execute(torch.from_numpy(v).cuda(), y)
            torch.cuda.synchronize()
            ys.append(y)
    assert torch.isfinite(ys[0]).all()
    assert torch.equal(ys[0], ys[1])


@pytest.mark.parametrize("dtype", [fdd.FDD_IN_U8, fdd.FDD_IN_F32])
@pytest.mark.parametrize("after", [0, 1, 2])
def test_a_call_after_a_failed_allocation_starts_over(after, dtype):
    x = torch.arange(1000 * 8, device="cuda") % 251
    x = x.to(torch.uint8 if dtype == fdd.FDD_IN_U8 else torch.float32)
    kw = dict(n_chan=8, nu_lo_mhz=1200.0, dnu_mhz=30.0, t_samp_s=1e-3, n_t=1000, in_dtype=dtype,
              dm_list=3.0 * np.arange(9), output=fdd.FDD_OUT_TIME)
    with fdd.Plan(**kw) as plan, fdd.Plan(**kw) as other:
        y, ref = [torch.empty((9, 1000 - plan.info["d_max"]), device="cuda") for _ in range(2)]
        fdd.fdd_debug_fail_alloc(after)
        try:
            with pytest.raises(fdd.FddError) as e:
                plan.tdd_execute(x, y)
            assert e.value.status == fdd.FDD_ERR_ALLOC
        finally:
            fdd.fdd_debug_fail_alloc(-1)
        plan.tdd_execute(x, y)
        other.tdd_execute(x, ref)
        torch.cuda.synchronize()
    assert torch.equal(y, ref)
