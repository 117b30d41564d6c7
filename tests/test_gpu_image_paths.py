"""The display map and the binning pass on every route they choose by size
and placement.  Needs a GPU."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2310_03505_gb300 import rr
from tests.test_gpu_binning import ULPS, returns, ulp32

pytestmark = pytest.mark.gpu


def db_values(cutoff, n, seed):
    """Energies over the whole range, on and next to every rounding boundary
    of the map, and the values a pixel can otherwise hold."""
    rng = np.random.default_rng(seed)
    step = 10.0 ** (((np.arange(256) - 0.5) / 255.0 * cutoff - cutoff) / 10.0)
    near = np.concatenate([step * (1.0 + k * 2.0 ** -23) for k in (-3, -1, 0, 1, 3)])
    spread = 10.0 ** (rng.uniform(-1.2 * cutoff, 0.2 * cutoff, max(n, 8)) / 10.0)
    special = [0.0, -0.0, -1.0, np.inf, -np.inf, np.nan, 1.0, 1e-45, 1e-38, 3e38]
    with np.errstate(over="ignore"):
        x = np.concatenate([special, near, spread]).astype(np.float32)
    return np.resize(rng.permutation(x) if n < x.size else x, n)


@pytest.mark.parametrize("cutoff", [1e-3, 1.0, 60.0, 120.0, 800.0])
@pytest.mark.parametrize("n,skip", [(1, 0), (3, 0), (4, 0), (5, 1), (1023, 2), (4096, 0), (4099, 0), (70001, 3)])
def test_display_map(rrlib, cutoff, n, skip):
    """Equal to the 64-bit map except where the value lies within the
    float32 form's error of a rounding boundary (2^-11 of a step: log10f 2
    ulps and four operations on values up to 255); skip: unaligned buffers."""
    import torch
    x = db_values(cutoff, n, seed=n)
    polar = torch.zeros(n + skip, device="cuda")
    polar[skip:] = torch.from_numpy(x).cuda()
    out = torch.full((n + skip + 5,), 77, dtype=torch.uint8, device="cuda")
    rr.rr_polar_to_db_u8(polar[skip:], cutoff, out[skip:skip + n])
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert (got[:skip] == 77).all() and (got[skip + n:] == 77).all()
    e = x.astype(np.float64)
    c = float(np.float32(cutoff))
    with np.errstate(divide="ignore", invalid="ignore"):
        v = np.where(e > 0, np.clip(255.0 * (10.0 * np.log10(e) + c) / c, 0.0, 255.0), 0.0)
    lo, hi = np.floor(v + 0.5 - 2.0 ** -11), np.floor(v + 0.5 + 2.0 ** -11)
    px = got[skip:skip + n].astype(np.float64)
    assert np.all((px >= lo) & (px <= hi))


@pytest.mark.parametrize("n_columns", [1, 300, 310, 600, 620])
@pytest.mark.parametrize("where", ["device", "host", "mixed"])
def test_binning_routes(rrlib, n_columns, where):
    """Wide blocks for few columns, device buffers used in place, host ones
    staged: the exactly rounded sums within the compensated bound."""
    import torch
    rng = np.random.default_rng(n_columns)
    n_bins = 257
    col, b, e = returns(rng, 20_011, n_columns, n_bins, heavy=3000)
    ref = orc.bin_returns(col, b, e, n_columns, n_bins)
    on = {"device": (1, 1, 1, 1), "host": (0, 0, 0, 0), "mixed": (1, 0, 1, 0)}[where]
    arrs = [torch.from_numpy(x).cuda() if d else x for x, d in zip((col, b, e), on)]
    out = torch.full((n_columns, n_bins), 5.0, device="cuda") if on[3] else np.full((n_columns, n_bins), 5.0, np.float32)
    rr.rr_accumulate_returns(*arrs, n_columns, n_bins, out)
    got = out.cpu().numpy() if on[3] else out
    assert np.all(np.abs(got.astype(np.float64) - ref) <= ULPS * ulp32(ref))
    if where == "device" and n_columns * n_bins <= e.size * 4:   # an image over its own inputs
        room = torch.zeros(max(e.size, n_columns * n_bins), device="cuda")
        room[:e.size] = arrs[2]
        rr.rr_accumulate_returns(arrs[0], arrs[1], room[:e.size], n_columns, n_bins,
                                 room[:n_columns * n_bins].view(n_columns, n_bins))
        assert torch.equal(room[:n_columns * n_bins].view(n_columns, n_bins).cpu(), torch.from_numpy(got))
    # a refused call leaves a device output as it was
    bad = torch.from_numpy(col.copy()).cuda()
    bad[-1] = n_columns
    kept = torch.full((n_columns, n_bins), 5.0, device="cuda")
    with pytest.raises(rr.RRError):
        rr.rr_accumulate_returns(bad, torch.from_numpy(b).cuda(), torch.from_numpy(e).cuda(), n_columns, n_bins, kept)
    assert (kept == 5.0).all()
