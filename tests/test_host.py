"""Host-side logic that needs no GPU: the autotuner's cache file and the
plane-by-plane spectral generator."""
import numpy as np
import pytest
import torch

from paper_2005_13193_gb300 import autotune, synth


def test_tune_cache_round_trip(tmp_path):
    p = str(tmp_path / "x.tune")
    autotune.write_cache(p, {"kernel": 2, "brick": (16, 8, 4)}, comment="two\nlines")
    text = open(p).read()
    assert text.splitlines()[:2] == ["# two", "# lines"]
    assert "brick 16 8 4" in text  # the line ps_batch_plan parses
    assert autotune.load_cache(p) == {"kernel": (2,), "brick": (16, 8, 4)}
    assert autotune.load_cache(str(tmp_path / "missing")) == {}


def test_spectral_field_planes_recipe():
    n, kmax = 24, 8
    f = synth.spectral_field_planes(n, kmax, seed=9, dtype=torch.float64).numpy()
    g = synth.spectral_field_planes(n, kmax, seed=9, dtype=torch.float64).numpy()
    np.testing.assert_array_equal(f, g)  # seeded
    assert np.allclose(np.sqrt((f ** 2).mean(axis=(1, 2, 3))), 1.0, atol=1e-12)
    F = np.fft.fftn(f, axes=(1, 2, 3))
    k = np.fft.fftfreq(n, 1.0 / n)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
    shell = (k2 >= 1) & (k2 <= kmax * kmax)
    # energy only on the shell 1 <= |k| <= kmax
    assert np.abs(F[:, ~shell]).max() <= 1e-9 * np.abs(F[:, shell]).max()
    # amplitude per shell falls off (k^-5/3 shell energy): compare shells 2 and 6
    e = lambda s: (np.abs(F[:, (np.sqrt(k2) >= s - 0.5) & (np.sqrt(k2) < s + 0.5)]) ** 2).sum()
    assert e(2) > e(6)


def test_tracker_rebin_modes(monkeypatch):
    # Tracker picks ps_rk2_step's rebin mode on the host: sort from the
    # positions and count (2) on the first step, then sort from the counts its
    # previous step took (3); a step with given bins (0), reset_bins() or
    # incremental=False go back to sorting from the positions
    import types

    import paper_2005_13193_gb300 as ps
    seen = []
    monkeypatch.setattr(ps, "ps_rk2_step", lambda *a, **k: seen.append(k["rebin"]))
    monkeypatch.setattr(ps, "workspace", lambda nbytes, device="cpu": torch.empty(0))
    field = types.SimpleNamespace(n=(16, 16, 16), L=(2 * np.pi,) * 3, coef=None, scale=None)
    pos = torch.zeros((3, 100), dtype=torch.float64)
    tr = ps.Tracker(field, pos, brick=(8, 8, 8), keep_velocity=False)
    for _ in range(3):
        tr.step(1e-3)
    tr.step(1e-3, rebin=False)
    tr.step(1e-3)
    tr.reset_bins()
    tr.step(1e-3)
    tr.step(1e-3)
    assert seen == [2, 3, 3, 0, 2, 2, 3]
    seen.clear()
    full = ps.Tracker(field, pos, brick=(8, 8, 8), keep_velocity=False, incremental=False)
    full.step(1e-3)
    full.step(1e-3)
    assert seen == [1, 1]


@pytest.mark.parametrize("np_,rows,bricks,pays", [
    (2_000_000, 12, 4096, True), (1_000_000, 18, 4096, False), (4_000_000, 12, 512, False),
    (4_000_000, 18, 729, False), (4_000_000, 18, 512, True), (12_000_000, 18, 512, True), (2_000_000, 18, 1331, True),
    (12_000_000, 3, 2744, False), (12_000_000, 3, 4096, True), (4_000_000, 3, 4096, False)])
def test_rows_by_way_of_bin_order_where_it_pays(np_, rows, bricks, pays):
    # few bricks write near one another as it is; few rows gain less
    import paper_2005_13193_gb300 as ps
    assert ps._unsort_pays(np_, rows, bricks) == pays


def test_differentiable_calls_binned_where_it_pays():
    # (position gradient, field gradient) by particles; beyond the L2 from some particles
    # per brick, within it by what is computed
    import paper_2005_13193_gb300 as ps
    for n, np_, want in [((64,) * 3, 700_000, (0, 0, 0, 0)), ((64,) * 3, 900_000, (1, 0, 1, 1)),
                         ((64,) * 3, 1_100_000, (1, 1, 1, 1)), ((96,) * 3, 5_000_000, (0, 1, 1, 1)),
                         ((192,) * 3, 300_000, (0, 0, 0, 0)), ((192,) * 3, 400_000, (1, 1, 1, 1)),
                         ((256,) * 3, 262_144, (1, 1, 1, 1)), ((384,) * 3, 800_000, (0, 0, 0, 0)), ((384,) * 3, 900_000, (1, 1, 1, 1))]:
        got = [ps._fn_binned(n, np_, p, f) for p, f in ((0, 0), (1, 0), (0, 1), (1, 1))]
        assert got == [bool(w) for w in want], (n, np_)
