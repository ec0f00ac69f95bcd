"""Spectra and thresholds with crossings everywhere: counts stay exact, and the time stays in proportion.

The times are ratios taken within one process, each side the median of several replays of a graph of calls.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _spectrum(n, red):
    """Noise of unit power; red: louder towards low bins, 20 times its power and more in the first hundredth."""
    import torch

    x = torch.from_numpy(synth.complex_noise(np.random.default_rng(n), n).astype(np.complex64)).cuda()
    if red:
        f = torch.arange(1, n + 1, device="cuda", dtype=torch.float32) / n
        x = (x * torch.sqrt(1 + 0.05 / f)).to(torch.complex64).contiguous()
    return x


def _us(fn, reps=10, groups=5):
    """Microseconds per call on the device: a replayed graph of `reps` calls, so that the host's share does not count."""
    import torch

    fn()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(reps):
            fn()
    graph.replay()
    times = []
    for _ in range(groups):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) / reps * 1e3)
    return sorted(times)[groups // 2]


def test_convolution_of_a_spectrum_with_a_loud_end(fd):
    """HP_1 of 2^21 bins that were not whitened, 480000 crossings in the first twentieth of the columns: at most 2.2
    times as long as without crossings (one counter update per row segment: 1.4; one for every 32 columns: 3 to 4.6)."""
    import torch

    n, p = 1 << 21, fd.Params()
    s = fd.Searcher(p, n)

    def convolve(spec):
        return lambda: fd.fdas_search_convolve(p, spec, n, s.tmpl, s.plane, s.ld, s.thresh, s.ws, s.ws_bytes)

    quiet = _us(convolve(_spectrum(n, False)))
    red = _spectrum(n, True)
    loud = _us(convolve(red))
    s.search(red)
    over = int((s.plane[:, :n] > torch.from_numpy(s.thresh_host[0]).cuda()[:, None]).sum())
    assert s.results()[1][0] == over > 400000
    assert loud < 2.2 * quiet, (loud, quiet)


def test_harmonic_sum_where_most_strips_cross(fd):
    """2^21 bins at 2 sigma, 4 million crossings of HP_1 alone: at most 10 times as long as at 6 sigma (one counter update
    per strip for all planes at once: 5.9; one for every 32 columns and plane in turn: 27)."""
    import torch

    n, p = 1 << 21, fd.Params()
    ta = {sigma: torch.from_numpy(fd.fdas_default_thresholds(p, sigma)).cuda() for sigma in (2.0, 6.0)}
    s = fd.Searcher(p, n)
    fd.fdas_convolve(p, _spectrum(n, False), n, s.tmpl, s.plane, s.ld)

    def harmonic_sum(sigma):
        return lambda: fd.fdas_harmonic_sum(p, s.plane, n, s.ld, ta[sigma], s.cands, s.counts, s.peaks, s.ws, s.ws_bytes)

    quiet, dense = _us(harmonic_sum(6.0)), _us(harmonic_sum(2.0))
    assert s.results()[1][0] == int((s.plane[:, :n] > ta[2.0][0][:, None]).sum()) > 3_000_000
    assert dense < 10 * quiet, (dense, quiet)


def test_harmonic_sum_of_one_plane(fd):
    """A threshold on a plane of 262144 bins as it stands is no dearer than two harmonic planes of it: at most 0.88 of
    their time (0.74; 0.94 while the first strip of every warp went through its columns one after the other)."""
    n = 262144
    plane = synth.exponential_plane(np.random.default_rng(3), 85, n)
    times = []
    for n_harm in (1, 2):
        import torch

        p = fd.Params(n_harm=n_harm, harm_mask=(1 << n_harm) - 1)
        s = fd.Searcher(p, n)
        s.plane[:, :n] = torch.from_numpy(plane).cuda()
        times.append(_us(lambda: fd.fdas_harmonic_sum(p, s.plane, n, s.ld, s.thresh, s.cands, s.counts, s.peaks, s.ws,
                                                      s.ws_bytes), reps=40))
    assert times[0] < 0.88 * times[1], times


@pytest.mark.parametrize("n,n_harm,bound", [(524288, 8, 8), (524288, 5, 8), (100003, 12, 4.5)])
def test_highest_harmonic_sum_where_most_tiles_cross(fd, n, n_harm, bound):
    """The sum by the highest harmonic at 2 sigma against 6 sigma (one counter update per warp and row for all planes at
    once: 3.6, 3.9 and 2.4 times as long; one for every 32 columns and plane in turn: 16, 15 and 6.6)."""
    import torch

    p = fd.Params(n_harm=n_harm, harm_mask=(1 << n_harm) - 1, harm_index=1)
    ta = {sigma: torch.from_numpy(fd.fdas_default_thresholds(p, sigma)).cuda() for sigma in (2.0, 6.0)}
    s = fd.Searcher(p, n)
    fd.fdas_convolve(p, _spectrum(n, False), n, s.tmpl, s.plane, s.ld)

    def harmonic_sum(sigma):
        return lambda: fd.fdas_harmonic_sum(p, s.plane, n, s.ld, ta[sigma], s.cands, s.counts, s.peaks, s.ws, s.ws_bytes)

    quiet, dense = _us(harmonic_sum(6.0)), _us(harmonic_sum(2.0))
    assert dense < bound * quiet, (dense, quiet)


@pytest.mark.parametrize("n_harm", [1, 2, 3, 5, 8, 9, 12, 16])
@pytest.mark.parametrize("sigma", [-1.0, 1.0, 2.5])
@pytest.mark.parametrize("index", ["fundamental", "highest"])
def test_crossings_beyond_the_workspace(fd, n_harm, sigma, index):
    """Counts and peaks are exact however many sums cross, and every record kept is a crossing of its own; where all
    crossings fit, the records are the oracle's (strips of 1 to 16 terms, tiles, whole and ragged)."""
    import torch

    from oracle import harmonic, thresholds

    n, n_temp = (30011, 43) if index == "fundamental" else (2531, 43)
    plane = synth.exponential_plane(np.random.default_rng(n_harm), n_temp, n)
    p = fd.Params(n_temp=n_temp, z_min=-21, n_harm=n_harm, harm_mask=(1 << n_harm) - 1, cand_cap=4096,
                  harm_index=int(index == "highest"))
    ta = thresholds.threshold_array(n_harm, n_temp, sigma=max(sigma, 1.0))
    if sigma < 0:
        ta = np.full_like(ta, -1.0)  # every sum crosses
    ref = harmonic.detect(plane, ta, n_harm, p.harm_mask, 1 << 30, index=index)
    s = fd.Searcher(p, n, thresh=ta)
    s.plane[:, :n] = torch.from_numpy(plane).cuda()
    fd.fdas_harmonic_sum(p, s.plane, n, s.ld, s.thresh, s.cands, s.counts, s.peaks, s.ws, s.ws_bytes)
    cands, counts, peaks = s.results()
    assert list(counts) == list(ref.counts)
    for k in range(n_harm):
        assert (peaks[k]["power"], peaks[k]["i"], peaks[k]["j"]) == ref.peaks[k]
        got, want = cands[k], ref.cands[k]
        if len(want) <= 16384:
            assert np.array_equal(got["power"], want["power"][:4096]) and np.array_equal(got["j"], want["j"][:4096])
            continue
        assert len(got) == 4096
        place = lambda r: r["i"].astype(np.int64) * (1 << 32) + r["j"]  # noqa: E731
        order = np.argsort(place(want))
        at = np.searchsorted(place(want), place(got), sorter=order)
        assert len(set(place(got).tolist())) == 4096
        assert np.array_equal(place(want)[order[at]], place(got))
        assert np.array_equal(want["power"][order[at]], got["power"])
