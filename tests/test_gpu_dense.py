"""Spectra and thresholds with crossings everywhere: counts stay exact, and the time stays in proportion.

The times are ratios taken within one process, each side the median of several event-timed groups of calls.
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
    import torch

    for _ in range(3):
        fn()
    times = []
    for _ in range(groups):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fn()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) / reps * 1e3)
    return sorted(times)[groups // 2]


def test_convolution_of_a_spectrum_with_a_loud_end(fd):
    """HP_1 of 2^21 bins that were not whitened, 480000 crossings in the first twentieth of the columns: at most 2.2
    times as long as without crossings (one counter update per row segment: 1.5; one for every 32 columns: 3 to 4.6)."""
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
