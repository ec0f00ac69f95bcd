"""Launch shapes and code paths that the library chooses by size: the results must not depend on the choice.

Every comparison is bit for bit: a work item runs the same arithmetic whichever templates share it, and
the harmonic sums are float32 additions in a fixed order.
"""
import numpy as np
import pytest

import synth
from oracle import harmonic, thresholds

from parity_helpers import assert_same_candidates

pytestmark = pytest.mark.gpu


def _spectrum(n, seed):
    import torch

    return torch.from_numpy(synth.complex_noise(np.random.default_rng(seed), n).astype(np.complex64)).cuda()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("n,n_temp", [(1, 85), (1629, 85), (4099, 9), (65536, 85), (200003, 43), (500001, 127)])
def test_chosen_templates_per_item_equal_one_item_per_segment(n, n_temp, prec):
    import torch

    import paper_1806_01556_gb300 as fd

    p = fd.Params(n_temp=n_temp, z_min=-(n_temp // 2), precision=prec)
    s = fd.Searcher(p, n)
    spec = _spectrum(n, n)
    s.plane.fill_(-1.0)
    fd.fdas_convolve(p, spec, n, s.tmpl, s.plane, s.ld)
    got = s.plane.clone()
    s.plane.fill_(-1.0)
    fd.fdas_convolve_cfg(p, spec, n, s.tmpl, s.plane, s.ld, 0, n_temp)
    torch.cuda.synchronize()
    assert torch.equal(got, s.plane)
    assert (got[:, :n] >= 0).all()


@pytest.mark.parametrize("kind", ["noise", "tones", "zeros", "copies"])
@pytest.mark.parametrize("n,n_temp,n_harm", [(1, 3, 1), (1629, 255, 2), (4099, 85, 8), (30011, 9, 1), (131072, 85, 8),
                                             (262147, 43, 16)])
def test_search_takes_hp1_like_the_harmonic_sum(n, n_temp, n_harm, kind, prec=0):
    """HP_1 comes from the convolution in a search (rows in a scattered order, shares that start inside a segment)
    and from the harmonic sum of the finished plane: the same records bit for bit, equal peaks (zeros; the same
    samples in every segment) included. At most two CTAs per SM write the same plane."""
    import torch

    import paper_1806_01556_gb300 as fd

    p = fd.Params(n_temp=n_temp, z_min=-(n_temp // 2), n_harm=n_harm, harm_mask=(1 << n_harm) - 1, cand_cap=300,
                  precision=prec)
    spec = _spectrum(n, n)
    if kind == "tones":
        spec[::997] += 40.0
    elif kind == "zeros":
        spec.zero_()
    elif kind == "copies":
        spec = spec[torch.arange(n, device="cuda") % 1628].contiguous()
    s = fd.Searcher(p, n, thresh=thresholds.threshold_array(n_harm, n_temp, sigma=4.0))
    fd.fdas_search(p, spec, n, s.tmpl, s.plane, s.ld, s.thresh, s.cands, s.counts, s.peaks, s.ws, s.ws_bytes)
    plane, got = s.plane[:, :n].clone(), s.results()
    for ctas in (1, 2):
        s.plane.fill_(-1.0)
        fd.fdas_convolve_cfg(p, spec, n, s.tmpl, s.plane, s.ld, ctas, 0)
        assert torch.equal(plane, s.plane[:, :n])
    fd.fdas_harmonic_sum(p, s.plane, n, s.ld, s.thresh, s.cands, s.counts, s.peaks, s.ws, s.ws_bytes)
    ref = s.results()
    assert np.array_equal(got[1], ref[1]) and np.array_equal(got[2], ref[2])
    for k in range(n_harm):
        if ref[1][k] <= 16384:  # all that the workspace keeps
            assert np.array_equal(got[0][k], ref[0][k])


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind", ["noise", "tones", "zeros", "copies"])
@pytest.mark.parametrize("n,n_temp,n_harm", [(1, 3, 1), (1629, 255, 2), (30011, 9, 1), (131072, 85, 8)])
def test_tensor_core_search_takes_hp1_like_the_harmonic_sum(n, n_temp, n_harm, kind, prec):
    """The same for the tensor-core forms (two rows of a pair per warp, an odd last row)."""
    test_search_takes_hp1_like_the_harmonic_sum(n, n_temp, n_harm, kind, prec)


def _plane(kind, n_temp, n):
    rng = np.random.default_rng(n + n_temp)
    plane = synth.exponential_plane(rng, n_temp, n)
    if kind == "zeros":
        plane[:] = 0.0
    elif kind == "ties":  # every value from a short list: equal sums everywhere
        plane = rng.integers(0, 3, size=(n_temp, n)).astype(np.float32)
    elif kind == "inf":
        plane[rng.random((n_temp, n)) < 0.002] = np.inf
    elif kind == "negative":
        plane -= np.float32(1.5)
    return plane


@pytest.mark.parametrize("kind", ["noise", "zeros", "ties", "inf", "negative"])
@pytest.mark.parametrize("n,n_temp,n_harm", [(1, 3, 1), (2, 5, 2), (1023, 3, 8), (1025, 255, 16), (4097, 85, 8),
                                             (8191, 43, 9), (30011, 85, 5), (100003, 17, 8)])
def test_harmonic_sum_equals_algorithm_1(fd, n, n_temp, n_harm, kind):
    """Units and strips of the harmonic sum at their edges (one column, one more or less than a unit, rows with
    1 to 16 planes, a row stride without 16-byte alignment), and the values that its limits have to get right:
    ties, zeros, infinities and negative sums. Bit for bit against Algorithm 1 on the same plane."""
    import torch

    plane = _plane(kind, n_temp, n)
    p = fd.Params(n_temp=n_temp, z_min=-(n_temp // 2), n_harm=n_harm, harm_mask=(1 << n_harm) - 1, cand_cap=300)
    ld = n + 3
    s = fd.Searcher(p, n, thresh=thresholds.threshold_array(n_harm, n_temp, sigma=4.0))
    d_plane = torch.full((n_temp, ld), 1e30, device="cuda")
    d_plane[:, :n] = torch.from_numpy(plane).cuda()
    with np.errstate(invalid="ignore"):
        ref = harmonic.detect(plane, s.thresh_host, n_harm, p.harm_mask, 300)
    s.ws.fill_(0xAB)
    fd.fdas_harmonic_sum(p, d_plane, n, ld, s.thresh, s.cands, s.counts, s.peaks, s.ws, s.ws_bytes)
    cands, counts, peaks = s.results()
    assert max(ref.counts) <= 16384
    # Powers are not negative: a plane whose sums all are has no peak, and its record decodes an empty key.
    none = (np.float32(0.0), 255 - n_temp // 2, 0xFFFFFF)
    ref.peaks[:] = [none if r[0] < 0 else r for r in ref.peaks]
    assert_same_candidates(cands, counts, peaks, ref, p.harm_mask)


@pytest.mark.parametrize("kind", ["noise", "zeros", "ties", "inf", "negative"])
@pytest.mark.parametrize("n,n_temp,n_harm", [(1, 3, 1), (239, 5, 16), (241, 43, 9), (839, 85, 8), (841, 9, 2),
                                             (2521, 85, 5), (1683, 101, 12), (6001, 17, 16), (70001, 17, 8)])
@pytest.mark.parametrize("pad", [0, 3])
def test_highest_harmonic_sum_equals_its_definition(fd, n, n_temp, n_harm, kind, pad):
    """Tiles of the sum by the highest harmonic at their edges (840 columns for up to 8 planes, 240 for more, the
    last rows of a CTA), with a row stride that allows 16-byte copies and one that does not."""
    import torch

    plane = _plane(kind, n_temp, n)
    p = fd.Params(n_temp=n_temp, z_min=-(n_temp // 2), n_harm=n_harm, harm_mask=(1 << n_harm) - 1, cand_cap=300,
                  harm_index=1)
    ld = (n + 3) // 4 * 4 + pad
    s = fd.Searcher(p, n, thresh=thresholds.threshold_array(n_harm, n_temp, sigma=4.5))
    d_plane = torch.full((n_temp, ld), 1e30, device="cuda")
    d_plane[:, :n] = torch.from_numpy(plane).cuda()
    with np.errstate(invalid="ignore"):
        ref = harmonic.detect(plane, s.thresh_host, n_harm, p.harm_mask, 300, index="highest")
    s.ws.fill_(0xAB)
    fd.fdas_harmonic_sum(p, d_plane, n, ld, s.thresh, s.cands, s.counts, s.peaks, s.ws, s.ws_bytes)
    cands, counts, peaks = s.results()
    none = (np.float32(0.0), 255 - n_temp // 2, 0xFFFFFF)
    ref.peaks[:] = [none if r[0] < 0 else r for r in ref.peaks]
    if max(ref.counts) > 16384:  # more than the workspace keeps: only counts and peaks are exact
        ref.cands, cands = [], []
    assert_same_candidates(cands, counts, peaks, ref, p.harm_mask)


def test_first_host_search_of_a_thread_leaves_an_open_capture_alone(fd):
    """fdas_search_host keeps page-locked words per thread. A thread's first call makes them while another thread
    captures a graph in thread-local mode, as a batch plan does: the capture survives, and both results are
    right. (In global mode no host call that waits is allowed in any thread.)"""
    import threading

    import torch

    p, n = fd.Params(n_temp=9, z_min=-4, n_harm=4, harm_mask=0xF), 5000
    a, b = fd.Searcher(p, n), fd.Searcher(p, n)
    spec = _spectrum(n, 7)
    host = spec.cpu().pin_memory()
    a.search(spec)
    want = a.results()
    a.counts.zero_()
    error, stream = [], torch.cuda.Stream()

    def other():
        try:
            b.search_host(host, stream=stream)
        except Exception as e:  # noqa: BLE001
            error.append(e)

    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        a.search(spec)
        t = threading.Thread(target=other)
        t.start()
        t.join()
    assert not error, error
    g.replay()
    torch.cuda.synchronize()
    for got in (a.results(), b.results(host=True)):
        assert np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
        assert all(np.array_equal(x, y) for x, y in zip(got[0], want[0]))


def test_end_of_a_host_search_thread_leaves_a_global_capture_alone(fd):
    """The thread's page-locked words are given back at its end, here while another thread captures a graph in
    global mode: the capture survives."""
    import threading
    import time

    import torch

    p, n = fd.Params(n_temp=9, z_min=-4, n_harm=4, harm_mask=0xF), 5000
    a, b = fd.Searcher(p, n), fd.Searcher(p, n)
    spec = _spectrum(n, 7)
    host, stream = spec.cpu().pin_memory(), torch.cuda.Stream()
    searched, go = threading.Event(), threading.Event()

    def other():
        b.search_host(host, stream=stream)
        searched.set()
        go.wait(60)

    t = threading.Thread(target=other)
    t.start()
    assert searched.wait(60)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="global"):
        a.search(spec)
        go.set()
        t.join()
        time.sleep(0.3)  # the thread's own storage goes after it has been joined
    g.replay()
    torch.cuda.synchronize()
    got, want = a.results(), b.results(host=True)
    assert np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_a_plan_tunes_the_kernel_it_replays(fd, prec):
    """tune() times the convolution that takes HP_1: it leaves every spectrum's HP_1 count in the workspace (its first
    word), and the plan's results are those of a search."""
    import torch

    p = fd.Params(n_temp=9, z_min=-4, n_harm=4, harm_mask=0xF, precision=prec)
    b = fd.Batch(p, [20000, 4099, 33333], thresh=thresholds.threshold_array(4, 9, sigma=3.0))
    for k, n in enumerate(b.lengths):
        b.specs[k].copy_(_spectrum(n, k))
    plan = b.plan()
    b.ws.fill_(0xAB)
    plan.tune()
    torch.cuda.synchronize()
    words = b.ws.view(torch.int64).view(len(b.lengths), -1)
    want = [int((b.planes[k][:, :n] > b.thresh[0][:, None]).sum()) for k, n in enumerate(b.lengths)]
    assert [int(c) for c in words[:, 0].cpu()] == want and min(want) > 0
    plan.launch()
    torch.cuda.synchronize()
    got = [b.results(k) for k in range(3)]
    for k, n in enumerate(b.lengths):
        s = fd.Searcher(p, n, thresh=b.thresh.cpu().numpy())
        s.search(b.specs[k])
        cands, counts, peaks = s.results()
        assert np.array_equal(got[k][1], counts) and np.array_equal(got[k][2], peaks)
        assert all(np.array_equal(x, y) for x, y in zip(got[k][0], cands))
    plan.close()


def _dependent_edges(graph):
    """(number of edges, number of programmatic ones) of a captured graph."""
    import ctypes

    rt = ctypes.CDLL("libcudart.so.13")
    raw, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert rt.cudaGraphGetEdges(raw, None, None, None, ctypes.byref(n)) == 0
    src, dst = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)()
    data = (ctypes.c_uint8 * (8 * n.value))()  # from_port, to_port, type, reserved[5]
    assert rt.cudaGraphGetEdges(raw, src, dst, data, ctypes.byref(n)) == 0
    return n.value, sum(data[8 * k + 2] == 1 for k in range(n.value))


@pytest.mark.parametrize("n_harm,prec,index", [(1, 0, 0), (1, 1, 0), (4, 0, 0), (4, 2, 0), (1, 0, 1), (4, 0, 1)])
def test_the_stages_never_overlap_a_callers_kernel(fd, n_harm, prec, index):
    """Each stage of a search called on its own behind a kernel of the caller: what a stage launches first waits for it
    in full, and only what follows inside the stage starts early. (With one plane the second stage is one kernel.)"""
    import torch

    if not hasattr(torch.cuda.CUDAGraph, "raw_cuda_graph"):
        pytest.skip("no access to the captured graph")
    p, n = fd.Params(n_temp=9, z_min=-4, n_harm=n_harm, harm_mask=(1 << n_harm) - 1, precision=prec, harm_index=index), 5000
    s, spec, x = fd.Searcher(p, n), _spectrum(n, 7), torch.zeros(8, device="cuda")
    s.search(spec)
    want = s.results()
    stages = (lambda: fd.fdas_search_convolve(p, spec, n, s.tmpl, s.plane, s.ld, s.thresh, s.ws, s.ws_bytes),
              lambda: fd.fdas_search_harmonic(p, s.plane, n, s.ld, s.thresh, s.cands, s.counts, s.peaks, s.ws, s.ws_bytes))
    for stage in stages:
        stage()  # no first-use work inside the capture
    for stage, kernels in zip(stages, (1 if index else 2, 3 if index else 2 if n_harm > 1 else 1)):
        g = torch.cuda.CUDAGraph(keep_graph=True)
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            x.add_(1)
            stage()
        edges, early = _dependent_edges(g)
        assert edges == kernels and early == kernels - 1, (edges, early)
        g.instantiate()
        g.replay()
    torch.cuda.synchronize()
    got = s.results()
    assert np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
