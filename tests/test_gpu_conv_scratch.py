"""Scratch of the single convolution calls (GB300): kept between calls across
synchronisations, bounded, given back, and one buffer per call in flight."""
import threading
import time

import numpy as np
import pytest

from test_gpu_wsnet import torch  # noqa: F401

pytestmark = pytest.mark.gpu


def _layer(torch, cin, cout, n, seed):  # noqa: F811
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.zeros(1, n + 2, n + 2, n + 2, cin, dtype=torch.bfloat16, device="cuda")
    x[:, 1:-1, 1:-1, 1:-1] = torch.randn(1, n, n, n, cin, generator=gen, device="cuda").bfloat16()
    w = torch.randn(cout, 27, cin, generator=gen, device="cuda").bfloat16()
    y = torch.empty(1, n + 2, n + 2, n + 2, cout, dtype=torch.bfloat16, device="cuda")
    return x, w, y


def _forward(t, stream):
    from paper_1806_10589_gb300 import conv3d_bf16

    x, w, y = t
    n = x.shape[1] - 2
    conv3d_bf16(0, x.data_ptr(), 0, w.data_ptr(), 0, 0, y.data_ptr(), 1, n, n, n, x.shape[4], y.shape[4], stream)


def test_scratch_is_kept_bounded_and_given_back(torch):  # noqa: F811
    from paper_1806_10589_gb300 import conv3d_release

    st = torch.cuda.current_stream()
    layers = [_layer(torch, c, c, 6, c) for c in (32, 64, 128, 256)]

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    for t in layers:  # kernels are loaded on their first use
        _forward(t, st)
    conv3d_release()
    empty = free()
    for t in layers:
        _forward(t, st)
    kept = free()
    for t in layers + layers:
        _forward(t, st)
        assert torch.cuda.mem_get_info()[0] == kept, "nothing is allocated again"
        assert free() == kept, "nothing is given back by a synchronisation"
    assert 0 <= empty - kept <= (16 << 20) + 4 * (2 << 20), "16 MB, in pages of 2 MB"
    conv3d_release()
    assert free() == empty


def test_a_call_after_a_synchronisation_costs_no_more(torch):  # noqa: F811
    """Median of single calls, each after a device synchronisation, against calls back
    to back: under twice (4 times when the synchronisation unmapped the scratch)."""
    st = torch.cuda.current_stream()
    t = _layer(torch, 32, 32, 6, 0)

    def us(sync):
        v = []
        for _ in range(60):
            if sync:
                torch.cuda.synchronize()
            a = time.perf_counter()
            _forward(t, st)
            v.append((time.perf_counter() - a) * 1e6)
        return float(np.median(v[10:]))

    alone, loop = us(True), us(False)
    assert alone <= 2 * loop, (alone, loop)


def test_calls_of_several_threads(torch):  # noqa: F811
    """Six threads with a stream each, layers of different sizes: the results of calls
    made one after another."""
    layers = [_layer(torch, 32 << (k % 4), 32 << (k % 3), 7, k) for k in range(6)]
    want = []
    for t in layers:
        _forward(t, torch.cuda.current_stream())
        want.append(t[2].clone())
    for t in layers:
        t[2].zero_()
    torch.cuda.synchronize()
    errors = []

    def work(t):
        try:
            s = torch.cuda.Stream()
            for _ in range(30):
                _forward(t, s)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in layers]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    for t, y in zip(layers, want):
        assert torch.equal(t[2], y)


def test_a_recording_stream_is_refused(torch):  # noqa: F811
    """The call ends with a synchronisation: under capture it reports an error, and the
    next call works."""
    from paper_1806_10589_gb300 import LBMError

    t = _layer(torch, 32, 32, 6, 1)
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        g.capture_begin(capture_error_mode="thread_local")
        t[2].add_(1)  # the graph is not empty
        with pytest.raises(LBMError):
            _forward(t, s)
        g.capture_end()
    _forward(t, torch.cuda.current_stream())
    assert bool(t[2].isfinite().all())
