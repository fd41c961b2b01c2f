"""Contexts of different sizes used from several host threads at once (the
bindings release the interpreter lock): every call succeeds and returns what it
returns alone."""

import threading

import pytest
import torch

import workloads
from tests.pair_setup import gpu_pair

pytestmark = pytest.mark.gpu


def _run(jobs):
    errors = []

    def guarded(f):
        try:
            f()
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    ts = [threading.Thread(target=guarded, args=(f,)) for f in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors[0]


def _pair(n, stream):
    fp, m0, m1 = workloads.film_pair_plain(n, 2, 3)
    fp.u0 = (0.3, -0.2, 0.0)
    return gpu_pair(fp, m0, m1, mech=False, stream=stream)


def test_gradients_of_short_and_long_boxes_side_by_side():
    """The transposed prefilter's shared memory grows with a box axis: under 2 KB
    for the short ones here, beyond the 48 KB any kernel may have for the long one."""
    sizes = [(6, 5, 1), (7, 6, 1), (5, 6, 1), (600, 20, 1)]
    streams = [torch.cuda.Stream() for _ in sizes]
    mms = [_pair(n, s) for n, s in zip(sizes, streams)]
    alone = [mm.backward_energy(0)[1:] for mm in mms]
    torch.cuda.synchronize()

    def loop(mm, ref, stream):
        with torch.cuda.stream(stream):
            for _ in range(400):
                gs, gt = mm.backward_energy(0)[1:]
            stream.synchronize()
        torch.testing.assert_close(gs, ref[0], rtol=1e-5, atol=1e-5 * ref[0].abs().max().item())
        torch.testing.assert_close(gt, ref[1], rtol=1e-5, atol=1e-5 * ref[1].abs().max().item())

    _run([lambda i=i: loop(mms[i], alone[i], streams[i]) for i in range(len(sizes))])
    for mm in mms:
        mm.close()


def test_contexts_of_short_and_long_lines_built_side_by_side():
    """The spectra's set-up transforms whole lines in shared memory: 1 KB for the
    short films, beyond 48 KB for the long one."""

    def build(n, times):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for _ in range(times):
                mm = _pair(n, stream)
                H = mm.compute_demag(0)
                stream.synchronize()
                assert torch.isfinite(H).all()
                mm.close()

    _run([lambda: build((1700, 4, 1), 12)] + [lambda: build((6, 5, 1), 60)] * 2)
