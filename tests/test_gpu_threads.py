"""Several host threads, each with a context and a stream of its own: what is set per function of the library (shared-memory limits)
may not depend on the size of one call."""
from __future__ import annotations

import threading

import numpy as np
import pytest

from paper_2509_25188_b200 import workloads as wl
from tests.helpers import small_shape

pytestmark = pytest.mark.gpu


def _together(jobs):
    """Runs the jobs in threads of their own, started together; raises what any of them raised."""
    import torch
    gate, errors = threading.Barrier(len(jobs)), []

    def run(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                gate.wait()
                job()
        except Exception as e:   # noqa: BLE001  (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def _decodes(dec, prompts, G, n, want):
    def job():
        for _ in range(n):
            toks, _, _, _ = dec.decode(prompts, G)
            assert np.array_equal(toks, want)
    return job


@pytest.mark.parametrize("shapes", [
    # blocks of 16 and 32: other records of the decision kernel
    [(dict(n_layers=1), 16, 16, 32), (dict(n_layers=1), 32, 16, 32)],
    # heads of 32 and 256, one and several key tiles: other tiles of the fp32 attention
    [(dict(n_layers=1), 16, 16, 32), (dict(n_layers=1, n_heads=1, head_dim=256), 16, 80, 32)]])
def test_contexts_of_different_sizes_decode_at_once(shapes):
    from paper_2509_25188_b200 import binding
    decs, jobs = [], []
    for kw, s, P, G in shapes:
        shape = small_shape(**kw)
        dec = binding.Decoder(shape, wl.make_weights(shape, seed=0, final_norm_gain=wl.spread_gain(shape)), None, block_len=s,
                              max_batch=1, max_seq=P + G, use_filter=False)
        prompts = wl.make_prompts(1, P, shape, seed=3)
        want = dec.decode(prompts, G)[0]
        decs.append(dec)
        jobs.append(_decodes(dec, prompts, G, 150, want))
    _together(jobs)
    for dec in decs:
        dec.close()


def test_filters_of_different_depths_train_at_once():
    """Filters of three and four layers share a kernel; what they hold in shared memory differs in size.  One update a launch, so that
    a call prepares a thousand of them."""
    import ctypes
    import torch
    from paper_2509_25188_b200 import binding as b
    s, n, epochs = 16, 32, 1000
    rng = np.random.default_rng(0)
    c = torch.from_numpy(rng.random((n, s), dtype=np.float32)).cuda()
    y = (c > 0.6).to(torch.uint8)
    cfg = b.TrainConfig(1e-3, 0.9, 0.999, 1e-8, 0.01, epochs, 0)

    def job(depth):
        layers = [((np.eye(s) + 0.1 * rng.standard_normal((s, s))).astype(np.float32), np.zeros(s, np.float32)) for _ in range(depth)]
        want, _ = b.filter_train_layers(layers, c, y, epochs)
        w, bias = [torch.from_numpy(q).cuda() for q, _ in layers], [torch.from_numpy(q).cuda() for _, q in layers]
        pw, pb = ((ctypes.c_void_p * depth)(*[t.data_ptr() for t in ts]) for ts in (w, bias))
        losses = np.zeros(epochs, np.float32)
        torch.cuda.synchronize()

        def run():
            r = b.lib.l2pd_debug_filter_train(torch.cuda.current_stream().cuda_stream, s, depth, n, c.data_ptr(), y.data_ptr(), pw, pb,
                                              ctypes.byref(cfg), losses.ctypes.data, 1, 2_000_000_000, -1)
            assert r == 0, b.lib.l2pd_last_error(None).decode()
            for t, u, (ww, wb) in zip(w, bias, want):
                assert np.array_equal(t.cpu().numpy(), ww) and np.array_equal(u.cpu().numpy(), wb)
        return run
    _together([job(3), job(4)])
