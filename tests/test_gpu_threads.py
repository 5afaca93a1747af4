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
