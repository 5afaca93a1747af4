"""Algorithm 1 on the CUDA path: EGP sample collection (stage 1) and AdamW training of the filter
(stage 2, Eq. 6) against the oracle.

Tolerances: the kernel works in fp32, the oracle in fp64.  One update moves a parameter by about lr
whatever the gradient's size (Adam normalises it), so an fp32 error of relative size ~1e-6 in a gradient
component shifts the update by ~1e-6 * lr and the parameter error after T updates stays near T * lr * 1e-5
as long as no gradient component sits at rounding level; the tests use 200-300 updates at lr 1e-3..1e-2 and
compare parameters to 2e-3 absolute and the loss curve to 2e-4.
"""
from __future__ import annotations

import numpy as np
import pytest

from oracle import l2pd_oracle as orc
from paper_2509_25188_b200 import workloads as wl
from tests.helpers import oracle_model

pytestmark = pytest.mark.gpu


def _b():
    from paper_2509_25188_b200 import binding
    return binding


def _data(s, n, seed):
    rng = np.random.default_rng(seed)
    C = rng.uniform(0.0, 1.0, size=(n, s)).astype(np.float32)
    Y = (C + 0.15 * rng.normal(size=(n, s)) > 0.6).astype(np.uint8)
    return C, Y


@pytest.mark.parametrize("s,n,batch", [(32, 1000, 0), (32, 1000, 256), (16, 77, 0), (64, 333, 100), (5, 40, 0)])
def test_training_matches_the_oracle(s, n, batch):
    """Several tiles per block and a ragged last tile (n not a multiple of 32), ragged last batch,
    the largest block length (64) and an odd one."""
    C, Y = _data(s, n, seed=s + n)
    f0 = wl.make_filter(s, seed=3)
    epochs = 200 if batch == 0 else 60
    want, wl_losses = orc.train_filter(f0, C.astype(np.float64), Y.astype(np.float64), epochs, lr=5e-3, batch_size=batch)
    got, losses = _b().filter_train(f0, C, Y, epochs, lr=5e-3, batch_size=batch)
    assert len(losses) == len(wl_losses)
    assert np.abs(losses - wl_losses).max() < 2e-4
    assert abs(losses[0] - wl_losses[0]) < 2e-6                       # the first loss involves no update at all
    for k in ("w1", "b1", "w2", "b2"):
        assert np.abs(got[k] - want[k]).max() < 2e-3, k
    assert losses[-1] < losses[0]


def test_training_is_bit_reproducible_and_zero_epochs_is_identity():
    s, n = 32, 500
    C, Y = _data(s, n, seed=9)
    f0 = wl.make_filter(s, seed=4)
    a, la = _b().filter_train(f0, C, Y, 50)
    b, lb = _b().filter_train(f0, C, Y, 50)
    assert np.array_equal(la, lb) and all(np.array_equal(a[k], b[k]) for k in a)
    z, lz = _b().filter_train(f0, C, Y, 0)
    assert len(lz) == 0 and all(np.array_equal(z[k], f0[k].astype(np.float32)) for k in z)


def test_bad_arguments():
    b = _b()
    C, Y = _data(8, 10, seed=1)
    f0 = wl.make_filter(8, seed=1)
    with pytest.raises(b.L2pdError) as e:
        b.filter_train(f0, C, Y, 1, lr=0.0)
    assert e.value.status == -1
    C2, Y2 = _data(65, 4, seed=1)
    with pytest.raises(b.L2pdError) as e:
        b.filter_train(wl.make_filter(65, seed=1), C2, Y2, 1)
    assert e.value.status == -2


def test_egp_collection_then_training_end_to_end():
    """Stage 1 on the GPU: an EGP decode against the model's own one-token-per-step answer appends one
    (filter input, target) sample per step; the samples equal the oracle's for the same decode.  Stage 2
    on those samples lowers the loss, and the trained filter drives a decode that still ends."""
    b = _b()
    shape = wl.TINY
    w = wl.make_weights(shape, seed=0, final_norm_gain=wl.spread_gain(shape))
    d = wl.DECODES["C0"]
    s, G = d.block_len, d.gen_len
    m = oracle_model(shape, w)
    B = 2
    prompts = wl.make_prompts(B, d.prompt_len, shape, seed=5)
    van = orc.DecodeConfig(block_len=s, use_filter=False, use_eotp=False)
    refs = np.stack([orc.decode(m, None, p, G, van, keep_trace=False).response for p in prompts])
    f0 = wl.make_filter(s, d.tau, seed=0)
    dec = b.Decoder(shape, w, f0, block_len=s, tau=d.tau, max_batch=B, max_seq=d.prompt_len + G, use_eotp=False)
    dec.set_unmask_rule("egp", reference=refs)
    sink_c, sink_y = dec.set_collect(B * G)
    toks, _, steps, total = dec.decode(prompts, G)
    n = dec.collect_count
    assert n == int(steps.sum()) and np.array_equal(toks, refs)
    got_c, got_y = sink_c[:n].cpu().numpy(), sink_y[:n].cpu().numpy()
    # the oracle's samples, interleaved the same way: step by step, unfinished sequences in order
    cfg = orc.DecodeConfig(block_len=s, rule="egp", use_eotp=False)
    per_seq = []
    for i in range(B):
        r = orc.decode(m, f0, prompts[i], G, cfg, ref=refs[i])
        per_seq.append(orc.egp_samples(r.trace, refs[i], s))
        assert r.steps == steps[i]
    want_c, want_y = [], []
    for k in range(int(steps.max())):
        for i in range(B):
            if k < steps[i]:
                want_c.append(per_seq[i][0][k]); want_y.append(per_seq[i][1][k])
    want_c, want_y = np.stack(want_c), np.stack(want_y)
    assert np.abs(got_c - want_c).max() < 1e-3                  # fp32 model: confidences to 1e-3
    sure = np.abs(want_c - 0.5) < 2.0                           # all positions
    assert np.array_equal(got_y[sure], want_y[sure].astype(np.uint8))
    with pytest.raises(b.L2pdError):                            # a full sink refuses the step
        dec.set_collect(1)
        dec.state_reset(prompts, G)
        dec.denoise_step()
    dec.set_collect(0)
    trained, losses = b.filter_train(f0, got_c, got_y, 300, lr=1e-2)
    want_f, want_l = orc.train_filter(f0, got_c.astype(np.float64), got_y.astype(np.float64), 300, lr=1e-2)
    assert np.abs(losses - want_l).max() < 2e-4 and losses[-1] < losses[0]
    dec.close()
    dec2 = b.Decoder(shape, w, trained, block_len=s, tau=d.tau, max_batch=B, max_seq=d.prompt_len + G)
    toks2, out_len, steps2, _ = dec2.decode(prompts, G)
    ref2 = [orc.decode(m, trained, p, G, orc.DecodeConfig(block_len=s, tau=d.tau), keep_trace=False) for p in prompts]
    for i in range(B):
        assert steps2[i] == ref2[i].steps and np.array_equal(toks2[i], ref2[i].response)
    dec2.close()


@pytest.mark.parametrize("depth,s,n,batch", [(1, 32, 300, 0), (4, 32, 500, 128), (3, 16, 77, 0), (4, 64, 200, 0), (2, 64, 333, 100)])
def test_depth_variant_training_matches_the_oracle(depth, s, n, batch):
    """Section 4.4's one- and four-layer filters (and three): the tiled kernel's backpropagation through
    the layers against the oracle's, ragged tiles and batches included; depth 2 at s = 64 runs the same
    kernel as the two-layer entry point."""
    C, Y = _data(s, n, seed=depth * 100 + s)
    rng = np.random.default_rng(depth)
    layers0 = [((rng.normal(size=(s, s)) / np.sqrt(s)).astype(np.float32), (0.1 * rng.normal(size=s)).astype(np.float32))
               for _ in range(depth)]
    epochs = 120 if batch == 0 else 40
    want, want_l = orc.train_filter_layers(layers0, C.astype(np.float64), Y.astype(np.float64), epochs, lr=5e-3, batch_size=batch)
    got, losses = _b().filter_train_layers(layers0, C, Y, epochs, lr=5e-3, batch_size=batch)
    assert len(losses) == len(want_l) and np.abs(losses - want_l).max() < 2e-4
    for (w, b), (ww, wb) in zip(got, want):
        assert np.abs(w - ww).max() < 2e-3 and np.abs(b - wb).max() < 2e-3
    assert losses[-1] < losses[0]
    b_ = _b()
    with pytest.raises(b_.L2pdError) as e:
        b_.filter_train_layers(layers0 * 5, C, Y, 1)          # more than four layers
    assert e.value.status == -1


@pytest.mark.parametrize("s,n,depth,batch", [
    (1, 1, 1, 0), (31, 31, 2, 0), (32, 33, 1, 0), (33, 65, 2, 64),          # one position; edges of 32-sample tiles and of the padding to 32 / 64
    (32, 64 * 148 - 1, 2, 0), (32, 64 * 148 + 65, 2, 0),                     # either side of the step from tiles of 32 to tiles of 64
    (64, 64 * 148 + 1, 4, 0), (40, 9600, 3, 9500), (32, 20000, 4, 0)])       # the deepest filters on large tiles, a ragged last batch
def test_training_at_the_edges_of_its_tiles(s, n, depth, batch):
    """Parameters after 3 epochs and the losses against the oracle.  An update moves a parameter by at most about lr
    = 1e-3; where a gradient component sits at fp32 rounding level Adam can take either sign, 2 lr per update apart, so
    single parameters may differ by 2 lr x updates <= 1.2e-2; all others agree to 1e-5 (fp32 sums of n terms)."""
    C, Y = _data(s, n, seed=7 * s + n)
    rng = np.random.default_rng(5)
    layers = [(np.eye(s) + rng.normal(size=(s, s)) * 0.5 / np.sqrt(s), rng.normal(size=s) * 0.02) for _ in range(depth)]
    layers = [(w.astype(np.float32), b.astype(np.float32)) for w, b in layers]
    want, want_losses = orc.train_filter_layers(layers, C.astype(np.float64), Y.astype(np.float64), 3, lr=1e-3, batch_size=batch)
    got, losses = _b().filter_train_layers(layers, C, Y, 3, lr=1e-3, batch_size=batch)
    assert np.abs(losses - want_losses).max() < 1e-5
    for (gw, gb), (ww, wb) in zip(got, want):
        d = np.concatenate([np.abs(gw - ww).ravel(), np.abs(gb - wb).ravel()])
        assert d.max() <= 2e-3 * len(losses) + 1e-6
        assert np.mean(d > 1e-5) <= 0.01 + 1.0 / d.size


def test_a_meeting_that_runs_out_leaves_the_weights_alone():
    """One update to a launch, the third launch one arrival short (host-side hook; its wait gives up after 2 ms): the call
    reports the time-out, the caller's arrays keep their initial values although two updates had been made, and the next
    training on the same device is that of an untouched process."""
    import ctypes
    import torch
    b = _b()
    s, n, depth = 32, 3000, 2
    C, Y = _data(s, n, seed=2)
    c, y = torch.from_numpy(C).cuda(), torch.from_numpy(Y).cuda()
    rng = np.random.default_rng(8)
    layers = [((np.eye(s) + 0.1 * rng.normal(size=(s, s))).astype(np.float32), np.zeros(s, np.float32)) for _ in range(depth)]
    cfg = b.TrainConfig(1e-3, 0.9, 0.999, 1e-8, 0.01, 5, 0)

    def run(short_launch):
        w, bias = [torch.from_numpy(q).cuda() for q, _ in layers], [torch.from_numpy(q).cuda() for _, q in layers]
        pw, pb = ((ctypes.c_void_p * depth)(*[t.data_ptr() for t in ts]) for ts in (w, bias))
        losses = np.zeros(5, np.float32)
        r = b.lib.l2pd_debug_filter_train(torch.cuda.current_stream().cuda_stream, s, depth, n, c.data_ptr(), y.data_ptr(), pw, pb,
                                          ctypes.byref(cfg), losses.ctypes.data, 1, 2_000_000, short_launch)
        return r, [(u.cpu().numpy(), v.cpu().numpy()) for u, v in zip(w, bias)], losses

    before, _ = b.filter_train_layers(layers, C, Y, 5)
    r, got, _ = run(2)
    assert r == -5
    for (gw, gb), (w, bias) in zip(got, layers):
        assert np.array_equal(gw, w) and np.array_equal(gb, bias)
    r, got, losses = run(-1)                                      # the hook without a short launch: the ordinary training
    assert r == 0 and losses[-1] < losses[0]
    for (gw, gb), (w, bias) in zip(got, before):
        assert np.array_equal(gw, w) and np.array_equal(gb, bias)


def test_a_decode_on_another_stream_runs_beside_the_training():
    """The training's launches are short and few are queued: while 4,000 updates (some 160 ms) run in a thread on one stream,
    a decode on another gets its steps (0.1 ms each alone) between them, and both results are those of runs on their own.
    With one launch for all updates the decode got a single step."""
    import threading
    import torch
    b = _b()
    shape, d = wl.TINY, wl.DECODES["C0"]
    w = wl.make_weights(shape, seed=0, final_norm_gain=wl.spread_gain(shape))
    f0 = wl.make_filter(d.block_len, d.tau, seed=0)
    prompts = wl.make_prompts(1, d.prompt_len, shape, seed=1)
    dec = b.Decoder(shape, w, f0, block_len=d.block_len, tau=d.tau, max_batch=1, max_seq=d.prompt_len + d.gen_len)
    want_tokens, _, want_steps, _ = dec.decode(prompts, d.gen_len)
    g = torch.Generator(device="cuda").manual_seed(3)
    c = torch.rand(84480, 32, generator=g, device="cuda")
    y = (c > 0.6).to(torch.uint8)
    start = wl.make_filter(32, seed=3)
    want, want_losses = b.filter_train(start, c, y, 4000)
    got = []

    def train():
        torch.cuda.set_device(0)
        with torch.cuda.stream(torch.cuda.Stream()):
            got.append(b.filter_train(start, c, y, 4000))

    torch.cuda.synchronize()
    th = threading.Thread(target=train)
    th.start()
    steps = 0
    with torch.cuda.stream(torch.cuda.Stream()):
        while th.is_alive():
            tokens, _, n, _ = dec.decode(prompts, d.gen_len)
            assert np.array_equal(tokens, want_tokens) and np.array_equal(n, want_steps)
            steps += int(n[0])
    th.join()
    dec.close()
    assert np.array_equal(got[0][1], want_losses) and all(np.array_equal(got[0][0][k], want[k]) for k in want)
    assert steps >= 2 * int(want_steps[0])


@pytest.mark.parametrize("s,n,depth", [(64, 1024, 4), (64, 1024, 2), (32, 1024, 4)])
def test_gradients_of_small_batches_keep_their_accuracy(s, n, depth):
    """One update with eps far above every gradient moves a parameter by (lr / eps) x gradient, here 1e6 x: the parameters
    then hold the gradient to their own rounding.  Each of its components is a sum of n products, added in fp32 in some
    fifty blocks; the relative error (2-norm, worst matrix, median of four batches) stays below one unit in the last
    place, 2^-23, where rows of the blocks' sums added one after the other gave 1.4e-7."""
    errs = []
    for seed in range(4):
        C, Y = _data(s, n, seed=30 + seed)
        rng = np.random.default_rng(seed)
        layers = [((1.5 * (np.eye(s) + 0.5 * rng.normal(size=(s, s)) / np.sqrt(s))).astype(np.float32),
                   (0.02 * rng.normal(size=s)).astype(np.float32)) for _ in range(depth)]
        got, _ = _b().filter_train_layers(layers, C, Y, 1, lr=1e9, eps=1e3, weight_decay=0.0)
        _, grads = orc.filter_layers_loss_and_grads([(w.astype(np.float64), q.astype(np.float64)) for w, q in layers],
                                                    C.astype(np.float64), Y.astype(np.float64))
        worst = 0.0
        for new, old, grad in zip(got, layers, grads):
            for a, a0, g in zip(new, old, grad):
                want = 1e9 * g / (np.abs(g) + 1e3)
                worst = max(worst, np.linalg.norm(a0.astype(np.float64) - a - want) / np.linalg.norm(want))
        errs.append(worst)
    assert np.median(errs) < 2.0 ** -23


def test_the_kept_scratch_is_bounded_and_given_back():
    """A training keeps at most 32 MB of device memory for the next; l2pd_destroy(NULL) gives it back without a context."""
    import torch
    b = _b()
    C, Y = _data(64, 2000, seed=4)
    c, y = torch.from_numpy(C).cuda(), torch.from_numpy(Y).cuda()
    layers = [(np.eye(64, dtype=np.float32), np.zeros(64, np.float32))] * 4
    b.filter_train_layers(layers, c, y, 2)
    b.lib.l2pd_destroy(None)
    free0 = torch.cuda.mem_get_info()[0]
    b.filter_train_layers(layers, c, y, 2)
    kept = free0 - torch.cuda.mem_get_info()[0]
    assert 0 < kept <= 32 << 20
    b.lib.l2pd_destroy(None)
    assert torch.cuda.mem_get_info()[0] == free0


def test_losses_beyond_the_host_memory_are_an_error():
    """The copy of the losses (32 MB here) cannot be allocated in a process whose address space is limited: the call says so,
    before any launch, and nothing is thrown through the C interface."""
    import subprocess
    import sys
    code = """
import ctypes, resource
import numpy as np, torch
from paper_2509_25188_b200 import binding as b
c, y = torch.zeros(1, 1, device="cuda"), torch.zeros(1, 1, dtype=torch.uint8, device="cuda")
p = [torch.ones(1, device="cuda") for _ in range(4)]
losses = np.zeros(8 << 20, np.float32)
def train(epochs):
    cfg = b.TrainConfig(1e-3, 0.9, 0.999, 1e-8, 0.01, epochs, 0)
    return b.lib.l2pd_filter_train(None, 1, 1, c.data_ptr(), y.data_ptr(), *[t.data_ptr() for t in p], ctypes.byref(cfg), losses.ctypes.data)
assert train(3) == 0
torch.cuda.synchronize()
size = int(next(l for l in open("/proc/self/status") if l.startswith("VmSize")).split()[1]) << 10
resource.setrlimit(resource.RLIMIT_AS, (size + (16 << 20), resource.RLIM_INFINITY))
print("status", train(8 << 20))
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "status -3" in r.stdout, r.stdout + r.stderr
