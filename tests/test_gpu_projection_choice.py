"""Which kernel a step's projections take, and what may not depend on it: the launch modes' agreement, the environment switches,
lockstep decodes with the oracle at the row counts and head sizes that reach each form.  The form that ran is told from the launches
of the kinds it does without (profile_read)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import l2pd_oracle as orc
from paper_2509_25188_b200 import workloads as wl
from tests.helpers import lockstep, oracle_model

pytestmark = pytest.mark.gpu

FIELDS = ("logits", "conf", "pred", "p", "unmask", "masks_left", "l_eff", "done", "forced")


def _shape(head_dim, n_heads, d, d_ff, layers=3):
    return wl.ModelShape(n_layers=layers, d_model=d, n_heads=n_heads, head_dim=head_dim, d_ff=d_ff, vocab=1000, rms_eps=1e-5,
                         rope_theta=10000.0, mask_id=999, eot_id=998, dtype="bf16")


def _decoder(shape, w, s, B, max_seq, kv=0, filt=None):
    from paper_2509_25188_b200 import binding
    return binding.Decoder(shape, w, filt, block_len=s, max_batch=B, max_seq=max_seq, kv_cache=kv, use_filter=filt is not None,
                           use_eotp=False)


def _launches(dec, kind):
    return dec.profile_read().get(kind, (0.0, 0))[1]


@pytest.mark.parametrize("head_dim,heads,kv,B,P,G,steps,unfused,m_side", [
    (128, 4, 2, 1, 172, 128, 1, False, True),    # 300 rows that fill the store
    (128, 4, 1, 3, 172, 128, 2, False, True),    # 900, then 384 rows against it
    (64, 8, 0, 2, 57, 96, 2, False, True),       # heads of 64: 306 rows
    (64, 8, 2, 1, 172, 128, 1, False, True),
    (64, 3, 0, 1, 193, 64, 2, False, False),     # q, k and v of 192 features: 257 rows
    (128, 4, 0, 1, 268, 32, 2, True, False)])    # the rotation kept apart by the switch
def test_modes_agree_where_the_rotation_is_not_fused(monkeypatch, head_dim, heads, kv, B, P, G, steps, unfused, m_side):
    """With more than 256 rows the three modes agree bit for bit also where q and k pass through bf16 before they are rotated.
    m_side: mode 0 rotates in a projection with the weights on the M side."""
    if unfused:
        monkeypatch.setenv("L2PD_NO_ROPE_FUSION", "1")
    shape = _shape(head_dim, heads, 512 if heads > 3 else 256, 1376)
    dec = _decoder(shape, wl.make_weights(shape, seed=0, final_norm_gain=wl.spread_gain(shape)), 32, B, P + G, kv)
    prompts = wl.make_prompts(B, P, shape, seed=5)
    got = []
    for mode in (0, 1, 2):
        dec.set_chain(mode)
        dec.state_reset(prompts, G)
        dec.profile_enable(["rope"])
        got.append([dec.denoise_step(want_logits=True) for _ in range(steps)])
        if not unfused:
            assert _launches(dec, "rope") == (0 if mode == 0 and m_side else steps * shape.n_layers)
        assert dec.last_step_rows > 256
    dec.close()
    for mode in (1, 2):
        for a, b in zip(got[0], got[mode]):
            for k in FIELDS:
                assert np.array_equal(a[k], b[k]), "mode %d and mode 0 differ in %s" % (mode, k)


@pytest.mark.parametrize("head_dim,heads,kv,B,L,m_side", [
    (64, 8, 0, 2, 153, True), (64, 8, 0, 2, 385, False),      # 306 and 770 rows
    (128, 4, 1, 1, 300, True), (128, 4, 1, 8, 512, False)])   # 300 and 4096 rows, with a store
def test_narrow_models_rotate_in_the_projection_only_where_that_is_faster(head_dim, heads, kv, B, L, m_side):
    """d = 512: few k-blocks, behind which the rotating epilogue of large tiles does not hide (step of 4 layers, rotation inside and
    apart: 306 rows 190 and 189 us, 770 rows 238 and 218; 300 rows with a store 188 and 196, 4096 rows 371 and 358)."""
    shape = _shape(head_dim, heads, 512, 1376)
    dec = _decoder(shape, wl.make_weights(shape, seed=0, final_norm_gain=1.0), 32, B, L, kv)
    dec.state_reset(wl.make_prompts(B, L - 32, shape, seed=5), 32)
    dec.profile_enable(["rope"])
    dec.denoise_step(outputs=False)
    assert _launches(dec, "rope") == (0 if m_side else shape.n_layers)
    dec.close()


@pytest.mark.parametrize("P", [12, 268])   # 44 and 300 rows
def test_switch_for_a_rotation_kernel_of_its_own(monkeypatch, P):
    shape = _shape(128, 4, 512, 1376)
    w = wl.make_weights(shape, seed=0, final_norm_gain=wl.spread_gain(shape))
    prompts = wl.make_prompts(1, P, shape, seed=5)
    logits = []
    for switch, rotations in (("0", 0), ("1", shape.n_layers)):
        monkeypatch.setenv("L2PD_NO_ROPE_FUSION", switch)
        dec = _decoder(shape, w, 32, 1, P + 32)
        dec.state_reset(prompts, 32)
        dec.profile_enable(["rope"])
        logits.append(dec.denoise_step(want_logits=True)["logits"][0])
        assert _launches(dec, "rope") == rotations
        dec.close()
    # q and k are rounded to bf16 once more
    assert np.abs(logits[1] - logits[0]).max() <= 2e-2 * np.abs(logits[0]).max()


@pytest.mark.parametrize("P,norms", [(12, 0), (268, 5)])   # 44 and 300 rows; RMSNorm kernels of a step of three layers
def test_switch_for_k_slices_in_completion_order(monkeypatch, P, norms):
    """Under the switch the slices add into x: no slices in a cluster (hence RMSNorm kernels), no partial sums to add (after the last
    layer a kernel of its own adds them)."""
    shape = _shape(128, 4, 512, 1376)
    w = wl.make_weights(shape, seed=0, final_norm_gain=wl.spread_gain(shape))
    m = oracle_model(shape, w)
    prompts = wl.make_prompts(1, P, shape, seed=5)
    for switch in ("0", "1"):
        monkeypatch.setenv("L2PD_ATOMIC_KSPLIT", switch)
        dec = _decoder(shape, w, 32, 1, P + 32)
        dec.profile_enable(["rmsnorm", "other"])
        lockstep(dec, m, None, orc.DecodeConfig(block_len=32, use_filter=False, use_eotp=False), prompts, 32, logit_rtol=2e-2,
                 conf_atol=1e-3, p_margin=0.02, max_steps=1)
        assert _launches(dec, "rmsnorm") == (5 if switch == "1" else norms)
        assert _launches(dec, "other") == (1 if switch == "0" and norms else 0)
        dec.close()


@pytest.mark.parametrize("head_dim,heads,d,d_ff,kv,s,B,P,G,m_side", [
    (64, 8, 512, 1376, 0, 32, 2, 110, 64, True),     # 348 rows, no cache; the down projection has two slices
    (64, 3, 1024, 2816, 0, 32, 1, 268, 32, True),    # 300 rows, q, k and v of 192 features: v ends inside a tile
    (64, 3, 256, 704, 0, 16, 1, 21, 16, True),       # the same in 37 rows
    (64, 8, 512, 1376, 2, 16, 1, 270, 32, True),     # 302 rows, then 16 against the store
    (64, 3, 256, 12288, 2, 8, 1, 272, 16, False),    # 288 rows, then 8; gate / up in tiles of 96 features, four slices of a cluster
    (64, 8, 512, 1376, 1, 16, 2, 250, 16, False),    # 532 rows, then 32 from the block's start
    (128, 2, 256, 12288, 2, 16, 1, 284, 32, True),   # 316 rows, then 16, heads of 128
    (128, 4, 512, 1376, 2, 5, 1, 300, 10, True)])    # 310 rows, then 5
def test_lockstep_where_the_weights_are_on_the_m_side(head_dim, heads, d, d_ff, kv, s, B, P, G, m_side):
    """Logits and decisions against the oracle's; bf16 roundings of two layers (2e-2 of a row's largest logit, as everywhere).
    m_side: the rotation is inside the projection in a block's first step too."""
    shape = _shape(head_dim, heads, d, d_ff, layers=2)
    w = wl.make_weights(shape, seed=1, final_norm_gain=wl.spread_gain(shape))
    dec = _decoder(shape, w, s, B, P + G, kv)
    dec.profile_enable(["rope", "rmsnorm"])
    st = lockstep(dec, oracle_model(shape, w), None,
                  orc.DecodeConfig(block_len=s, kv_cache=kv > 0, dual_cache=kv == 2, use_filter=False, use_eotp=False),
                  wl.make_prompts(B, P, shape, seed=2), G, logit_rtol=2e-2, conf_atol=1e-3, p_margin=0.02, max_steps=s + 2)
    rows = B * (P + G)
    # steps of at most 48 rows have neither rotation nor RMSNorm kernels
    first = sum(1 for i in range(st["steps"]) if kv == 0 or i in (0, s))
    assert _launches(dec, "rope") == (0 if m_side else 2 * first)
    assert _launches(dec, "rmsnorm") == (3 * first if rows > 48 else 0)
    assert st["replay_checked"] > 0 and st["pred_checked"] > 0
    dec.close()


def test_partial_sums_and_sums_in_a_cluster_are_the_ones_that_ran():
    """306 rows at d = 512: the down projection's slices leave partial sums, which a kernel adds after the last layer; 33 rows: sums
    meet in clusters and no kernel adds or normalises.  (A plan without slices would take the test from the lockstep above.)"""
    shape = _shape(64, 8, 512, 1376, layers=2)
    w = wl.make_weights(shape, seed=1, final_norm_gain=wl.spread_gain(shape))
    for P, added, norms in ((274, 1, 3), (1, 0, 0)):
        dec = _decoder(shape, w, 32, 1, P + 32)
        dec.state_reset(wl.make_prompts(1, P, shape, seed=2), 32)
        dec.profile_enable(["other", "rmsnorm"])
        dec.denoise_step(outputs=False)
        assert (_launches(dec, "other"), _launches(dec, "rmsnorm")) == (added, norms)
        dec.close()
