"""Projections of at most 128 rows (CTA pairs, tensor-memory tiles of 64 rows per CTA): edges of the row, column and K tiles, and the
row statistics the LM head leaves when a generation has that few response rows."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import forward as F
from oracle import rowstats as RS
from oracle.scheduler import SlowFastState, rows_needed, slowfast_step
from paper_2506_10848_b200 import binding as sfs
from paper_2506_10848_b200 import workloads as W

from bf16_reference import forward_bf16_points
from helpers import params_pair
from test_gpu_linear import run

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# rows on both sides of a CTA's 64; one tile, a ragged last tile and one that ends inside an N-block; K of one k-block, a tail of 8
@pytest.mark.parametrize("M", [1, 63, 64, 65, 127, 128])
@pytest.mark.parametrize("N,K", [(8, 64), (3000, 136), (9480, 520), (40008, 72)])
def test_linear_edges(M, N, K):
    for out_dtype in (0, 1):
        got, ref = run(M, N, K, out_dtype, seed=M + N)
        err = np.abs(got - ref)
        # fp32 sums of K exact products (at most K roundings of 2^-24 of the running sum, |terms| < 4); bf16 output: half an ulp more
        assert np.all(err <= 4.0 * K * K * 2.0 ** -24 + (2.0 ** -8 * np.abs(ref) if out_dtype == 0 else 0.0)), float(err.max())


@pytest.mark.parametrize("B,L,vocab,scale", [(1, 24, 70008, 60.0), (2, 61, 65536, 60.0), (1, 128, 99992, 60.0), (1, 40, 70008, 600.0), (2, 131, 65544, 600.0)])
def test_generation_with_few_long_rows_is_reproduced_by_the_oracle(B, L, vocab, scale):
    """Long vocabulary rows, at most 128 of them (ragged last column tile): the decisions come from the LM head's own records.  At the
    larger scale most rows' other terms all truncate to zero (several rows tie exactly at S_q = 2^28); the last case has more rows."""
    P = 8 - L % 8
    S = P + L
    shape = W.Shape(n_layers=1, d_model=256, n_heads=2, head_dim=128, d_ff=512, vocab=vocab, mask_id=vocab - 1, rms_eps=1e-5,
                    rope_theta=10000.0, logit_scale=scale)
    w = W.model_weights(shape, seed=9, device=DEV)
    model = sfs.Model(shape, w)
    session = sfs.sfs_session_create(model, B, S)
    po, pg = params_pair()
    try:
        trace = torch.zeros((L, B, sfs.TRACE_INTS), dtype=torch.int32, device=DEV)
        dump = torch.zeros((B * L, vocab), dtype=torch.bfloat16, device=DEV)
        rows_d = torch.zeros(B * L, dtype=torch.int32, device=DEV)
        n_d = torch.zeros(1, dtype=torch.int32, device=DEV)
        sfs.sfs_generate_begin(session, W.prompt_ids(B, P, vocab - 2, seed=1).to(DEV), B, P, L, pg)
        ost = [SlowFastState.fresh(L, po) for _ in range(B)]
        for step in range(6):
            if all(s.done for s in ost):
                break
            sfs.sfs_generate_steps(session, 1, trace, L, dump, rows_d, n_d)
            torch.cuda.synchronize()
            need = [(b, i) for b in range(B) for i in rows_needed(ost[b])]
            assert rows_d[:int(n_d.item())].tolist() == [b * S + P + i for (b, i) in need]
            st = RS.row_stats(W.bf16_bits(dump[:len(need)].cpu()))
            for b in range(B):
                if ost[b].done:
                    continue
                idx = {i: j for j, (bb, i) in enumerate(need) if bb == b}
                rec = slowfast_step(ost[b], {i: int(st["argmax"][j]) for i, j in idx.items()}, {i: int(st["sq"][j]) for i, j in idx.items()}, po)
                assert trace[step, b].tolist()[:6] == [rec.phase, rec.s, rec.hi, rec.e_cand, rec.stable, len(rec.positions)], (step, b)
        sfs.sfs_check_device_status()
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


# small models (fused 32 x 32 tiles): rows below, at and across a tile; both head widths; a d_ff whose K tail is 8; a ragged vocabulary;
# the last shape has one row tile more than these kernels take
@pytest.mark.parametrize("dims", [dict(d_model=256, n_heads=4, head_dim=64, d_ff=1000, vocab=1000), dict(d_model=384, n_heads=3, head_dim=128, d_ff=264, vocab=4104),
                                  # more LM-head tiles than one wave: the projections in front stay fused, the LM head is the tensor-memory kernel's
                                  dict(d_model=256, n_heads=2, head_dim=128, d_ff=264, vocab=10000)])
@pytest.mark.parametrize("B,S", [(1, 8), (3, 8), (1, 40), (2, 24), (1, 712)])
def test_small_model_edges(dims, B, S):
    shape = W.Shape(n_layers=2, mask_id=dims["vocab"] - 1, rms_eps=1e-5, rope_theta=10000.0, logit_scale=8.0, **dims)
    w = W.model_weights(shape, seed=6, gain_std=0.2)
    wd = {k: (v.to(DEV) if k != "layers" else [{kk: vv.to(DEV) for kk, vv in lw.items()} for lw in v]) for k, v in w.items()}
    model = sfs.Model(shape, wd)
    session = sfs.sfs_session_create(model, B, S)
    try:
        tok = W.prompt_ids(B, S, shape.vocab, seed=S)
        picked = [(b, t) for b in range(B) for t in range(0, S, max(1, S // 9))]
        n, cap = len(picked), B * S                              # fewer rows than the call allows for
        rows = torch.zeros(cap, dtype=torch.int32); rows[:n] = torch.tensor([b * S + t for b, t in picked])
        for dtype in (sfs.LOGITS_F32, sfs.LOGITS_BF16):
            lg = torch.full((cap, shape.vocab), 7.0, dtype=torch.float32 if dtype else torch.bfloat16, device=DEV)
            sfs.sfs_forward(session, tok.to(DEV), B, S, rows.to(DEV), torch.tensor([n], dtype=torch.int32, device=DEV), cap, lg, dtype)
            sfs.sfs_check_device_status()
            assert torch.all(lg[n:] == 7.0)                       # rows beyond the device's count untouched
            got = lg[:n].float().cpu().double().numpy()
            ref = F.forward(F.ModelConfig(**shape.asdict()), W.weights_to_numpy(w, np.float64), tok.numpy(), rows=picked, dtype=np.float64)
            # what rounding to bf16 at the stored operands alone gives, plus 10 % (and the rounding of a stored bf16 logit: 2^-9 rms)
            emu = np.concatenate([forward_bf16_points(F.ModelConfig(**shape.asdict()), w, tok[b].numpy(), [t for bb, t in picked if bb == b]) for b in range(B)])
            rel, rel_model = np.linalg.norm(got - ref) / np.linalg.norm(ref), np.linalg.norm(emu - ref) / np.linalg.norm(ref)
            assert rel <= 1.10 * rel_model + (0.0 if dtype else 2.0 ** -9), (rel, rel_model)
            # a list of exactly n entries; the same without a count (fewer rows in the call's bound may be another kernel's)
            again = torch.zeros_like(lg)
            sfs.sfs_forward(session, tok.to(DEV), B, S, rows[:n].clone().to(DEV), torch.tensor([n], dtype=torch.int32, device=DEV), cap, again, dtype)
            sfs.sfs_check_device_status()
            assert torch.equal(again[:n], lg[:n])
            sfs.sfs_forward(session, tok.to(DEV), B, S, rows[:n].clone().to(DEV), None, n, again, dtype)
            sfs.sfs_check_device_status()
            rel = np.linalg.norm(again[:n].float().cpu().double().numpy() - ref) / np.linalg.norm(ref)
            assert rel <= 1.10 * rel_model + (0.0 if dtype else 2.0 ** -9), (rel, rel_model)
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


# d_ff 344 to 368: tiles near the 48 KB of shared memory that a launch has unasked.  A process of its own: what a launch has once asked
# for stays granted, and other tests ask for more.
@pytest.mark.parametrize("d_ff", [312, 336, 344, 368, 376])
def test_small_model_is_the_first_to_use_its_shared_memory(d_ff):
    code = f"""if True:
        import torch
        from paper_2506_10848_b200 import binding as sfs, workloads as W
        shape = W.Shape(n_layers=1, d_model=128, n_heads=2, head_dim=64, d_ff={d_ff}, vocab=512, mask_id=511, rms_eps=1e-5, rope_theta=10000.0, logit_scale=1.0)
        model = sfs.Model(shape, W.model_weights(shape, seed=1, device="cuda:0"))
        session = sfs.sfs_session_create(model, 1, 64)
        out = torch.full((64, 512), float("nan"), device="cuda:0")
        sfs.sfs_forward(session, W.prompt_ids(1, 64, 512, seed=1).to("cuda:0"), 1, 64, None, None, 64, out, sfs.LOGITS_F32)
        sfs.sfs_check_device_status()
        assert bool(torch.isfinite(out).all())
    """
    r = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


# heads of 64, short sequences: one key block, blocks that end inside a warp's share, keys over 4 and 8 warps, one and two row tiles
# per CTA, a last row tile of 8 rows, the longest of them
@pytest.mark.parametrize("B,S,H", [(1, 8, 1), (2, 40, 3), (1, 128, 4), (1, 136, 4), (4, 224, 4), (8, 64, 8), (1, 512, 4), (2, 264, 8)])
def test_short_attention_edges(B, S, H):
    d = H * 64
    g = torch.Generator().manual_seed(S)
    q, k, v = (torch.randn((B * S, d), generator=g).to(torch.bfloat16) for _ in range(3))
    out = torch.zeros((B * S, d), dtype=torch.bfloat16, device=DEV)
    sfs.sfs_attention(torch.cat([2 * q, k], dim=1).contiguous().to(DEV), v.t().contiguous().to(DEV), out, B, S, H, 64)
    sfs.sfs_check_device_status()
    got = out.cpu().double().numpy()
    for b in range(B):
        sl = slice(b * S, (b + 1) * S)
        qq, kk, vv = (t[sl].double().numpy().reshape(S, H, 64) for t in (2 * q, k, v))
        ref, mag = F.attention(qq, kk, vv).reshape(S, d), F.attention(qq, kk, np.abs(vv)).reshape(S, d)
        # probabilities and the output rounded to bf16 (unit roundoff 2^-8 each), exponentials to about 2^-20
        assert np.all(np.abs(got[sl] - ref) <= 2.0 ** -8 * (mag + np.abs(ref)) + 2.0 ** -16), b


@pytest.mark.parametrize("scale,B,L,kw", [(60.0, 1, 64, {}), (60.0, 3, 40, {}), (1.0, 2, 24, {}), (8.0, 1, 1, {}),
                                          (60.0, 1, 32, dict(sampler=sfs.SAMPLER_RANDOM, max_steps=4)), (8.0, 2, 16, dict(k_slow=5, k_fast=3))])
def test_generation_enqueues_what_it_needs(scale, B, L, kw):
    """The host runs ahead of the device except where a step may be the last: the same tokens as step by step, at most one step more."""
    dct = W.TINY.asdict()
    dct["logit_scale"] = scale
    shape, P = W.Shape(**dct), 8 - L % 8
    model = sfs.Model(shape, W.model_weights(shape, seed=4, device=DEV))
    session = sfs.sfs_session_create(model, B, P + L)
    try:
        prompt = W.prompt_ids(B, P, shape.vocab - 2, seed=2).to(DEV)
        params = sfs.Params.default(**kw)
        one, whole = (torch.zeros((B, P + L), dtype=torch.int32, device=DEV) for _ in range(2))
        state = torch.zeros((B, sfs.STATE_INTS), dtype=torch.int32, device=DEV)
        sfs.sfs_generate_begin(session, prompt, B, P, L, params)
        before, steps, active = sfs.sfs_profile(session, False, read=False)[2], 0, B
        while active:
            sfs.sfs_generate_steps(session, 1)
            active, steps = sfs.sfs_generate_end(session, one)
        per_step = (sfs.sfs_profile(session, False, read=False)[2] - before) / steps
        for _ in range(3):
            before = sfs.sfs_profile(session, False, read=False)[2]
            sfs.sfs_generate(session, prompt, B, P, L, params, whole, state_out=state)
            enqueued = round((sfs.sfs_profile(session, False, read=False)[2] - before) / per_step)
            done = int(state[:, sfs.STATE_FIELDS.index("steps_done")].max())
            assert done == steps and done <= enqueued <= done + 1, (steps, done, enqueued)
            assert torch.equal(one, whole)
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


@pytest.mark.parametrize("P,L", [(16, 24), (19, 197), (8, 712)])
def test_similarities_of_unchanged_tokens(P, L):
    """With nothing changed the fresh values are the cached ones bit for bit, so the three sums are one number a, and a / (sqrt(a) sqrt(a)) is
    1 up to the roundings of the root (twice), the product and the quotient: 4 * 2^-24."""
    shape = W.Shape(n_layers=1, d_model=2048, n_heads=16, head_dim=128, d_ff=256, vocab=1024, mask_id=1023, rms_eps=1e-5,
                    rope_theta=10000.0, logit_scale=1.0)
    model = sfs.Model(shape, W.model_weights(shape, seed=3, device=DEV))
    S = P + L
    session = sfs.sfs_session_create(model, 1, S)
    try:
        sfs.sfs_cache_enable(session, 100, 100, 0.25)
        tok = W.prompt_ids(1, S, shape.vocab, seed=5).to(DEV)
        rows = torch.arange(P, S, dtype=torch.int32, device=DEV)
        lg = torch.zeros((L, shape.vocab), dtype=torch.bfloat16, device=DEV)
        sims = torch.zeros((1, 1, L), dtype=torch.float32, device=DEV)
        for step in range(2):
            sfs.sfs_forward_cached(session, tok, 1, S, P, None, rows, None, L, lg, sfs.LOGITS_BF16, sims=sims if step else None)
        sfs.sfs_check_device_status()
        assert float((1.0 - sims).abs().max()) <= 2.0 ** -22
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


# the widths at which rows have fewer, as many and more 16-byte chunks than a block has threads
@pytest.mark.parametrize("d,head_dim,d_ff,S", [(384, 128, 1536, 480), (640, 128, 256, 304), (2048, 128, 256, 304), (2560, 128, 256, 304), (4096, 128, 256, 304),
                                               (5120, 128, 256, 304)])
def test_norm_of_a_row_does_not_depend_on_how_many_rows_there_are(d, head_dim, d_ff, S):
    """The full refresh normalises all tokens, a partial step the response, a call the rows it is asked for: each row must come out the
    same, bit for bit (the identity as head shows the final norm's output)."""
    shape = W.Shape(n_layers=1, d_model=d, n_heads=d // head_dim, head_dim=head_dim, d_ff=d_ff, vocab=d, mask_id=d - 1, rms_eps=1e-5, rope_theta=10000.0,
                    logit_scale=1.0)
    w = W.model_weights(shape, seed=d, gain_std=0.2, device=DEV)
    w["lm_head"].copy_(torch.eye(d, device=DEV))
    model = sfs.Model(shape, w)
    session = sfs.sfs_session_create(model, 1, S)
    try:
        tok = W.prompt_ids(1, S, d, seed=1).to(DEV)
        every = torch.zeros((S, d), dtype=torch.float32, device=DEV)
        sfs.sfs_forward(session, tok, 1, S, None, None, S, every, sfs.LOGITS_F32)
        for n in (1, 50, 288):
            rows = torch.randperm(S, generator=torch.Generator().manual_seed(n))[:n].to(torch.int32).to(DEV)
            some = torch.zeros((n, d), dtype=torch.float32, device=DEV)
            sfs.sfs_forward(session, tok, 1, S, rows, None, n, some, sfs.LOGITS_F32)
            sfs.sfs_check_device_status()
            assert torch.equal(some, every[rows.long()]), (n, int((some != every[rows.long()]).sum()))
    finally:
        sfs.sfs_session_destroy(session)
        model.close()
