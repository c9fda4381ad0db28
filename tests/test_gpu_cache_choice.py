"""The row choice of cached partial steps, derived without the library's similarities: residual branches of zero keep every layer's
input the embedding, so the value vectors are one projection each, and the sums of the similarity are replayed in numpy operation by
operation.  What decides among unchanged rows is the last bit of those sums."""
import numpy as np
import pytest
import torch

from oracle import cache as C
from paper_2506_10848_b200 import binding as sfs
from paper_2506_10848_b200 import workloads as W

from test_gpu_cache import state_tensor

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SLICES = 32                                  # the similarity's feature slices


def silent_model(d, head_dim, n_layers, d_ff, vocab, seed):
    """Embeddings of +-1 and a norm gain per layer: RMSNorm is exact (mean square 1; the epsilon is far below half a bf16 ulp), so the
    input of layer l's projections is embedding * gain_l.  W_o and W_down are zero: x stays the embedding."""
    shape = W.Shape(n_layers=n_layers, d_model=d, n_heads=d // head_dim, head_dim=head_dim, d_ff=d_ff, vocab=vocab, mask_id=vocab - 1, rms_eps=1e-6,
                    rope_theta=10000.0, logit_scale=1.0)
    w = W.model_weights(shape, seed=seed, gain_std=0.2, device=DEV)
    w["tok_emb"].copy_(torch.where(w["tok_emb"] >= 0, 1.0, -1.0))
    for layer in w["layers"]:
        layer["wo"].zero_()
        layer["w_down"].zero_()
    return shape, w


def value_rows(w, layer, tokens):
    """bf16 V of every token [n, d] as float32, by one projection whose sum runs over all of K."""
    lw = w["layers"][layer]
    h = (w["tok_emb"][tokens.long()].float() * lw["attn_norm"].float()).to(torch.bfloat16).contiguous()
    n, d = h.shape
    v = torch.zeros((n, d), dtype=torch.bfloat16, device=DEV)
    sfs.sfs_linear(h, d, lw["wv"], d, v, d, n, d, d, 0, 1.0)
    sfs.sfs_check_device_status()
    return v.float().cpu().numpy()


def ordered_sum(a, b):
    """sum over the features of a * b in the kernels' order: a slice's features go to eight running sums, those are added, then the slices.
    A product of two bf16 values is exact in fp32, so a fused multiply-add is one rounded addition."""
    n, d = a.shape
    p = np.zeros((n, SLICES, -(-d // SLICES)), np.float32)
    p.reshape(n, -1)[:, :d] = a * b
    per = p.shape[2]
    p = np.concatenate([p, np.zeros((n, SLICES, -per % 8), np.float32)], axis=2).reshape(n, SLICES, -1, 8)
    run = np.zeros((n, SLICES, 8), np.float32)
    for u in range(p.shape[2]):
        run = run + p[:, :, u]
    sl = run[:, :, 0]
    for k in range(1, 8):
        sl = sl + run[:, :, k]
    tot = np.zeros(n, np.float32)
    for s in range(SLICES):
        tot = tot + sl[:, s]
    return tot


def similarity(a, b):
    return ordered_sum(a, b) / (np.sqrt(ordered_sum(a, a)) * np.sqrt(ordered_sum(b, b)))


# one sequence (odd and even first response token) and two; a small model; as many K ranges as a planner might like for few rows; the
# long prompt; a width that is no multiple of 8 slices
@pytest.mark.parametrize("d,head_dim,B,P,L", [(256, 64, 1, 32, 64), (256, 64, 2, 24, 40), (384, 128, 1, 9, 55), (2048, 128, 1, 19, 197), (2048, 128, 1, 64, 256),
                                              (2048, 128, 2, 40, 120), (4096, 128, 1, 1024, 512), (4096, 128, 1, 24, 768)])
def test_row_sets_are_those_of_the_unsplit_values(d, head_dim, B, P, L):
    nl, S, rho = 2, P + L, 0.25
    shape, w = silent_model(d, head_dim, nl, 256, 1024, seed=d + L)
    model = sfs.Model(shape, w)
    session = sfs.sfs_session_create(model, B, S)
    try:
        sfs.sfs_cache_enable(session, 100, 4, rho)
        g = torch.Generator().manual_seed(L)
        tok = torch.full((B, S), shape.mask_id, dtype=torch.int32)
        tok[:, :P + L // 2] = torch.randint(0, shape.vocab - 1, (B, P + L // 2), generator=g, dtype=torch.int32)
        n_adapt = C.adaptive_count(rho, L)
        lg = torch.zeros((B * S, shape.vocab), dtype=torch.bfloat16, device=DEV)
        rows = torch.arange(B * S, dtype=torch.int32, device=DEV)
        sets = torch.zeros((nl * B * S,), dtype=torch.int32, device=DEV)
        sims = torch.zeros((nl, B, L), dtype=torch.float32, device=DEV)
        cached = None
        for step in range(7):
            for b in range(B):                                    # nothing changed before the second step; then two tokens a step
                for i in ([] if step < 2 else [(17 * step + 5 * b) % L, (L // 2 + 3 * step) % L]):
                    tok[b, P + i] = int(torch.randint(0, shape.vocab - 1, (1,), generator=g))
            fast = step in (3, 6)
            span = (L // 4, L // 4 + 3 * L // 8) if fast else (0, L)
            state = state_tensor(B, 1, *span) if fast else state_tensor(B)
            n_sel = sfs.sfs_forward_cached(session, tok.to(DEV), B, S, P, state, rows, None, B * S, lg, sfs.LOGITS_BF16, sets=sets, sims=sims)
            sfs.sfs_check_device_status()
            fresh = [value_rows(w, l, tok[:, P:].reshape(-1).to(DEV)).reshape(B, L, d) for l in range(nl)]
            if step % 4 == 0:
                cached = [f.copy() for f in fresh]
                continue
            got_sets, got_sims = sets[:nl * B * n_sel].cpu().numpy().reshape(nl, B, n_sel), sims.cpu().numpy()
            for l in range(nl):
                for b in range(B):
                    sim = similarity(fresh[l][b], cached[l][b])
                    assert np.array_equal(got_sims[l, b].view(np.uint32), sim.astype(np.float32).view(np.uint32)), \
                        (step, l, b, int((got_sims[l, b] != sim).sum()))
                    cand = list(range(*span))
                    mine = C.least_similar(sim[cand], cand, min(n_adapt, len(cand)))
                    assert sorted(set(int(r) - b * S - P for r in got_sets[l, b])) == mine, (step, l, b)
                    cached[l][b][mine] = fresh[l][b][mine]
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


# a candidate takes 4 bytes of the choice's shared memory, a recomputed row 4 per feature: both sides of the 48 KB that a launch has unasked
@pytest.mark.parametrize("d,P,L", [(128, 8, 10240), (128, 8, 12256), (128, 8, 12280), (128, 8, 12288), (12288, 8, 8)])
def test_shared_memory_of_long_responses_and_wide_models(d, P, L):
    shape = W.Shape(n_layers=1, d_model=d, n_heads=d // 128, head_dim=128, d_ff=128, vocab=64, mask_id=63, rms_eps=1e-5, rope_theta=10000.0, logit_scale=1.0)
    model = sfs.Model(shape, W.model_weights(shape, seed=1, device=DEV))
    session = sfs.sfs_session_create(model, 1, P + L)
    try:
        sfs.sfs_cache_enable(session, 100, 100, 0.25)
        tok = W.prompt_ids(1, P + L, shape.vocab, seed=2).to(DEV)
        rows = torch.arange(P + L - 8, P + L, dtype=torch.int32, device=DEV)
        lg = [torch.zeros((8, shape.vocab), dtype=torch.float32, device=DEV) for _ in range(2)]
        sets, sims = torch.zeros(P + L, dtype=torch.int32, device=DEV), torch.zeros(L, dtype=torch.float32, device=DEV)
        for step in range(2):
            if step:
                tok[0, P:P + L // 8] = 1
            n_sel = sfs.sfs_forward_cached(session, tok, 1, P + L, P, None, rows, None, 8, lg[step], sfs.LOGITS_F32, sets=sets, sims=sims)
        sfs.sfs_check_device_status()
        assert sorted(int(r) - P for r in sets[:n_sel]) == C.least_similar(sims.cpu().numpy(), list(range(L)), C.adaptive_count(0.25, L))
        assert bool(torch.isfinite(lg[1]).all())
    finally:
        sfs.sfs_session_destroy(session)
        model.close()
