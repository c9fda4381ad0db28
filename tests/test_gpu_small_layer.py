"""GPU parity of the fused layer of small models (attention to the next QKV projection in one launch) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import forward as F
from paper_2506_10848_b200 import binding as sfs
from paper_2506_10848_b200 import workloads as W

from bf16_reference import forward_bf16_points

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# tokens below, at and above a tile of 16 and of 32 rows; one tile of features per CTA or none for some (d_ff 8, 24), an odd number of them
# (24, 56, 344, 1032), an even one; both widths; several sequences with ragged last tiles; row tiles of 32 (2 x 224, 7 x 40, 240)
@pytest.mark.parametrize("d,ff,B,S", [(256, 688, 1, 8), (256, 688, 1, 40), (256, 688, 3, 24), (256, 8, 1, 16), (256, 24, 2, 72), (256, 344, 1, 200),
                                      (128, 352, 1, 24), (128, 1032, 2, 40), (128, 64, 1, 136), (256, 688, 2, 224), (128, 1032, 7, 40),
                                      (256, 344, 1, 408), (128, 24, 7, 40), (128, 56, 1, 240)])
def test_logits_match_the_oracle(d, ff, B, S):
    dct = W.TINY.asdict()
    dct.update(n_layers=3, d_model=d, d_ff=ff, n_heads=d // 64, vocab=512, mask_id=511, logit_scale=1.0)
    shape = W.Shape(**dct)
    # weights large enough that attention is not uniform and both branches move the residual stream
    w = W.model_weights(shape, seed=d + ff, std=0.08, gain_std=0.2)
    wd = {k: (v.to(DEV) if k != "layers" else [{kk: vv.to(DEV) for kk, vv in lw.items()} for lw in v]) for k, v in w.items()}
    model = sfs.Model(shape, wd)
    tok = W.prompt_ids(B, S, 510, seed=S)
    session = sfs.sfs_session_create(model, B, S)
    try:
        got = torch.zeros((B * S, shape.vocab), dtype=torch.float32, device=DEV)
        sfs.sfs_forward(session, tok.to(DEV), B, S, None, None, B * S, got, sfs.LOGITS_F32)
        again = torch.zeros_like(got)
        sfs.sfs_forward(session, tok.to(DEV), B, S, None, None, B * S, again, sfs.LOGITS_F32)
        sfs.sfs_check_device_status()
        assert torch.equal(got, again)
        rows = [(b, t) for b in range(B) for t in range(S)]
        ref = F.forward(F.ModelConfig(**shape.asdict()), W.weights_to_numpy(w, np.float64), tok.numpy(), rows=rows, dtype=np.float64)
        err = got.cpu().double().numpy() - ref
        # the bar is what rounding the operands to bf16 costs by itself at these weights, with a quarter more for other last bits
        emu = np.concatenate([forward_bf16_points(F.ModelConfig(**shape.asdict()), w, tok[b].numpy(), range(S)) for b in range(B)]) - ref
        assert np.linalg.norm(err) <= 1.25 * np.linalg.norm(emu)
        assert np.linalg.norm(err, axis=1).max() <= 1.6 * np.linalg.norm(emu, axis=1).max()
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


def leave_nan_in_shared_memory():
    """A forward pass whose weights are NaN throughout: what its kernels leave in shared memory is NaN almost everywhere."""
    dct = W.TINY.asdict()
    dct.update(n_layers=2, d_model=128, d_ff=1024, n_heads=2, vocab=4096, mask_id=4095, logit_scale=1.0)
    shape = W.Shape(**dct)
    w = W.model_weights(shape, seed=0)
    for t in [v for k, v in w.items() if k != "layers"] + [v for lw in w["layers"] for v in lw.values()]:
        t.fill_(float("nan"))
    wd = {k: (v.to(DEV) if k != "layers" else [{kk: vv.to(DEV) for kk, vv in lw.items()} for lw in v]) for k, v in w.items()}
    model = sfs.Model(shape, wd)
    session = sfs.sfs_session_create(model, 1, 448)
    try:
        logits = torch.zeros((448, shape.vocab), dtype=torch.float32, device=DEV)
        sfs.sfs_forward(session, W.prompt_ids(1, 448, 4094, seed=0).to(DEV), 1, 448, None, None, 448, logits, sfs.LOGITS_F32)
        sfs.sfs_check_device_status()
        assert torch.isnan(logits).all()
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


# fewer tiles of features than CTAs: the first CTA has none, and the half k-step beside an odd last tile has no features to read.  Row tiles of
# 32 (15 and more tiles of 16), whose row 16 would then read the padding between two weight rows, which nobody writes
@pytest.mark.parametrize("ff", [8, 24, 40, 56])
@pytest.mark.parametrize("B,S", [(1, 240), (7, 40)])
def test_what_other_kernels_left_in_shared_memory_is_not_read(ff, B, S):
    dct = W.TINY.asdict()
    dct.update(n_layers=3, d_model=128, d_ff=ff, n_heads=2, vocab=512, mask_id=511, logit_scale=1.0)
    shape = W.Shape(**dct)
    w = W.model_weights(shape, seed=ff, std=0.08, gain_std=0.2)
    wd = {k: (v.to(DEV) if k != "layers" else [{kk: vv.to(DEV) for kk, vv in lw.items()} for lw in v]) for k, v in w.items()}
    model = sfs.Model(shape, wd)
    tok = W.prompt_ids(B, S, 510, seed=S).to(DEV)
    session = sfs.sfs_session_create(model, B, S)
    try:
        first = None
        for _ in range(4):
            leave_nan_in_shared_memory()
            got = torch.zeros((B * S, shape.vocab), dtype=torch.float32, device=DEV)
            sfs.sfs_forward(session, tok, B, S, None, None, B * S, got, sfs.LOGITS_F32)
            sfs.sfs_check_device_status()
            assert torch.isfinite(got).all(), torch.unique((~torch.isfinite(got)).any(dim=1).nonzero()[:, 0] % S).tolist()
            first = got if first is None else first
            assert torch.equal(got, first)
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


# two heads: attention units for two, four, and (a single sequence of 440 tokens, 32-row tiles) four of a cluster's eight CTAs
@pytest.mark.parametrize("B,P,L", [(1, 40, 32), (3, 88, 32), (1, 392, 48)])
def test_steps_after_the_last_sequence_is_done_change_nothing(B, P, L):
    """All steps enqueued at once: those after the end find no active sequence and leave the kernel early, and the next generation is as
    the first."""
    dct = W.TINY.asdict()
    dct.update(n_layers=3, d_model=128, d_ff=352, n_heads=2, vocab=512, mask_id=511, logit_scale=60.0)
    shape = W.Shape(**dct)
    model = sfs.Model(shape, W.model_weights(shape, seed=3, std=0.08, gain_std=0.2, device=DEV))
    session = sfs.sfs_session_create(model, B, P + L)
    prompt = W.prompt_ids(B, P, 510, seed=L).to(DEV)
    try:
        want = torch.zeros((B, P + L), dtype=torch.int32, device=DEV)
        state = torch.zeros((B, sfs.STATE_INTS), dtype=torch.int32, device=DEV)
        sfs.sfs_generate(session, prompt, B, P, L, sfs.Params.default(), want, state)
        done_after = int(state[:, sfs.STATE_FIELDS.index("steps_done")].max())
        assert done_after < L
        for _ in range(3):
            got, end = torch.zeros_like(want), torch.zeros_like(state)
            sfs.sfs_generate_begin(session, prompt, B, P, L, sfs.Params.default())
            sfs.sfs_generate_steps(session, L)
            sfs.sfs_generate_end(session, got, end)
            sfs.sfs_check_device_status()
            assert torch.equal(got, want) and torch.equal(end, state)
    finally:
        sfs.sfs_session_destroy(session)
        model.close()
