"""GPU parity of the QKV projection whose epilogue rotates queries and keys (16 pairs of several heads a tile), through a one-layer model."""
import numpy as np
import pytest
import torch

from oracle import forward as F
from paper_2506_10848_b200 import binding as sfs
from paper_2506_10848_b200 import workloads as W

from bf16_reference import forward_bf16_points

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# at most 128 rows: a last tile of fewer heads (10 heads of 64, 6 and 9 of 128: tiles of 2, 4 or 6), ragged rows; more rows: tiles of whole
# heads where they divide (8 and 16 heads), a rotary kernel where they do not; several sequences, whose positions begin again
@pytest.mark.parametrize("heads,dh,B,S", [(10, 64, 1, 40), (6, 128, 1, 128), (9, 128, 3, 40), (8, 128, 1, 136), (8, 128, 2, 264), (16, 64, 1, 520),
                                          (8, 128, 3, 344), (10, 64, 2, 200), (9, 128, 1, 264)])
def test_logits_match_the_oracle(heads, dh, B, S):
    d = heads * dh
    shape = W.Shape(n_layers=1, d_model=d, n_heads=heads, head_dim=dh, d_ff=64, vocab=512, mask_id=511, rms_eps=1e-5, rope_theta=1e4, logit_scale=1.0)
    # weights large enough that attention depends on the rotation
    w = W.model_weights(shape, seed=d + S, std=0.08, gain_std=0.2)
    wd = {k: (v.to(DEV) if k != "layers" else [{kk: vv.to(DEV) for kk, vv in lw.items()} for lw in v]) for k, v in w.items()}
    model = sfs.Model(shape, wd)
    tok = W.prompt_ids(B, S, 510, seed=S)
    session = sfs.sfs_session_create(model, B, S)
    try:
        rows = [(b, t) for b in range(B) for t in range(0, S, 3)]
        d_rows = torch.tensor([b * S + t for b, t in rows], dtype=torch.int32, device=DEV)
        got = torch.zeros((len(rows), shape.vocab), dtype=torch.float32, device=DEV)
        sfs.sfs_forward(session, tok.to(DEV), B, S, d_rows, None, len(rows), got, sfs.LOGITS_F32)
        sfs.sfs_check_device_status()
        cfg = F.ModelConfig(**shape.asdict())
        ref = F.forward(cfg, W.weights_to_numpy(w, np.float64), tok.numpy(), rows=rows, dtype=np.float64)
        err = got.cpu().double().numpy() - ref
        # the bar is what rounding the operands to bf16 costs by itself at these weights, with a quarter more for other last bits
        emu = np.concatenate([forward_bf16_points(cfg, w, tok[b].numpy(), [t for bb, t in rows if bb == b]) for b in range(B)]) - ref
        assert np.linalg.norm(err) <= 1.25 * np.linalg.norm(emu)
        assert np.linalg.norm(err, axis=1).max() <= 1.6 * np.linalg.norm(emu, axis=1).max()
    finally:
        sfs.sfs_session_destroy(session)
        model.close()
