"""GPU parity of the QKV projection whose epilogue rotates queries and keys (16 pairs of several heads a tile): through a one-layer model, and
bit for bit against the plain projection and its rotary kernel."""
import ctypes
import os
import subprocess

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


CSRC = os.path.join(os.path.dirname(sfs.__file__), "csrc")


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    """The library's two forms of the projection, whichever of them a forward pass would take."""
    so = str(tmp_path_factory.mktemp("qkv") / "qkv_forms.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-I", "/usr/local/cuda/include",
                    os.path.join(os.path.dirname(os.path.abspath(__file__)), "qkv_forms.cpp"), "-o", so], check=True)
    sfs.lib()
    ctypes.CDLL(sfs.LIB_PATH, mode=ctypes.RTLD_GLOBAL)
    lib = ctypes.CDLL(so)
    p, i = ctypes.c_void_p, ctypes.c_int32
    lib.qkv_table.argtypes = [p, i, i, ctypes.c_float]
    lib.qkv_rotates.argtypes = [i] * 4
    lib.qkv_project.argtypes = [p, p] + [i] * 6 + [p] * 6 + [i] * 3
    return lib


# M rows; heads of dh; tokens T of sequences of S; listed: the rows are listed tokens, some of them twice; mb, bn: tile of the rotating form (0: the
# planner's).  At most 128 rows: the kernel for few rows, last tiles of fewer heads.  mb 1 and 2: the pair kernel with one and two blocks of 256 rows
@pytest.mark.parametrize("M,heads,dh,S,T,listed,mb,bn", [
    (40, 10, 64, 40, 40, False, 0, 0), (120, 9, 128, 40, 120, False, 0, 0), (128, 6, 128, 64, 128, False, 0, 256), (8, 16, 128, 8, 8, False, 0, 64),
    (128, 32, 128, 1536, 1536, True, 0, 0), (52, 9, 128, 264, 264, True, 0, 192), (77, 10, 64, 120, 240, True, 0, 128), (1, 6, 128, 72, 72, True, 0, 0),
    (40, 1, 128, 40, 40, False, 0, 0), (24, 1, 64, 48, 48, True, 0, 0), (16, 3, 64, 16, 16, False, 0, 128),
    (136, 8, 128, 136, 136, False, 1, 256), (528, 8, 128, 264, 528, False, 2, 256), (520, 16, 64, 520, 520, False, 2, 128), (1032, 32, 128, 344, 1032, False, 0, 0),
    (200, 8, 128, 512, 1024, True, 1, 64), (384, 8, 128, 768, 1536, True, 2, 128), (400, 9, 128, 200, 400, False, 1, 256)])
def test_both_forms_give_the_same_bits(forms, M, heads, dh, S, T, listed, mb, bn):
    n = K = heads * dh
    g = torch.Generator(device=DEV).manual_seed(M + n)
    h = torch.randn((M, K), generator=g, device=DEV).to(torch.bfloat16)
    w = [(torch.randn((n, K), generator=g, device=DEV) * K ** -0.5).to(torch.bfloat16) for _ in range(3)]
    wp = (ctypes.c_void_p * 3)(*[t.data_ptr() for t in w])
    table = torch.zeros((S, dh // 2, 2), dtype=torch.float32, device=DEV)
    sfs._check(forms.qkv_table(table.data_ptr(), S, dh, 1e4))
    rows = None
    if listed:
        rows = torch.randperm(T, generator=torch.Generator().manual_seed(M))[:M].sort().values.to(torch.int32)
        if M > 4:
            rows[-3:] = rows[-4]                             # the row choice pads its list by repeating the last one
        rows = rows.to(DEV)
        h[-3:] = h[-4 if M > 4 else -1]                      # (a token's rows are the same)
    out = []
    for rotate in (0, 1):
        qk = torch.full((M, 2 * n), 7.0, dtype=torch.bfloat16, device=DEV)
        k_dst, vt, compact = (torch.full(shape, 7.0, dtype=torch.bfloat16, device=DEV) for shape in ((T, n), (n, T), (n, T)))
        torch.cuda.synchronize()
        sfs._check(forms.qkv_project(h.data_ptr(), wp, M, K, heads, dh, S, T, table.data_ptr(), rows.data_ptr() if listed else None,
                                     k_dst.data_ptr() if listed or M % 16 == 0 else None, qk.data_ptr(), vt.data_ptr(), compact.data_ptr(), rotate, mb, bn))
        sfs.sfs_check_device_status()
        # queries; the keys where they were asked for (a plain projection leaves the unrotated ones in qk as well)
        out.append((qk[:, :n], k_dst if listed or M % 16 == 0 else qk[:, n:], k_dst, vt))
    for a, b in zip(*out):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    assert not torch.equal(out[0][0][M - 1], torch.full_like(out[0][0][0], 7.0))


def rotary_launches(heads, dh, B, S):
    """Launches of the rotary kernel in a forward pass of one layer."""
    d = heads * dh
    shape = W.Shape(n_layers=1, d_model=d, n_heads=heads, head_dim=dh, d_ff=64, vocab=512, mask_id=511, rms_eps=1e-5, rope_theta=1e4, logit_scale=1.0)
    model = sfs.Model(shape, W.model_weights(shape, seed=1, device=DEV))
    session = sfs.sfs_session_create(model, B, S)
    try:
        out = torch.zeros((8, shape.vocab), dtype=torch.float32, device=DEV)
        rows = torch.arange(8, dtype=torch.int32, device=DEV)
        sfs.sfs_profile(session, True)
        sfs.sfs_forward(session, W.prompt_ids(B, S, 510, seed=1).to(DEV), B, S, rows, None, 8, out, sfs.LOGITS_F32)
        return sfs.sfs_profile(session, False)[1]["rope"]
    finally:
        sfs.sfs_session_destroy(session)
        model.close()


@pytest.mark.parametrize("heads,dh,B,S", [(10, 64, 1, 40), (9, 128, 3, 40), (32, 128, 1, 104), (32, 128, 1, 512), (32, 128, 1, 1000), (8, 128, 2, 264), (9, 128, 1, 264)])
def test_a_rotary_kernel_runs_where_the_projection_does_not_rotate(forms, heads, dh, B, S):
    assert rotary_launches(heads, dh, B, S) == (0 if forms.qkv_rotates(B * S, heads * dh, heads, dh) else 1)


# at the 8B width 512 rows want tiles that whole heads do not fill
def test_forms_at_the_8b_width(forms):
    assert [forms.qkv_rotates(M, 4096, 32, 128) for M in (128, 512, 1000, 1536, 2048, 6144)] == [1, 0, 1, 1, 1, 1]


# up to 128 rows: beyond 48 heads of 128 one wave takes two weight blocks a tile, which only the plain form has
def test_forms_of_few_rows(forms):
    for M in (8, 64, 128):
        assert [forms.qkv_rotates(M, 128 * heads, heads, 128) for heads in (6, 9, 16, 20, 32, 48, 49, 56, 64)] == [1, 1, 1, 1, 1, 1, 0, 0, 0]
        assert [forms.qkv_rotates(M, 64 * heads, heads, 64) for heads in (10, 16, 32, 64)] == [1, 1, 1, 1]
