"""Steps replayed as recorded graphs against the same steps launched one by one (a session that is being profiled never replays): from
its sixteenth use on a kind of step sets the arguments of recorded launches, and everything a call brings has to reach them."""
import threading

import pytest
import torch

from paper_2506_10848_b200 import binding as sfs
from paper_2506_10848_b200 import workloads as W

from test_gpu_cache import state_tensor

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CALLS = 40
WIDE = W.Shape(n_layers=2, d_model=1024, n_heads=8, head_dim=128, d_ff=1536, vocab=5000, mask_id=4999, rms_eps=1e-5, rope_theta=10000.0, logit_scale=1.0)


class Pair:
    """One model, a session that replays and one that does not; every output buffer is new to its call."""

    def __init__(self, shape, B, S):
        self.model = sfs.Model(shape, W.model_weights(shape, seed=12, gain_std=0.2, device=DEV))
        self.sessions = [sfs.sfs_session_create(self.model, B, S) for _ in range(2)]
        sfs.sfs_profile(self.sessions[1], True)

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        for s in self.sessions:
            sfs.sfs_session_destroy(s)
        self.model.close()

    def both(self, call, rows, vocab, dtype):
        out = [torch.full((rows, vocab), 3.0, device=DEV, dtype=torch.float32 if dtype == sfs.LOGITS_F32 else torch.bfloat16) for _ in range(2)]
        for s, o in zip(self.sessions, out):
            call(s, o)
        sfs.sfs_check_device_status()
        assert torch.equal(out[0], out[1]), int((out[0] != out[1]).sum())
        return out                                      # (kept by the caller: the next call's buffers lie elsewhere)


def draw_rows(g, B, S, first, cap):
    n = int(torch.randint(1, cap + 1, (1,), generator=g))
    where = torch.randperm(B * (S - first), generator=g)[:n]
    rows = torch.zeros(cap, dtype=torch.int32)
    rows[:n] = (where // (S - first) * S + first + where % (S - first)).to(torch.int32)
    return rows.to(DEV), torch.tensor([n], dtype=torch.int32, device=DEV)


@pytest.mark.parametrize("shape,lengths", [(W.TINY, [(1, 64)]), (WIDE, [(2, 72)]), (WIDE, [(1, 72), (1, 160)])])
def test_replayed_forward_takes_every_argument_of_its_call(shape, lengths):
    g = torch.Generator().manual_seed(5)
    kept = []
    with Pair(shape, 2, 160) as p:
        for call in range(CALLS * len(lengths)):
            B, S = lengths[call // 20 % len(lengths)]       # two lengths in turn: plans and recordings come and go
            tok = torch.randint(0, shape.vocab, (B, S), generator=g, dtype=torch.int32).to(DEV)
            for dtype, listed, counted in ((sfs.LOGITS_F32, True, True), (sfs.LOGITS_BF16, False, False), (sfs.LOGITS_BF16, True, False)):
                rows, n = draw_rows(g, B, S, 0, 24) if listed else (None, None)
                cap = 24 if listed else B * S
                kept.append((tok, rows, n, p.both(lambda s, o: sfs.sfs_forward(s, tok, B, S, rows, n if counted else None, cap, o, dtype), cap, shape.vocab, dtype)))
            kept = kept[-9:]


@pytest.mark.parametrize("shape,B,P,L,kp,kr", [(W.TINY, 1, 24, 40, 12, 4), (W.TINY, 2, 23, 41, 100, 3), (WIDE, 1, 33, 87, 9, 3), (WIDE, 2, 24, 40, 100, 2)])
def test_replayed_cached_steps_take_every_argument_of_their_call(shape, B, P, L, kp, kr):
    g, S = torch.Generator().manual_seed(6), P + L
    kept = []
    with Pair(shape, B, S) as p:
        for s in p.sessions:
            sfs.sfs_cache_enable(s, kp, kr, 0.25)
        tok = torch.randint(0, shape.vocab, (B, S), generator=g, dtype=torch.int32)
        for call in range(3 * CALLS):
            tok[:, P:] = torch.where(torch.rand((B, L), generator=g) < 0.1, torch.randint(0, shape.vocab, (B, L), generator=g, dtype=torch.int32), tok[:, P:])
            d_tok = tok.to(DEV)
            lo = int(torch.randint(0, L // 2, (1,), generator=g))
            state = state_tensor(B, call % 2, lo, lo + L // 2)
            rows, n = draw_rows(g, B, S, P, 24)
            kept.append((d_tok, state, rows, n, p.both(lambda s, o: sfs.sfs_forward_cached(s, d_tok, B, S, P, state, rows, n, 24, o, sfs.LOGITS_BF16), 24, shape.vocab,
                                                       sfs.LOGITS_BF16)))
            kept = kept[-9:]


@pytest.mark.parametrize("where", ["same thread", "other thread"])
def test_recording_does_not_end_a_capture_that_goes_on_elsewhere(where):
    """A program captures work of its own (in the mode that watches all threads) while steps run on another stream: their recording, replay
    and the loss of a recording when the length changes leave that capture alone, and the capture leaves them alone."""
    shape = W.TINY
    with Pair(shape, 1, 64) as p:
        session, stream = p.sessions[0], torch.cuda.Stream()
        tok = W.prompt_ids(1, 64, shape.vocab, seed=1).to(DEV)
        out, plain = {}, {}
        for S in (64, 56):
            out[S], plain[S] = (torch.zeros((S, shape.vocab), dtype=torch.bfloat16, device=DEV) for _ in range(2))
            sfs.sfs_forward(p.sessions[1], tok, 1, S, None, None, S, plain[S], sfs.LOGITS_BF16)
        raised = []

        def calls(S, n):
            try:
                torch.cuda.set_device(0)
                for _ in range(n):
                    sfs.sfs_forward(session, tok, 1, S, None, None, S, out[S], sfs.LOGITS_BF16, stream=stream)
            except Exception as e:  # noqa: BLE001
                raised.append(e)

        def steps():
            calls(64, 30)
            calls(56, 30)
            calls(64, 3)

        calls(64, 3)                                            # what a first call sets up is set up
        torch.cuda.synchronize()
        x, g = torch.zeros(1000, device=DEV), torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode="global"):
            x += 1
            if where == "same thread":
                steps()
            else:
                t = threading.Thread(target=steps)
                t.start()
                t.join()
            x += 1
        g.replay()
        torch.cuda.synchronize()
        assert not raised and torch.all(x == 2.0)
        assert all(torch.equal(out[S], plain[S]) for S in out)
