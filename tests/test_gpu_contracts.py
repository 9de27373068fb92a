"""What the entry points promise beside their values on ordinary inputs: excluded scores, cuts of a sequence,
alignment, several host threads, and what an error leaves behind.

Slots are compared exactly.  Weights are within 2e-5 relative of float64 (fp32 scores and softmax, as in
tests/test_gpu_parity.py), or bit-equal where two calls have to agree.
"""
import threading

import numpy as np
import pytest

from oracle import sdm_oracle as O

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

from synth.torch_io import to_torch  # noqa: E402


@pytest.fixture(scope="module")
def sdm():
    import paper_2607_07386_gb300 as sdm
    from paper_2607_07386_gb300 import build as B
    B.build()
    return sdm


def _stored(x, dtype):
    return to_torch(O.to_bf16_bits(x) if dtype == "bf16" else np.asarray(x, np.float32), dtype)


def _lists(B, H, T, kw, kr):
    return [torch.empty((B, H, T, k), dtype=t, device="cuda") for k in (kw, kr) for t in (torch.int32, torch.float32)]


def _address(sdm, shape, P, x):
    out = _lists(shape.B, shape.H, shape.T, shape.k_write, shape.k_read)
    ws = torch.empty(sdm.workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    sdm.address(shape, P[0], P[1], x[0], x[1], *out, ws)
    torch.cuda.synchronize()
    return out


def _shifted(x):
    """The same values one element past the start of an allocation (element-aligned only)."""
    out = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)[1:].view(x.shape)
    out.copy_(x)
    return out


# ------------------------------------------------------------------ excluded scores

# one launch (tensor cores, FFMA) and the passes for large problems (two list lengths each)
@pytest.mark.parametrize("dtype,B,H,T,dk,S,k", [("bf16", 2, 2, 3, 64, 100, 8), ("f32", 1, 2, 7, 32, 70, 20),
                                                ("bf16", 1, 2, 1100, 128, 128, 32), ("bf16", 1, 1, 300, 64, 96, 40),
                                                ("f32", 1, 2, 2200, 16, 64, 24), ("bf16", 1, 1, 2100, 64, 600, 16)])
def test_rows_of_P_with_a_nan_are_never_selected(sdm, dtype, B, H, T, dk, S, k):
    """A row of P that holds a NaN has no score: the selection is the exact one over the other rows."""
    rng = np.random.default_rng(S + T)
    P = [O.round_storage(rng.standard_normal((H, 2 * S, dk)), dtype) for _ in range(2)]
    x = [O.round_storage(rng.standard_normal((B, H, T, dk)) / np.sqrt(dk), dtype) for _ in range(2)]
    gone = [3, S // 2, S + 1, 2 * S - 1]
    Pn = [p.copy() for p in P]
    for p in Pn:
        p[:, gone, dk // 3] = np.nan
    shape = sdm.SdmShape.make(B, H, T, dk, 16, S * S, k, k, dtype)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    sdm.device_status()
    got = _address(sdm, shape, [torch.from_numpy(p).cuda().to(dt) for p in Pn], [_stored(v, dtype) for v in x])
    assert sdm.device_status() == 0
    for side, (idx, w) in enumerate(((got[2], got[3]), (got[0], got[1]))):
        for b in range(B):
            for h in range(H):
                s = O.half_scores(P[side][h], x[side][b, h])
                s[:, gone] = -np.inf
                iw, _, ww = O.pkm_select(s[:, :S], s[:, S:], k)
                assert np.array_equal(idx[b, h].cpu().numpy(), iw), (side, b, h)
                assert np.all(np.abs(w[b, h].cpu().numpy() - ww) <= 2e-5 * ww), (side, b, h)


@pytest.mark.parametrize("dtype,T", [("bf16", 3), ("bf16", 2100), ("f32", 3), ("f32", 4200)])
def test_rows_with_a_nan_stay_out_of_the_rescans(sdm, dtype, T):
    """Near-equal scores around the boundary (a band past the kept list) beside rows with a NaN: the rescan of the
    whole half takes no NaN for a score either.  Every token is the same."""
    from tests.test_gpu_parity import _clustered_projection
    S, dk, k, x0 = 64, 64, 16, 2.0 ** (-10 if dtype == "bf16" else -14)
    P = np.concatenate([_clustered_projection(np.random.default_rng(2 + i), S, dk, x0, 6, 40, 1) for i in range(2)])[None]
    X = np.zeros((1, 1, T, dk))
    X[..., 0], X[..., 1] = x0, 1.0
    gone = [i for hf in range(2) for i in (hf * S + np.flatnonzero(P[0, hf * S:(hf + 1) * S, 1] == 1.0)[::9])]
    s = O.half_scores(P[0], X[0, 0, :1])
    s[:, gone] = -np.inf
    iw, _, ww = O.pkm_select(s[:, :S], s[:, S:], k)
    P[0, gone, 5] = np.nan
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    dP, dX = torch.from_numpy(P).cuda().to(dt), torch.from_numpy(X).cuda().to(dt)
    sdm.device_status()
    got = _address(sdm, sdm.SdmShape.make(1, 1, T, dk, 16, S * S, k, k, dtype), [dP, dP], [dX, dX])
    assert sdm.device_status() == 0
    for idx, w in ((got[0], got[1]), (got[2], got[3])):
        assert np.array_equal(idx[0, 0].cpu().numpy(), np.broadcast_to(iw, (T, k)))
        assert np.all(np.abs(w[0, 0].cpu().numpy() - ww) <= 2e-5 * ww)


# ------------------------------------------------------------------ cuts of a sequence

@pytest.mark.parametrize("dtype,addr,k", [("f32", "projected", 48), ("f32", "projected", 64), ("bf16", "direct", 33)])
def test_wide_lists_do_not_depend_on_how_a_sequence_is_cut(sdm, dtype, addr, k):
    """k > 32 on the FFMA scores: 1024 tokens of 16 heads leave one list per half, 70 and 1 of them
    two, and different passes finish them; slots and weights are the same bits.  Every seventh score is
    tied with its neighbour, so that boundaries also go through the rescoring passes."""
    H, T, S = 16, 1024, 128
    dk = 2 * S if addr == "direct" else 32
    g = torch.Generator(device="cuda").manual_seed(k)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    x = [torch.randn((1, H, T, dk), generator=g, device="cuda") for _ in range(2)]
    P = [torch.randn((H, 2 * S, dk), generator=g, device="cuda") for _ in range(2)]
    for t in (x if addr == "direct" else P):
        dim = 3 if addr == "direct" else 1
        t.index_copy_(dim, torch.arange(1, 2 * S, 7, device="cuda"), t.index_select(dim, torch.arange(0, 2 * S - 1, 7, device="cuda")))
    x, P = [t.to(dt) for t in x], ([None, None] if addr == "direct" else [t.to(dt) for t in P])
    run = lambda a, b: _address(sdm, sdm.SdmShape.make(1, H, b - a, dk, 16, S * S, k, k, dtype, addr), P,
                                [t[:, :, a:b].contiguous() for t in x])
    whole = run(0, T)
    assert sdm.device_status() == 0
    for a, b in ((0, 70), (500, 570), (T - 1, T)):
        for f, p in zip(whole, run(a, b)):
            assert torch.equal(f[:, :, a:b], p), (a, b)


# masked scores: DIRECT addressing takes the scores themselves.  One launch, the warp passes (two chunks per half),
# the thread passes and the band pass per thread; k equal to the half; lists of 64
@pytest.mark.parametrize("dtype,H,T,S,kw,kr", [("f32", 2, 40, 40, 16, 12), ("bf16", 1, 9, 33, 32, 33), ("f32", 1, 4200, 128, 32, 8),
                                               ("bf16", 1, 4200, 48, 20, 16), ("bf16", 2, 8800, 36, 16, 3), ("f32", 1, 40, 128, 48, 33),
                                               ("bf16", 2, 600, 96, 64, 40), ("f32", 1, 300, 40, 40, 36), ("f32", 3, 4200, 16, 16, 1)])
@pytest.mark.parametrize("mask", ["inf", "lowest"])
def test_masked_scores_direct(sdm, dtype, H, T, S, kw, kr, mask):
    """Tokens whose halves keep 1, a few, k - 1, k, k + 1 or all of their scores and hold the mask (-inf, or the type's
    lowest number) elsewhere: the slots of the float64 definition, by (score desc, index asc) also among
    the masked ones, whose weights are 0."""
    rng = np.random.default_rng(S * 7 + kw)
    low = -np.inf if mask == "inf" else float(torch.finfo(torch.bfloat16 if dtype == "bf16" else torch.float32).min)
    kinds = 12                                            # the tokens repeat these
    X = []
    for k in (kr, kw):
        s = O.round_storage(rng.standard_normal((H, kinds, 2 * S)), dtype)
        for i in range(kinds):
            for hf in range(2):
                keep = (1, 3, k - 1, k, k + 1, S)[(i + hf * (i // 6)) % 6]
                drop = rng.permutation(S)[max(1, min(keep, S)):]
                s[:, i, hf * S + drop] = low
        X.append(s)
    shape = sdm.SdmShape.make(1, H, T, 2 * S, 16, S * S, kw, kr, dtype, "direct")
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    x = [torch.from_numpy(s).cuda().to(dt).repeat(1, -(-T // kinds), 1)[None, :, :T].contiguous() for s in X]
    sdm.device_status()
    got = _address(sdm, shape, [None, None], x)
    assert sdm.device_status() == 0
    for (idx, w), s, k in (((got[2], got[3]), X[0], kr), ((got[0], got[1]), X[1], kw)):
        idx, w = idx.cpu().numpy(), w.cpu().numpy()
        for h in range(H):
            with np.errstate(invalid="ignore"):
                iw, _, ww = O.address(None, s[h], S * S, k)
            for i in range(min(kinds, T)):
                assert np.array_equal(idx[0, h, i::kinds], np.broadcast_to(iw[i], idx[0, h, i::kinds].shape)), (k, h, i)
                assert np.all(np.abs(w[0, h, i::kinds] - ww[i]) <= 2e-5 * ww[i]), (k, h, i)


# ------------------------------------------------------------------ several host threads

def _decode_call(sdm, dtype, B, H, dk, S, k):
    st = torch.bfloat16 if dtype == "bf16" else torch.float32
    shape = sdm.SdmShape.make(B, H, 1, dk, 16, S * S, k, k, dtype)
    P = torch.randn((H, 2 * S, dk), device="cuda").to(st)
    x = torch.randn((B, H, 1, dk), device="cuda").to(st)
    out = _lists(B, H, 1, k, k)
    ws = torch.empty(sdm.workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    return lambda s: sdm.address(shape, P, P, x, x, *out, ws, stream=s)


def _head_mix_call(sdm, B):
    shape = sdm.SdmShape.make(B, 1, 1, 16, 64, 100, 3, 3, "bf16")
    z, w = [torch.ones((n, 64), dtype=torch.bfloat16, device="cuda") for n in (B, 32)]
    out = torch.empty((B, 32), dtype=torch.bfloat16, device="cuda")
    return lambda s: sdm.head_mix(shape, 32, z, w, out, stream=s)


def _in_threads(calls, repeat):
    """Each call `repeat` times from a host thread of its own on a stream of its own; the errors."""
    streams = [torch.cuda.Stream() for _ in calls]
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(calls))

    def work(call, stream):
        try:
            start.wait()
            for i in range(repeat):
                call(stream)
                if i % 100 == 99:
                    stream.synchronize()
        except Exception as e:                       # noqa: BLE001 (returned)
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=a) for a in zip(calls, streams)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    return errors


@pytest.mark.parametrize("name", ["small", "large", "wide", "head_mix"])
def test_first_cuda_call_of_a_thread(sdm, name):
    """A host thread whose first CUDA call is one of the tensor-map paths (it has no context yet)."""
    call = {"small": lambda: _decode_call(sdm, "bf16", 1, 1, 64, 40, 32), "large": lambda: _decode_call(sdm, "bf16", 80, 16, 64, 40, 32),
            "wide": lambda: _decode_call(sdm, "bf16", 2, 2, 128, 70, 64), "head_mix": lambda: _head_mix_call(sdm, 40)}[name]()
    assert not _in_threads([call], 1)


def _lists_in(C, T, N, k):
    idx = torch.stack([torch.randperm(N, device="cuda")[:k].sort().values for _ in range(T)]).int()
    return idx.expand(C, T, k).contiguous(), torch.full((C, T, k), 1.0 / k, device="cuda")


def _recurrence_call(sdm, dv, T, k, kind, chunk=0):
    N = 200
    shape = sdm.SdmShape.make(1, 1, T, 16, dv, N, k, k, "bf16")
    (iw, ww), (ir, wr) = _lists_in(1, T, N, k), _lists_in(1, T, N, k)
    f = lambda *s: torch.rand(s, device="cuda").to(torch.bfloat16)
    mem, v, y, al, be = f(1, 1, N, dv), f(1, 1, T, dv), f(1, 1, T, dv), f(1, 1, T), f(1, 1, T)
    if kind == "chunkwise":
        return lambda s: sdm.recur_chunkwise(shape, iw, ww, ir, wr, v, al, be, mem, y, chunk, stream=s)
    if kind == "recurrence":
        ws = torch.empty(sdm.recur_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
        return lambda s: sdm.recur(shape, iw, ww, ir, wr, v, al, be, mem, y, ws, stream=s)
    undo = torch.zeros(sdm.undo_log_bytes(shape), dtype=torch.uint8, device="cuda")
    e = lambda *s: torch.zeros((1, 1, *s), dtype=torch.float32, device="cuda")
    grads = (e(T, dv), e(T), e(T), e(T, k), e(T, k), e(N, dv))
    return lambda s: sdm.recur_backward(shape, iw, ww, ir, wr, v, al, be, mem, undo, y, *grads, stream=s)


def _gates_call(sdm, d):
    shape = sdm.SdmShape.make(1, 4, 2, 16, 16, 100, 3, 3, "f32")
    f = lambda *s: torch.rand(s, device="cuda")
    x, wa, wb, b_dt, A, al, be = f(1, 2, d), f(4, d), f(4, d), f(4), f(4), f(1, 4, 2), f(1, 4, 2)
    return lambda s: sdm.gates(shape, d, x, wa, wb, b_dt, A, al, be, stream=s)


PAIRS = {
    "small_ffma": lambda sdm: (_decode_call(sdm, "f32", 1, 1, 16, 40, 32), _decode_call(sdm, "f32", 1, 1, 64, 1000, 32)),
    "small_tensor": lambda sdm: (_decode_call(sdm, "bf16", 1, 1, 64, 40, 32), _decode_call(sdm, "bf16", 2, 1, 128, 1000, 32)),
    "large_tensor": lambda sdm: (_decode_call(sdm, "bf16", 80, 16, 64, 40, 32), _decode_call(sdm, "bf16", 80, 16, 128, 40, 32)),
    "large_ffma": lambda sdm: (_decode_call(sdm, "f32", 80, 64, 8, 40, 32), _decode_call(sdm, "f32", 80, 64, 256, 40, 32)),
    "backward": lambda sdm: (_recurrence_call(sdm, 32, 8, 32, "backward"), _recurrence_call(sdm, 128, 8, 32, "backward")),
    "chunkwise": lambda sdm: (_recurrence_call(sdm, 32, 8, 4, "chunkwise", 4), _recurrence_call(sdm, 32, 32, 60, "chunkwise", 32)),
    "hazard": lambda sdm: (_recurrence_call(sdm, 32, 40, 20, "recurrence"), _recurrence_call(sdm, 32, 40, 64, "recurrence")),
    "gates": lambda sdm: (_gates_call(sdm, 2000), _gates_call(sdm, 6000)),
}


@pytest.mark.parametrize("name", sorted(PAIRS))
def test_calls_of_different_sizes_from_two_threads(sdm, name):
    """Two host threads, a stream each, call one kernel with shared memory of different sizes: no
    launch fails because the other thread's call came between its set-up and its launch."""
    assert not _in_threads(PAIRS[name](sdm), 3000)
    sdm.device_status()


# ------------------------------------------------------------------ alignment

@pytest.mark.parametrize("B,H,T,dk,S,k,which", [(1, 2, 33, 64, 100, 40, "P"), (1, 2, 33, 128, 70, 64, "x"),
                                                (2, 1, 5, 64, 600, 33, "Px"), (1, 16, 1100, 64, 64, 64, "Px")])
def test_wide_lists_take_element_aligned_operands(sdm, B, H, T, dk, S, k, which):
    """bf16, k > 32, P or the tokens aligned to their elements only: the slots of the definition."""
    rng = np.random.default_rng(S)
    P = [O.round_storage(rng.standard_normal((H, 2 * S, dk)), "bf16") for _ in range(2)]
    x = [O.round_storage(rng.standard_normal((B, H, T, dk)) / np.sqrt(dk), "bf16") for _ in range(2)]
    shape = sdm.SdmShape.make(B, H, T, dk, 16, S * S, k, k, "bf16")
    dP, dx = [_stored(p, "bf16") for p in P], [_stored(v, "bf16") for v in x]
    got = _address(sdm, shape, [_shifted(p) for p in dP] if "P" in which else dP,
                   [_shifted(v) for v in dx] if "x" in which else dx)
    assert sdm.device_status() == 0
    for side, (idx, w) in enumerate(((got[2], got[3]), (got[0], got[1]))):
        for b in range(B):
            for h in range(0, H, 7):
                iw, _, ww = O.address(P[side][h], x[side][b, h], S * S, k)
                assert np.array_equal(idx[b, h].cpu().numpy(), iw), (side, b, h)
                assert np.all(np.abs(w[b, h].cpu().numpy() - ww) <= 2e-5 * ww), (side, b, h)


# ------------------------------------------------------------------ what an error leaves behind

def test_refused_forward_m0_leaves_no_broadcast_behind(sdm):
    """A forward_m0 that fails at its addressing (operands the tensor maps refuse) after the broadcast of
    M0 went to the library's stream: what the caller enqueues next on its own stream comes after it."""
    B, H, S, d = 8, 16, 256, 128
    shape = sdm.SdmShape.make(B, H, 1, 64, d, S * S, 8, 8, "bf16")
    bf = dict(dtype=torch.bfloat16, device="cuda")
    M0, mem = torch.ones((H, S * S, d), **bf), torch.empty((B, H, S * S, d), **bf)
    P = _shifted(torch.ones((H, 2 * S, 64), **bf))
    q = torch.ones((B, H, 1, 64), **bf)
    v, y, g = torch.ones((B, H, 1, d), **bf), torch.empty((B, H, 1, d), **bf), torch.ones((B, H, 1), **bf)
    ws = torch.empty(sdm.workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    with pytest.raises(sdm.SdmError):
        sdm.forward_m0(shape, M0, P, P, q, q, v, g, g, mem, y, ws)
    mem[B - 1].fill_(3.0)
    torch.cuda.synchronize()
    assert bool((mem[B - 1] == 3.0).all())


FIRST_CALLS = """
import sys, threading, torch
sys.path.insert(0, {root!r})
import paper_2607_07386_gb300 as sdm
sdm.lib()
bf = dict(dtype=torch.bfloat16, device="cuda")
def args():
    shape = sdm.SdmShape.make(1, 1, 1, 64, 16, 256, 4, 4, "bf16")
    M0, mem = torch.ones((1, 256, 16), **bf), torch.zeros((1, 1, 256, 16), **bf)
    P, q, v = torch.randn((1, 32, 64), device="cuda").bfloat16(), torch.ones((1, 1, 1, 64), **bf), torch.ones((1, 1, 1, 16), **bf)
    g = torch.full((1, 1, 1), 0.5, **bf)
    ws = torch.empty(sdm.workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    return shape, M0, P, P, q, q, v, g, g, mem, torch.empty_like(v), ws
calls = [(args(), torch.cuda.Stream()) for _ in range(12)]
torch.cuda.synchronize()
start, errors = threading.Barrier(len(calls)), []
def work(a, s):
    try:
        start.wait()
        sdm.forward_m0(*a, stream=s)
    except Exception as e:
        errors.append(repr(e))
ts = [threading.Thread(target=work, args=c) for c in calls]
for t in ts: t.start()
for t in ts: t.join()
torch.cuda.synchronize()
assert not errors, errors
for a, _ in calls:
    assert bool((a[9] != 0).all())
assert sdm.device_status() == 0
"""


def test_first_forward_m0_calls_from_several_threads(sdm):
    """The library's side stream is made by the first call on a device: several threads may make it."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", FIRST_CALLS.format(root=root)], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]


# ------------------------------------------------------------------ rescans of wide lists

@pytest.mark.parametrize("dtype,S,k,T,n,dup", [("bf16", 256, 64, 20, 20, 1), ("bf16", 600, 40, 7, 20, 4), ("f32", 96, 64, 300, 20, 1),
                                               ("f32", 128, 33, 2100, 60, 1)])
def test_rescan_of_a_half_ranks_the_band_alone(sdm, dtype, S, k, T, n, dup):
    """k > 32, one list per half, a band of n near-equal scores (each dup times) past the kept list: the rescan of the half finds the
    exact slots among the columns that reach the band and leaves no half to the serial resolver."""
    from tests.test_gpu_parity import _clustered_projection
    dk, x0 = 64, 2.0 ** (-10 if dtype == "bf16" else -14)
    rng = np.random.default_rng(S)
    P = np.concatenate([_clustered_projection(rng, S, dk, x0, k - 8, n, dup) for _ in range(2)])[None]
    X = np.zeros((1, 1, T, dk))
    X[..., 0], X[..., 1] = x0, 1.0
    H = 16 if dtype == "f32" else 1                       # (enough token tiles for one chunk per half)
    dP, dX = _stored(np.repeat(P, H, 0), dtype), _stored(np.repeat(X, H, 1), dtype)
    iw, _, ww = O.address(P[0], X[0, 0, :1], S * S, k)
    sdm.device_stats()
    got = _address(sdm, sdm.SdmShape.make(1, H, T, dk, 16, S * S, k, k, dtype), [dP, dP], [dX, dX])
    stats = sdm.device_stats()
    assert sdm.device_status() == 0
    assert stats["half_full"] > 0 and stats["serial"] == stats["comb_full"], stats
    for idx, w in ((got[0], got[1]), (got[2], got[3])):
        assert np.array_equal(idx.cpu().numpy(), np.broadcast_to(iw, (1, H, T, k)))
        assert np.all(np.abs(w.cpu().numpy() - ww) <= 2e-5 * ww)


# ------------------------------------------------------------------ the broadcast beside the addressing

def _forward_m0_call(sdm, B, T, N, seed=1):
    H, d, k, S = 16, 128, 32, int(N ** 0.5)
    g = torch.Generator(device="cuda").manual_seed(seed)
    rn = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    shape = sdm.SdmShape.make(B, H, T, d, d, N, k, k, "bf16")
    args = [shape, rn(H, N, d), rn(H, 2 * S, d), rn(H, 2 * S, d), rn(B, H, T, d), rn(B, H, T, d), rn(B, H, T, d),
            torch.sigmoid(rn(B, H, T)), torch.sigmoid(rn(B, H, T)), torch.empty((B, H, N, d), dtype=torch.bfloat16, device="cuda"),
            torch.empty((B, H, T, d), dtype=torch.bfloat16, device="cuda"),
            torch.empty(sdm.workspace_bytes(shape), dtype=torch.uint8, device="cuda")]
    return args


@pytest.mark.parametrize("T", [4, 16])
def test_queued_forward_m0_calls_take_no_longer_than_single_ones(sdm, T):
    """Calls queued one behind another against the same calls with a wait after each, where the addressing leaves
    SMs empty: at most 1.5 times as long (the broadcast's CTAs on a few SMs took 2 to 3.5 times)."""
    import time
    args = _forward_m0_call(sdm, 8, T, 1 << 16)

    def per_call(wait):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(20):
            sdm.forward_m0(*args)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return time.perf_counter() - t0

    per_call(True)
    single, queued = [min(per_call(w) for _ in range(3)) for w in (True, False)]
    assert queued <= 1.5 * single, (queued, single)


@pytest.mark.parametrize("T", [1, 40])
def test_forward_m0_in_a_graph(sdm, T):
    """Captured and replayed: the same bits as the call itself."""
    args = _forward_m0_call(sdm, 2, T, 4096)
    sdm.forward_m0(*args)
    torch.cuda.synchronize()
    want = args[9].clone(), args[10].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sdm.forward_m0(*args)
    for _ in range(2):
        args[9].zero_()
        args[10].zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(args[9], want[0]) and torch.equal(args[10], want[1])
    assert sdm.device_status() == 0


def test_tokens_of_zeros_with_wide_lists(sdm):
    """Padding tokens (all scores equal) at k = 64: the first slots in order, equal weights, and no serial walk
    (25 ms for 2,400 of them; a lane deciding each by itself took 73)."""
    import time
    H, T, S, dk, k = 8, 300, 256, 128, 64
    P = torch.randn((H, 2 * S, dk), device="cuda").to(torch.bfloat16)
    x = torch.zeros((1, H, T, dk), dtype=torch.bfloat16, device="cuda")
    shape = sdm.SdmShape.make(1, H, T, dk, 16, S * S, k, k, "bf16")
    best = 1.0
    for _ in range(3):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        got = _address(sdm, shape, [P, P], [x, x])
        best = min(best, time.perf_counter() - t0)
    assert sdm.device_status() == 0
    want = torch.arange(k, dtype=torch.int32, device="cuda")
    for idx, w in ((got[0], got[1]), (got[2], got[3])):
        assert bool((idx == want).all()) and bool((w == 1.0 / k).all())
    assert best <= 0.025, best


# ------------------------------------------------------------------ the score kernel of large problems
# (up to 2048 token-sides with k <= 32 take the one-launch kernel, which has no retries to count)

@pytest.mark.parametrize("B,T,S,k", [(1, 130, 128, 8), (5, 40, 128, 8), (3, 50, 256, 32), (2, 66, 1100, 16)])
def test_ragged_score_tiles_of_large_problems(sdm, B, T, S, k):
    """Tiles of the tensor-core score kernel with rows past the batch: the lists of the same tokens in full tiles, and
    no retry; the same shape with equal rows of P retries, which shows that it takes this kernel."""
    H, dk, TT = 16, 64, 256
    g = torch.Generator(device="cuda").manual_seed(5)
    rn = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    P, x = [rn(H, 2 * S, dk) for _ in range(2)], [rn(B, H, TT, dk) for _ in range(2)]
    run = lambda P_, T_: _address(sdm, sdm.SdmShape.make(B, H, T_, dk, 16, S * S, k, k, "bf16"), P_,
                                  [t[:, :, :T_].contiguous() for t in x])
    full = run(P, TT)
    sdm.device_stats()
    part = run(P, T)
    assert sdm.device_stats()["select_retry"] == 0
    for f, p in zip(full, part):
        assert torch.equal(f[:, :, :T], p)
    run([p[:, :1].expand_as(p).contiguous() for p in P], T)
    assert sdm.device_stats()["select_retry"] > 0
    assert sdm.device_status() == 0


# the inputs of test_selection_of_near_ties and wider ones, past the range of the one-launch kernel; `retry`: more
# scores at or above the cluster than the survivor buffer holds (40, 56, 72 and 121 for k up to 8, 16, 32 and 64)
@pytest.mark.parametrize("S,k,T,clusters,retry", [(96, 32, 1100, (29, 5, 1), False), (300, 20, 1100, (0, 300, 1), True),
                                                  (300, 12, 1100, (0, 1, 300), True), (700, 32, 1050, (10, 200, 1), True),
                                                  (1100, 8, 1030, (3, 90, 1), True), (256, 64, 33, (20, 200, 1), True),
                                                  (600, 40, 20, (0, 2, 100), True)])
def test_near_ties_and_overflows_of_large_problems(sdm, S, k, T, clusters, retry):
    """Bands, exact ties, survivor buffers that overflow (with a new threshold, and to the exact scan), with one chunk
    of columns and with several: the slots of the float64 definition."""
    from tests.test_gpu_parity import _clustered_projection
    n_hi, cluster, dup = clusters
    dk, x0 = 64, 2.0 ** -10
    rng = np.random.default_rng(23)
    P = O.round_storage(np.concatenate([_clustered_projection(rng, S, dk, x0, n_hi, cluster, dup) for _ in range(2)]), "bf16")
    X = np.zeros((1, 1, T, dk))
    X[..., 0], X[..., 1] = x0, 1.0
    iw, _, ww = O.address(P, X[0, 0, :1], S * S, k)
    dP, dX = _stored(P[None], "bf16"), _stored(X, "bf16")
    sdm.device_stats()
    got = _address(sdm, sdm.SdmShape.make(1, 1, T, dk, 16, S * S, k, k, "bf16"), [dP, dP], [dX, dX])
    stats = sdm.device_stats()
    assert sdm.device_status() == 0
    assert (stats["select_retry"] > 0) == retry, stats
    for idx, w in ((got[0], got[1]), (got[2], got[3])):
        assert np.array_equal(idx[0, 0].cpu().numpy(), np.broadcast_to(iw, (T, k)))
        assert np.all(np.abs(w[0, 0].cpu().numpy() - ww) <= 2e-5 * ww)


@pytest.mark.parametrize("dtype,B,H,dv,k", [("bf16", 16, 16, 128, 48), ("bf16", 4, 16, 512, 64), ("f32", 8, 16, 128, 33)])
def test_wide_lists_decode_as_in_a_longer_call(sdm, dtype, B, H, dv, k):
    """k > 32 on many chains: the last token alone (the one-token kernel) gives the bits of the call that holds it."""
    N, T = 200, 3
    g = torch.Generator(device="cuda").manual_seed(k)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    rn = lambda *s: torch.randn(s, generator=g, device="cuda").to(dt)
    lists = lambda: torch.rand((B, H, T, N), generator=g, device="cuda").topk(k, dim=-1).indices.sort(dim=-1).values.int()
    w = lambda: torch.softmax(torch.randn((B, H, T, k), generator=g, device="cuda"), -1)
    L = [lists(), w(), lists(), w(), rn(B, H, T, dv), torch.sigmoid(rn(B, H, T)), torch.sigmoid(rn(B, H, T))]
    M0 = rn(B, H, N, dv)

    def run(mem, a, b):
        shape = sdm.SdmShape.make(B, H, b - a, 16, dv, N, k, k, dtype)
        sl = [t[:, :, a:b].contiguous() for t in L]
        y = torch.empty_like(sl[4])
        sdm.recur(shape, *sl, mem, y, torch.empty(sdm.recur_workspace_bytes(shape), dtype=torch.uint8, device="cuda"))
        return y

    whole, cut = M0.clone(), M0.clone()
    y = run(whole, 0, T)
    parts = torch.cat([run(cut, 0, T - 1), run(cut, T - 1, T)], 2)
    assert sdm.device_status() == 0
    assert torch.equal(whole, cut) and torch.equal(y, parts)
