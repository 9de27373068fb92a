"""Kernel edges: sizes at which a tile, slice, vector or window of the kernels is partly empty.

Bars follow tests/test_gpu_parity.py: selected slots bit-exact; gradients of the backward within
1e-4 (fp32) or 5e-3 (bf16) relative Frobenius of the oracle's; the recurrence within 1e-5 (f32) or
2e-3 (bf16); quantised codes and scales bit-exact.
"""
import numpy as np
import pytest

from oracle import sdm_oracle as O
from oracle.reference_run import rel_fro

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


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


# (B, H, dtype, d_v, N, k_write, k_read, T): sixteen warps (few chains), eight and four; lists of 64
# slots (rows asked for one token ahead); tokens fewer than, equal to and one more than the warps or the
# window; so few slots that almost every token waits for, rereads and overwrites rows of the last ones
@pytest.mark.parametrize("B,H,dtype,dv,N,kw,kr,T,w", [
    (1, 2, "bf16", 128, 96, 32, 32, 200, 16), (1, 3, "f32", 64, 40, 8, 5, 49, 16), (1, 2, "bf16", 64, 4096, 64, 64, 97, 16),
    (1, 2, "bf16", 128, 128, 64, 33, 41, 16), (1, 1, "bf16", 8, 64, 16, 16, 65, 16), (1, 2, "bf16", 64, 50, 3, 7, 16, 16),
    (1, 2, "bf16", 64, 50, 3, 7, 17, 16), (3, 8, "bf16", 128, 64, 16, 16, 90, 8), (2, 16, "bf16", 128, 96, 64, 64, 61, 8),
    (4, 16, "f32", 64, 80, 40, 40, 33, 4), (8, 16, "bf16", 128, 80, 48, 64, 35, 4), (8, 16, "bf16", 128, 40, 32, 9, 29, 4)])
def test_recurrence_warps_depth_and_window(sdm, B, H, dtype, dv, N, kw, kr, T, w):
    rng = np.random.default_rng(N * 31 + T)
    shape = sdm.SdmShape.make(B, H, T, 16, dv, N, kw, kr, dtype)
    assert sdm.recur_plan(shape)["w"] == w
    C = B * H
    lists = lambda k: np.stack([np.sort(rng.choice(N, k, replace=False)) for _ in range(C * T)]).reshape(C, T, k)
    weights = lambda k: rng.dirichlet(np.ones(k), (C, T)).astype(np.float32)
    iw, ir, ww, wr = lists(kw), lists(kr), weights(kw), weights(kr)
    a = O.round_storage(1 / (1 + np.exp(-rng.standard_normal((C, T)) - 1)), dtype)
    b = O.round_storage(1 / (1 + np.exp(-rng.standard_normal((C, T)))), dtype)
    V = O.round_storage(rng.standard_normal((C, T, dv)), dtype)
    M0 = O.round_storage(rng.standard_normal((C, N, dv)) * 0.5, dtype)
    i32 = lambda x: _cuda(x.astype(np.int32)).view(B, H, T, -1)
    mem = _stored(M0, dtype).cuda().view(B, H, N, dv)
    y = torch.empty((B, H, T, dv), dtype=mem.dtype, device="cuda")
    ws = torch.empty(sdm.recur_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    sdm.device_status()
    sdm.recur(shape, i32(iw), _cuda(ww).view(B, H, T, kw), i32(ir), _cuda(wr).view(B, H, T, kr),
              _stored(V, dtype).cuda().view(B, H, T, dv), _stored(a, dtype).cuda().view(B, H, T),
              _stored(b, dtype).cuda().view(B, H, T), mem, y, ws)
    torch.cuda.synchronize()
    assert sdm.device_status() == 0
    yg, mg = y.double().cpu().numpy().reshape(C, T, dv), mem.double().cpu().numpy().reshape(C, N, dv)
    tol = 1e-5 if dtype == "f32" else 2e-3
    for c in sorted({0, C // 2, C - 1}):
        Mo = M0[c].copy()
        _, yo = O.recur(Mo, iw[c], ww[c].astype(np.float64), ir[c], wr[c].astype(np.float64), V[c], a[c], b[c], dtype)
        assert rel_fro(yg[c], yo) <= tol and rel_fro(mg[c], Mo) <= tol, c


def _shifted(x):
    """The same values in a buffer that starts one element past an allocation (element-aligned only)."""
    big = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)
    out = big[1:].view(x.shape)
    out.copy_(x)
    return out


def _sorted_lists(rng, N, k, *lead):
    n = int(np.prod(lead))
    return np.stack([np.sort(rng.choice(N, k, replace=False)) for _ in range(n)]).reshape(*lead, k)


# ------------------------------------------------------------------ addressing: tiles with rows past the batch

@pytest.mark.parametrize("B,T", [(1, 1), (3, 1), (2, 130), (5, 40)])
def test_score_tile_rows_past_the_batch_select_nothing(sdm, B, T):
    """A tile of the tensor-core score kernel with rows past the batch: the lists equal those of
    the same tokens in full tiles, and no row runs the overflow retries (rows past the batch hold
    equal scores, which would)."""
    H, dk, S, k = 2, 64, 128, 8
    g = torch.Generator(device="cuda").manual_seed(5)
    rn = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    P = [rn(H, 2 * S, dk) for _ in range(2)]
    # the same tokens, padded to T' = 256 per sequence: every tile is full
    TT = 256
    x = [rn(B, H, TT, dk) for _ in range(2)]

    def lists(T_, xs):
        sh = sdm.SdmShape.make(B, H, T_, dk, 16, S * S, k, k, "bf16")
        o = [torch.empty((B, H, T_, k), dtype=t, device="cuda") for t in (torch.int32, torch.float32) * 2]
        ws = torch.empty(sdm.workspace_bytes(sh), dtype=torch.uint8, device="cuda")
        sdm.address(sh, P[0], P[1], xs[0], xs[1], *o, ws)
        return o

    full = lists(TT, x)
    sdm.device_stats()
    part = lists(T, [t[:, :, :T].contiguous() for t in x])
    stats = sdm.device_stats()
    assert sdm.device_status() == 0
    assert stats["select_retry"] == 0, stats
    for f, p in zip(full, part):
        assert torch.equal(f[:, :, :T], p)


def _address(sdm, dtype, B, H, T, dk, S, kw, kr, P, x):
    shape = sdm.SdmShape.make(B, H, T, dk, 16, S * S, kw, kr, dtype)
    o = [torch.empty((B, H, T, k), dtype=t, device="cuda") for k in (kw, kr) for t in (torch.int32, torch.float32)]
    ws = torch.empty(sdm.workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    sdm.address(shape, _stored(P[0], dtype), _stored(P[1], dtype), _stored(x[0], dtype), _stored(x[1], dtype), *o, ws)
    torch.cuda.synchronize()
    assert sdm.device_status() == 0
    return [t.cpu().numpy() for t in o]


def _check_address(got, P, x, S, kw, kr):
    """Slots equal to the float64 definition's, weights within 2e-5 relative (fp32 softmax)."""
    for side, (idx, w, k) in enumerate(((got[2], got[3], kr), (got[0], got[1], kw))):
        for b in range(x[side].shape[0]):
            for h in range(P[side].shape[0]):
                iw, _, ww = O.address(P[side][h], x[side][b, h], S * S, k)
                assert np.array_equal(idx[b, h], iw), (side, b, h)
                assert np.all(np.abs(w[b, h] - ww) <= 2e-5 * ww), (side, b, h)


@pytest.mark.parametrize("S,kw,kr,dk,B,T", [
    (16, 8, 5, 64, 2, 9), (33, 16, 16, 128, 1, 140), (40, 32, 31, 64, 1, 33), (64, 64, 33, 64, 1, 17),
    (69, 64, 64, 128, 2, 40), (100, 3, 20, 64, 3, 50), (130, 8, 8, 128, 1, 300), (256, 17, 32, 128, 1, 129),
    (257, 32, 9, 64, 2, 64), (300, 50, 12, 128, 1, 70), (512, 32, 32, 128, 1, 200), (513, 32, 16, 64, 1, 130),
    (1100, 64, 32, 128, 1, 60), (1030, 8, 20, 128, 2, 20)])
def test_selection_sizes(sdm, S, kw, kr, dk, B, T):
    """Tensor-core scores and the thread passes at list lengths 12 to 68, halves of one partial block to
    three chunks, odd slot counts, tiles with rows past the batch."""
    rng = np.random.default_rng(S * 100 + kw)
    H = 2
    P = [O.round_storage(rng.standard_normal((H, 2 * S, dk)), "bf16") for _ in range(2)]
    x = [O.round_storage(rng.standard_normal((B, H, T, dk)) / np.sqrt(dk), "bf16") for _ in range(2)]
    _check_address(_address(sdm, "bf16", B, H, T, dk, S, kw, kr, P, x), P, x, S, kw, kr)


@pytest.mark.parametrize("S,k,T,clusters", [(128, 64, 12, (20, 90, 1)), (128, 64, 12, (61, 6, 2)), (96, 32, 300, (29, 5, 1)),
                                            (700, 32, 5, (10, 200, 1)), (300, 20, 3, (0, 300, 1)), (300, 12, 3, (0, 1, 300))])
def test_selection_of_near_ties(sdm, S, k, T, clusters):
    """Scores closer than the fp32 error bound around the boundary (n_hi rows above, a cluster of distinct
    near-equal rows, each repeated): bands, whole-half rescans, exact ties, and more equal scores
    than the survivor buffer holds."""
    from tests.test_gpu_parity import _clustered_projection
    rng = np.random.default_rng(23)
    n_hi, cluster, dup = clusters
    dk, x0 = 64, 2.0 ** -10
    P = [np.stack([np.concatenate([_clustered_projection(rng, S, dk, x0, n_hi, cluster, dup) for _ in range(2)])])
         for _ in range(2)]
    P = [O.round_storage(p, "bf16") for p in P]
    X = np.zeros((1, 1, T, dk))
    X[..., 0], X[..., 1] = x0, 1.0
    _check_address(_address(sdm, "bf16", 1, 1, T, dk, S, k, k, P, [X, X]), P, [X, X], S, k, k)


# ------------------------------------------------------------------ backward

BACKWARD = {
    # one token, one slot; slices = 1 with dense conflicts; three slices, element-aligned buffers;
    # two phases of eight slices; long enough for several conflict windows; vectors of four slots
    "one_token": ("f32", 1, 1, 1, 8, 1, 1, 32, False),
    "one_slice_dense": ("bf16", 2, 1, 33, 64, 9, 32, 32, False),
    "three_slices_unaligned": ("bf16", 1, 2, 49, 300, 17, 3, 96, True),
    "eight_slices": ("bf16", 1, 1, 65, 120, 32, 32, 256, False),
    "f32_eight_slices": ("f32", 1, 1, 40, 90, 32, 5, 256, False),
    "f32_unaligned": ("f32", 1, 2, 100, 1000, 4, 8, 128, True),
}


@pytest.mark.parametrize("name", sorted(BACKWARD))
def test_backward_edges(sdm, name):
    dtype, B, H, T, N, kw, kr, dv, shift = BACKWARD[name]
    rng = np.random.default_rng(17)
    M0 = O.round_storage(rng.standard_normal((B * H, N, dv)) * 0.3, dtype)
    iw, ir = _sorted_lists(rng, N, kw, B, H, T), _sorted_lists(rng, N, kr, B, H, T)
    ww = rng.dirichlet(np.ones(kw), B * H * T).astype(np.float32).reshape(B, H, T, kw)
    wr = rng.dirichlet(np.ones(kr), B * H * T).astype(np.float32).reshape(B, H, T, kr)
    a = O.round_storage(1 / (1 + np.exp(-rng.standard_normal((B, H, T)) - 2)), dtype)
    b = O.round_storage(1 / (1 + np.exp(-rng.standard_normal((B, H, T)))), dtype)
    V = O.round_storage(rng.standard_normal((B, H, T, dv)), dtype)
    dY = O.round_storage(rng.standard_normal((B, H, T, dv)), dtype)
    shape = sdm.SdmShape.make(B, H, T, 32, dv, N, kw, kr, dtype)
    L = [_cuda(iw.astype(np.int32)), _cuda(ww), _cuda(ir.astype(np.int32)), _cuda(wr), _stored(V, dtype),
         _stored(a, dtype), _stored(b, dtype)]
    mem = _stored(M0.reshape(B, H, N, dv), dtype)
    y = torch.empty((B, H, T, dv), dtype=mem.dtype, device="cuda")
    undo = torch.empty(sdm.undo_log_bytes(shape), dtype=torch.uint8, device="cuda")
    ws = torch.empty(sdm.recur_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    sdm.recur_undo(shape, *L, mem, y, undo, ws)
    dy = _stored(dY, dtype)
    g = {n: torch.full((B, H, *s), 7.0, dtype=torch.float32, device="cuda")
         for n, s in (("dv", (T, dv)), ("dalpha", (T,)), ("dbeta", (T,)), ("dw_w", (T, kw)), ("dw_r", (T, kr)))}
    g["dM0"] = torch.zeros((B, H, N, dv), dtype=torch.float32, device="cuda")
    if shift:
        L[4], dy = _shifted(L[4]), _shifted(dy)
        g = {n: _shifted(t) for n, t in g.items()}
    sdm.recur_backward(shape, *L, mem, undo, dy, *(g[n] for n in ("dv", "dalpha", "dbeta", "dw_w", "dw_r", "dM0")))
    torch.cuda.synchronize()
    assert sdm.device_status() == 0
    assert torch.equal(mem, _stored(M0.reshape(B, H, N, dv), dtype))
    tol = 1e-4 if dtype == "f32" else 5e-3
    for c in range(B * H):
        bb, hh = divmod(c, H)
        Mo = M0[c].copy()
        args = (iw[bb, hh], ww[bb, hh].astype(np.float64), ir[bb, hh], wr[bb, hh].astype(np.float64), V[bb, hh],
                a[bb, hh], b[bb, hh])
        _, und = O.recur_forward_undo(Mo, *args, dtype)
        ref = O.recur_backward(Mo, und, *args, dY[bb, hh])
        for n, got in g.items():
            e = rel_fro(got[bb, hh].cpu().numpy().astype(np.float64), ref[n])
            assert e <= tol, (c, n, e)


# ------------------------------------------------------------------ chunkwise form

CHUNKWISE = {
    # rows of 1, 2, 3 (padded d-range), 16 and 32 pieces; more chains than one d-range needs; lists longer
    # than a warp; every slot shared (dense systems); a gate of exactly 0; a last chunk of one token
    "one_piece": ("bf16", 1, 1, 5, 8, 3, 2, 8, 4),
    "three_pieces_dense": ("bf16", 2, 1, 33, 40, 33, 40, 24, 32),
    "dense_f32": ("f32", 1, 2, 50, 12, 7, 9, 64, 7),
    "wide_rows": ("f32", 1, 1, 40, 500, 64, 64, 256, 32),
    "split_rows": ("bf16", 3, 2, 65, 600, 32, 17, 128, 16),
    "whole_rows": ("bf16", 8, 16, 18, 90, 5, 32, 128, 8),
    "token_chunks": ("f32", 1, 1, 9, 30, 4, 4, 8, 1),
}


@pytest.mark.parametrize("name", sorted(CHUNKWISE))
def test_chunkwise_edges(sdm, name):
    """Against the chunkwise oracle with the same chunk size: 1e-4 (fp32) and 2e-3 (bf16) relative
    Frobenius, the bars of the other sizes; rows nobody wrote bit-identical."""
    dtype, B, H, T, N, kw, kr, dv, C = CHUNKWISE[name]
    rng = np.random.default_rng(29)
    M0 = O.round_storage(rng.standard_normal((B * H, N, dv)) * 0.3, dtype)
    iw, ir = _sorted_lists(rng, N, kw, B, H, T), _sorted_lists(rng, N, kr, B, H, T)
    ww = rng.dirichlet(np.ones(kw), B * H * T).astype(np.float32).reshape(B, H, T, kw)
    wr = rng.dirichlet(np.ones(kr), B * H * T).astype(np.float32).reshape(B, H, T, kr)
    a = O.round_storage(1 / (1 + np.exp(-rng.standard_normal((B, H, T)) - 2)), dtype)
    a[0, 0, T // 2] = 0.0
    b = O.round_storage(1 / (1 + np.exp(-rng.standard_normal((B, H, T)))), dtype)
    V = O.round_storage(rng.standard_normal((B, H, T, dv)), dtype)
    shape = sdm.SdmShape.make(B, H, T, 32, dv, N, kw, kr, dtype)
    mem = _stored(M0.reshape(B, H, N, dv), dtype)
    y = torch.empty((B, H, T, dv), dtype=mem.dtype, device="cuda")
    sdm.recur_chunkwise(shape, _cuda(iw.astype(np.int32)), _cuda(ww), _cuda(ir.astype(np.int32)), _cuda(wr),
                        _stored(V, dtype), _stored(a, dtype), _stored(b, dtype), mem, y, C)
    torch.cuda.synchronize()
    assert sdm.device_status() == 0
    tol = 1e-4 if dtype == "f32" else 2e-3
    gy, gm = y.double().cpu().numpy(), mem.double().cpu().numpy()
    for c in range(0, B * H, 1 if B * H < 16 else 31):
        bb, hh = divmod(c, H)
        Mo = M0[c].copy()
        _, yo = O.recur_chunkwise(Mo, iw[bb, hh], ww[bb, hh].astype(np.float64), ir[bb, hh],
                                  wr[bb, hh].astype(np.float64), V[bb, hh], np.maximum(a[bb, hh], np.exp(-80.0)),
                                  b[bb, hh], C, dtype)
        assert rel_fro(gy[bb, hh], yo) <= tol, (c, rel_fro(gy[bb, hh], yo))
        assert rel_fro(gm[bb, hh], Mo) <= tol, (c, rel_fro(gm[bb, hh], Mo))
        untouched = np.setdiff1d(np.arange(N), iw[bb, hh].ravel())
        assert np.array_equal(gm[bb, hh][untouched], M0[c][untouched])


# ------------------------------------------------------------------ quantised snapshots

@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("kind", ["fp8", "int4"])
@pytest.mark.parametrize("dv", [32, 96, 160, 224, 256])
def test_undo_quantize_row_widths(sdm, kind, dtype, dv):
    """Codes and scales bit-exact at row widths of 1, 2, 3, 5 and 7 vectors per lane, with a row count
    that leaves the last warp partly empty, rows at the ends of the float range and exact ties."""
    from tests.test_gpu_parity import _decode_codes, _host_undo_log
    rows = 1 * 1 * 131 * 3
    rng = np.random.default_rng(3)
    log = _host_undo_log(rng, rows, dv, dtype)
    log[3] *= 2.0 ** -120
    log[4] = np.sign(log[4]) * np.minimum(np.abs(log[4]), 1.5) * 2.0 ** 126
    log[5] = np.arange(dv) % 15 - 7 + 0.5 * (np.arange(dv) % 2)     # ties of the int4 grid ...
    log[5, 0] = 7.0                                                # ... at scale 1
    log = O.round_storage(log, dtype)
    shape = sdm.SdmShape.make(1, 1, 131, 32, dv, 1000, 3, 3, dtype)
    codes = torch.empty(sdm.undo_code_bytes(shape, kind), dtype=torch.uint8, device="cuda")
    scales = torch.empty(rows, dtype=torch.float32, device="cuda")
    sdm.undo_quantize(shape, _stored(log, dtype), kind, codes, scales)
    torch.cuda.synchronize()
    q_ref, s_ref = O.undo_codes(log, kind)
    assert np.array_equal(scales.cpu().numpy(), s_ref)
    assert np.array_equal(_decode_codes(codes.cpu().numpy(), kind, rows, dv), q_ref)


@pytest.mark.parametrize("kind", ["fp8", "int4"])
def test_undo_quantize_passes_nan_over(sdm, kind):
    """A NaN entry leaves its row's scale and the other codes alone; its own code is e4m3's NaN or 0."""
    rows, dv = 9, 64
    log = O.round_storage(np.random.default_rng(4).standard_normal((rows, dv)), "bf16")
    shape = sdm.SdmShape.make(1, 1, 3, 32, dv, 1000, 3, 3, "bf16")
    out = []
    for nan in (False, True):
        x = log.copy()
        x[2, 7] = x[5, 60] = np.nan if nan else 0.0
        t = torch.from_numpy(x).to("cuda", torch.bfloat16)
        codes = torch.zeros(sdm.undo_code_bytes(shape, kind), dtype=torch.uint8, device="cuda")
        scales = torch.empty(rows, dtype=torch.float32, device="cuda")
        sdm.undo_quantize(shape, t, kind, codes, scales)
        out.append((codes.cpu().numpy().reshape(rows, -1), scales.cpu().numpy()))
    assert np.array_equal(out[0][1], out[1][1])
    want = out[0][0].copy()
    if kind == "fp8":
        want[2, 7] = want[5, 60] = 0x7F
    assert np.array_equal(out[1][0], want)


# ------------------------------------------------------------------ norm-gate and head mix

@pytest.mark.parametrize("dtype,B,H,T,dv", [("bf16", 1, 1, 1, 8), ("bf16", 3, 5, 7, 24), ("bf16", 2, 3, 67, 320),
                                            ("f32", 1, 7, 33, 192), ("f32", 5, 1, 130, 4), ("f32", 2, 2, 9, 256)])
def test_norm_gate_row_widths(sdm, dtype, B, H, T, dv):
    """Rows of 1 to 64 vectors, row counts that leave the last pass partly empty: every element within
    (d_v / 2 + 6) 2^-24 of the float64 value plus one rounding to storage."""
    rng = np.random.default_rng(8)
    y = O.round_storage(rng.standard_normal((B, H, T, dv)), dtype)
    g = O.round_storage(1 / (1 + np.exp(-rng.standard_normal((B, H, T, dv)))), dtype)
    gamma = (1 + 0.1 * rng.standard_normal(dv)).astype(np.float32)
    shape = sdm.SdmShape.make(B, H, T, 32, dv, 1000, 3, 3, dtype)
    z = torch.full((B, T, H, dv), 3.0, dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device="cuda")
    sdm.norm_gate(shape, _stored(y, dtype), _stored(g, dtype), _cuda(gamma), 1e-6, z)
    ref = (g * gamma.astype(np.float64) * y / np.sqrt((y * y).mean(-1, keepdims=True) + 1e-6)).transpose(0, 2, 1, 3)
    bound = np.abs(ref) * ((dv / 2 + 6) * 2.0 ** -24 + (2.0 ** -8 if dtype == "bf16" else 2.0 ** -23))
    assert np.all(np.abs(z.double().cpu().numpy() - ref) <= bound)


@pytest.mark.parametrize("M,N,K", [(9000, 544, 120), (257, 19488, 64), (128 * 1024, 32, 200)])
def test_head_mix_pair_tiles(sdm, M, N, K):
    """The paired-CTA head mix (a tile for every pair of SMs) with ragged last tiles in M, N and K: every
    element within the blocked-accumulation bound 18 ceil(K / 16) 2^-23 sum |z w| plus one bf16 rounding."""
    g = torch.Generator(device="cuda").manual_seed(2)
    rn = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    z, w = rn(M, K), rn(N, K)
    out = torch.full((M, N), 5.0, dtype=torch.bfloat16, device="cuda")
    shape = sdm.SdmShape.make(1, 1, M, 32, K, 1000, 3, 3, "bf16")
    sdm.head_mix(shape, N, z, w, out)
    ref = z.double() @ w.double().t()
    bound = 18 * -(-K // 16) * 2.0 ** -23 * (z.double().abs() @ w.double().abs().t()) + 2.0 ** -8 * ref.abs()
    assert bool(((out.double() - ref).abs() <= bound).all())
    assert sdm.device_status() == 0


# The one-launch kernels for small problems against the kernels for large ones: the same tokens, alone and inside a
# batch beyond the small range, give the same bits.  Sizes: one token per CTA and several, a short last CTA, halves
# that fill no block of P, one and two of them, two rounds of TMEM; the fp32 path with short rows of P, several
# pieces of a row, rows that fill no group, misaligned operands; k at both list lengths' ends.
@pytest.mark.parametrize("dtype,B,H,T,dk,S,kw,kr,shift", [
    ("bf16", 1, 2, 1, 128, 16, 1, 3, False), ("bf16", 3, 5, 1, 64, 130, 32, 31, False), ("bf16", 1, 3, 41, 128, 250, 16, 9, False),
    ("bf16", 2, 2, 200, 128, 513, 32, 32, False), ("bf16", 9, 16, 1, 128, 512, 17, 32, False), ("bf16", 1, 1, 9, 64, 1024, 8, 8, False),
    ("f32", 1, 2, 1, 128, 64, 32, 20, False), ("f32", 2, 3, 37, 36, 50, 8, 5, True), ("f32", 1, 4, 5, 256, 300, 33 - 1, 1, False),
    ("f32", 3, 1, 1, 4, 16, 4, 16, False), ("bf16", 1, 3, 50, 40, 100, 12, 16, True), ("bf16", 2, 2, 3, 256, 65, 20, 32, False)])
def test_small_problems_select_as_large_ones(sdm, dtype, B, H, T, dk, S, kw, kr, shift):
    g = torch.Generator(device="cuda").manual_seed(S + T)
    st = torch.bfloat16 if dtype == "bf16" else torch.float32
    rn = lambda *s: torch.randn(s, generator=g, device="cuda").to(st)
    P = [rn(H, 2 * S, dk) for _ in range(2)]
    TT = T + 8400 // (2 * H * B) + 1                     # more than 8192 token-sides
    x = [rn(B, H, TT, dk) for _ in range(2)]

    def lists(T_, P_, xs):
        sh = sdm.SdmShape.make(B, H, T_, dk, 16, S * S, kw, kr, dtype)
        o = [torch.empty((B, H, T_, k), dtype=t, device="cuda") for k, t in
             ((kw, torch.int32), (kw, torch.float32), (kr, torch.int32), (kr, torch.float32))]
        ws = torch.empty(sdm.workspace_bytes(sh), dtype=torch.uint8, device="cuda")
        sdm.address(sh, P_[0], P_[1], xs[0], xs[1], *o, ws)
        return o

    full = lists(TT, P, x)
    if shift:
        P = [_shifted(p) for p in P]
    for at in (0, TT - T):
        part = lists(T, P, [t[:, :, at:at + T].contiguous() for t in x])
        assert sdm.device_status() == 0
        for f, p in zip(full, part):
            assert torch.equal(f[:, :, at:at + T], p)
