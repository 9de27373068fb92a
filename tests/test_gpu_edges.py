"""Kernel edges: sizes at which a tile, slice, vector or window of the kernels is partly empty.

Bars follow tests/test_gpu_parity.py: selected slots bit-exact; gradients of the backward within
1e-4 (fp32) or 5e-3 (bf16) relative Frobenius of the oracle's; quantised codes and scales bit-exact.
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
