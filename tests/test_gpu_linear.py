"""The projection kernel through the C-ABI (dvi_linear): tcgen05/TMA for bf16,
FP32 FMA for f32, against a float64 matmul of the (bf16-rounded) weights and
the f32 input -- the bf16 kernel carries the input as a bf16 pair hi + lo, so
only the weights are rounded -- over shapes spanning several 128-row tiles,
split-K and ragged tails.
Also: bitwise determinism, and a row's result does not depend on how many
rows share the launch (what makes the verify pass agree bit for bit with AR
decoding)."""
import numpy as np
import pytest
import torch

from workloads import workload
from workloads.gen import bf16_round
from gpu_helpers import engine_for

pytestmark = pytest.mark.gpu

SHAPES = [(128, 64, 1), (256, 256, 5), (384, 4096, 16), (1000, 512, 17), (4096, 4096, 40),
          (512, 11008, 5), (32000, 4096, 1), (640, 2048, 128), (256, 1024, 256), (12288, 4096, 5)]


@pytest.fixture(scope="module", params=["bf16", "f32"])
def eng(request):
    w = workload("tiny")
    e, _, _ = engine_for(w, dtype=request.param, use_graphs=False)
    yield e
    e.close()


def _case(n_out, k, m, dtype, seed):
    g = np.random.default_rng(seed)
    W = (g.standard_normal((n_out, k)) * 0.02).astype(np.float32)
    X = g.standard_normal((m, k)).astype(np.float32)
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    Wd = torch.from_numpy(W).cuda().to(td)
    Xd = torch.from_numpy(X).cuda()
    if dtype == "bf16":
        W = bf16_round(W)
    ref = X.astype(np.float64) @ W.astype(np.float64).T
    return Wd, Xd, ref


@pytest.mark.parametrize("shape", SHAPES)
def test_linear_matches_float64(eng, shape):
    n_out, k, m = shape
    Wd, Xd, ref = _case(n_out, k, m, eng.dtype, hash(shape) % 1000)
    y = eng.linear(Wd, Xd)
    torch.cuda.synchronize()
    y = y.cpu().numpy().astype(np.float64)
    scale = np.abs(ref).max()
    err = np.abs(y - ref).max() / scale
    assert err < (2e-5 if eng.dtype == "f32" else 1e-4), err
    assert eng.stats()["device_status"] == 0


def test_linear_deterministic_and_row_independent(eng):
    Wd, Xd, _ = _case(4096, 4096, 40, eng.dtype, 7)
    y1 = eng.linear(Wd, Xd)
    y2 = eng.linear(Wd, Xd)
    y_one = eng.linear(Wd, Xd[:1].contiguous())
    y_five = eng.linear(Wd, Xd[:5].contiguous())
    torch.cuda.synchronize()
    assert torch.equal(y1, y2)
    assert torch.equal(y_one[0], y1[0])
    assert torch.equal(y_five, y1[:5])


@pytest.mark.parametrize("n,k,m,off", [(1, 1, 1, 0), (130, 33, 3, 0), (130, 66, 5, 1), (300, 100, 4, 1),
                                       (257, 1000, 17, 3), (64, 31, 16, 2)])
def test_f32_any_k_and_alignment(n, k, m, off):
    """The f32 kernel's weight blocks: K not a multiple of 4 or of the block,
    operands at any 4-byte address (no float4 loads then), row counts on both
    sides of the four-column variant; against a float64 matmul."""
    from paper_2510_05421_gb300.dvi import linear_noalloc
    g = np.random.default_rng(n + k)
    W = g.standard_normal((n, k)).astype(np.float32)
    X = g.standard_normal((m, k)).astype(np.float32)
    w = torch.empty(n * k + off, device="cuda")[off:].view(n, k)
    x = torch.empty(m * k + off, device="cuda")[off:].view(m, k)
    w.copy_(torch.from_numpy(W))
    x.copy_(torch.from_numpy(X))
    y = torch.empty(m, n, device="cuda")
    assert linear_noalloc(w, x, y) == 0
    torch.cuda.synchronize()
    ref = X.astype(np.float64) @ W.astype(np.float64).T
    # K products and sums of f32: at most (K + 1) 2^-24 of sum |x||w|
    bound = (k + 1) * 2.0 ** -24 * (np.abs(X).astype(np.float64) @ np.abs(W).astype(np.float64).T)
    assert (np.abs(y.cpu().numpy() - ref) <= bound).all()


# columns of the second weight and rows it is multiplied with: one K range;
# ranges that meet in a cluster; in global scratch (more than four rows, more
# than eight ranges)
CHAINED = [(64, 4), (512, 4), (512, 16), (4096, 4)]


@pytest.mark.parametrize("entry", ["noalloc", "context"])
@pytest.mark.parametrize("k,m", CHAINED)
def test_f32_weight_is_the_output_of_the_call_before(entry, k, m):
    """y = x a^T (24 rows), then z = q y^T right behind it on the same stream: the second
    call reads its weight only when the first is done.  Bit for bit the same
    calls with a synchronisation between them; y is NaN before each pair."""
    import ctypes
    from paper_2510_05421_gb300.dvi import lib, linear_noalloc
    g = torch.Generator(device="cuda")
    g.manual_seed(k + m)
    a = torch.randn(k, 2048, device="cuda", generator=g)
    q = torch.randn(m, k, device="cuda", generator=g)
    e, _, _ = engine_for(workload("tiny"), use_graphs=False)
    torch.cuda.synchronize()

    def linear(w, x, y):
        if entry == "noalloc":
            return linear_noalloc(w, x, y, stream=e.stream)
        p = [ctypes.c_void_p(t.data_ptr()) for t in (w, x, y)]
        return lib().dvi_linear(e.ctx, p[0], w.shape[0], w.shape[1], p[1], x.shape[0], p[2])

    def pair(x, between):
        y = torch.full((24, k), float("nan"), device="cuda")
        z = torch.full((m, 24), float("nan"), device="cuda")
        torch.cuda.synchronize()
        assert linear(a, x, y) == 0
        between()
        assert linear(y, q, z) == 0
        torch.cuda.synchronize()
        return y, z

    for _ in range(10):
        x = torch.randn(24, 2048, device="cuda", generator=g)
        y1, z1 = pair(x, lambda: None)
        y2, z2 = pair(x, torch.cuda.synchronize)
        assert torch.equal(y1, y2) and torch.equal(z1, z2)
    assert e.stats()["device_status"] == 0
    e.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_projection_right_behind_the_update_that_steps_its_weight(dtype):
    """linear_noalloc on W^S right behind a full-head update on the engine's
    stream multiplies the stepped W^S (bit for bit the call after a
    synchronisation), which the step has moved."""
    from dataclasses import replace
    from workloads import make_prompts
    from paper_2510_05421_gb300.dvi import linear_noalloc
    w = workload("tiny")
    w = w.with_(shape=replace(w.shape, d_model=512, vocab=8192), dtype=dtype, update_every=4)
    e, _, dw = engine_for(w, head_mode=1)
    P = make_prompts(w)
    u = torch.randn(4, 512, device="cuda")
    y1, y2, old = (torch.full((4, 8192), float("nan"), device="cuda") for _ in range(3))
    torch.cuda.synchronize()
    for _ in range(3):
        e.generate(P, 10 ** 6, max_steps=w.update_every, log=True)
        assert linear_noalloc(dw.draft_head, u, old, stream=e.stream) == 0
        e.sync()
        e.update(w.update)
        assert linear_noalloc(dw.draft_head, u, y1, stream=e.stream) == 0
        e.sync()
        assert linear_noalloc(dw.draft_head, u, y2, stream=e.stream) == 0
        e.sync()
        assert torch.equal(y1, y2)
        assert not torch.equal(y1, old)
    assert e.stats()["device_status"] == 0
    e.close()
