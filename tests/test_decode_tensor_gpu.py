"""The decode's tensor-core streaming kernel (bf16, d = 64 and 128) at the edges of its tiles of 64 keys, with the options
that change which rows a tile reads, with short caches beside long ones, and with a first tile whose maximum is useless
as the reference of the weights.  Tolerances are those of the other bf16 parity tests on an fp32 output buffer."""
import ctypes
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2510_01450_b200 import binding as L, inputs
from tests.conftest import ROOT
from tests.gpu_util import dev, row_err, stream_ptr
from tests.test_parity_gpu import TOL_BF16, _to_pages

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,mode,splits", [(64, "plain", 1), (64, "late_max", 1), (64, "late_max", 2), (64, "short", 1), (64, "plain", 12),
                                           (128, "plain", 1), (128, "plain", 3), (128, "plain", 12), (128, "late_max", 1),
                                           (128, "late_max", 2), (128, "short", 1), (128, "paged_gqa", 1), (128, "paged_gqa", 2),
                                           (128, "paged_gqa_short", 1), (128, "window", 1)])
def test_tile_edges_and_options(oracle, d, mode, splits):
    H, Hkv = 4, 2 if mode.startswith("paged_gqa") else 4
    w = inputs.CONFIGS[5].shrink(B=6, H=H, n=1100, d=d, dv=d, len_min=10, len_max=1100, seed=400 + d)
    q, _, _, _ = inputs.make_decode(w)
    _, kc, vc, _ = inputs.make_decode(w.shrink(H=Hkv))
    lens = np.array([2 * d, 2 * d + 1, 319, 384, 385, 1100], dtype=np.int32)
    if mode.endswith("short"):
        lens[:3] = [1, 17, 2 * d - 1]           # solved directly
    kw = {}
    if mode == "late_max":
        # the first 64 keys score about 2^100 below the rest
        qn = q / (np.linalg.norm(q, axis=-1, keepdims=True) ** 2)
        kc[:, :, :64] += (-70.0 / w.scale) * qn[:, :, None, :]
        kc = inputs.round_to_bf16(kc)
    if mode == "window":
        kw["window"] = 2 * d + 17
        cnt = np.minimum(lens, kw["window"]).astype(np.int32)
        kr, vr = np.zeros_like(kc), np.zeros_like(vc)
        for b in range(w.B):
            kr[b, :, : cnt[b]], vr[b, :, : cnt[b]] = (x[b, :, lens[b] - cnt[b]: lens[b]] for x in (kc, vc))
        ref = oracle.decode(q, kr, vr, cnt, w.scale, w.lam)
    else:
        ref = oracle.decode(q, np.repeat(kc, H // Hkv, axis=1), np.repeat(vc, H // Hkv, axis=1), lens, w.scale, w.lam)
    for b in range(w.B):                      # slots past the end may hold anything
        kc[b, :, lens[b]:] = np.nan
        vc[b, :, lens[b]:] = np.nan
    if mode.startswith("paged_gqa"):         # pages of 128 keys: the directly solved 2 d - 1 keys take two of them at d = 128
        kc, table, max_pages, num_pages = _to_pages(kc, lens, 128, np.random.default_rng(401))
        vc, _, _, _ = _to_pages(vc, lens, 128, np.random.default_rng(401))
        kw.update(kv_heads=Hkv, block_table=torch.from_numpy(table).cuda(), page_size=128, max_pages=max_pages, num_pages=num_pages)
    dq, dk, dv_, dl = dev(q, "bf16"), dev(kc, "bf16"), dev(vc, "bf16"), torch.from_numpy(lens).cuda()
    nbytes = 4 * w.B * H * splits * (2 * d * d + 2 * d + 4)
    # with room for the moment records in the workspace, and (one part) without a workspace
    for ws in [torch.empty(nbytes, dtype=torch.uint8, device="cuda")] + ([None] if splits == 1 else []):
        status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
        out = torch.full((w.B, H, d), float("nan"), dtype=torch.float32, device="cuda")
        L.lla_decode_ex(dq, dk, dv_, dl, out, w.B, H, w.n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32, splits=splits,
                        device_status=status, workspace=ws, workspace_bytes=nbytes if ws is not None else 0, stream=stream_ptr(), **kw)
        torch.cuda.synchronize()
        err = row_err(out.cpu().numpy(), ref)
        assert np.isfinite(err).all() and err.max() <= TOL_BF16, (float(err.max()), int(err.argmax()))
        assert status.cpu().numpy()[L.STATUS_TIMEOUT] == 0


@pytest.mark.parametrize("d", [64, 128])
def test_solve_falls_back_to_elimination(oracle, d):
    """Keys on which the conjugate gradients of the solve do not converge within their cap (features scaled over six
    decades, a tiny ridge): the elimination must take over.  The reference is the oracle's own direct solve; fp32 moments
    bound what can be asked: the output is an affine fit, so it reproduces values that are affine in the keys."""
    B, H, n = 2, 2, 700
    rng = np.random.default_rng(410 + d)
    sc = np.logspace(0, -3, d).astype(np.float32)
    kc = inputs.round_to_bf16(rng.standard_normal((B, H, n, d)).astype(np.float32) * sc)
    q = inputs.round_to_bf16(rng.standard_normal((B, H, d)).astype(np.float32) * sc * 0.5)
    vc = inputs.round_to_bf16(np.einsum("bhjc,ec->bhje", kc, rng.standard_normal((d, d)).astype(np.float32)) + 1.0)
    lens = np.array([n, 520], dtype=np.int32)
    lam = 1e-9
    ref = oracle.decode(q, kc, vc, lens, 0.1, lam)
    out = torch.full((B, H, d), float("nan"), dtype=torch.float32, device="cuda")
    ws = torch.empty(4 * B * H * (2 * d * d + 2 * d + 4), dtype=torch.uint8, device="cuda")
    L.lla_decode_ex(dev(q, "bf16"), dev(kc, "bf16"), dev(vc, "bf16"), torch.from_numpy(lens).cuda(), out, B, H, n, d, d, 0.1, lam,
                    out_dtype=L.LLA_F32, splits=1, workspace=ws, workspace_bytes=ws.numel(), stream=stream_ptr())
    torch.cuda.synchronize()
    # bf16 operand pairs of w k carry 2^-17 relative error per key, features at 1e-3 of the largest: 1e-2 covers it
    assert row_err(out.cpu().numpy(), ref).max() <= 1e-2


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("mode", ["zero", "constant", "paired"])
def test_query_at_the_weighted_key_mean(oracle, d, mode):
    """A right-hand side of the solve that is exactly zero: the slope term vanishes and the output is the weighted value
    mean.  Runs behind an ordinary decode, so that shared memory holds another unit's solution."""
    B, H, n = 2, 4, 512
    w = inputs.CONFIGS[5].shrink(B=B, H=H, n=n, d=d, dv=d, len_min=n, len_max=n, seed=430 + d)
    q, kc, vc, _ = inputs.make_decode(w)
    lens = np.array([n, 256], dtype=np.int32)          # (powers of two: the mean of equal keys is exact)
    q0, k0 = np.zeros_like(q), np.zeros_like(kc)
    if mode == "constant":
        q0 = q.copy()
        k0 = np.ascontiguousarray(np.broadcast_to(q[:, :, None], kc.shape))
    if mode == "paired":                              # keys in +/- pairs, a zero query
        k0 = kc.copy()
        k0[:, :, 1::2] = -k0[:, :, ::2]
    ref = oracle.decode(q0, k0, vc, lens, w.scale, w.lam)
    nbytes = 4 * B * H * (2 * d * d + 2 * d + 4)
    dl, dv_ = torch.from_numpy(lens).cuda(), dev(vc, "bf16")
    for ws in (torch.empty(nbytes, dtype=torch.uint8, device="cuda"), None):
        for qq, kk in ((q, kc), (q0, k0)):
            out = torch.full((B, H, d), float("nan"), dtype=torch.float32, device="cuda")
            L.lla_decode_ex(dev(qq, "bf16"), dev(kk, "bf16"), dv_, dl, out, B, H, n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32,
                            splits=1, workspace=ws, workspace_bytes=nbytes if ws is not None else 0, stream=stream_ptr())
        torch.cuda.synchronize()
        err = row_err(out.cpu().numpy(), ref)
        assert np.isfinite(err).all() and err.max() <= TOL_BF16, (float(err.max()), int(err.argmax()))


def test_more_parts_than_the_merge_takes(oracle):
    """More than 64 parts: at d = 128 the call runs (with a caller's buffer and with the library's), at d = 64 it is refused
    before anything has been launched."""
    B, H, n, splits = 1, 2, 6000, 80
    for d in (128, 64):
        w = inputs.CONFIGS[5].shrink(B=B, H=H, n=n, d=d, dv=d, len_min=n, len_max=n, seed=440 + d)
        q, kc, vc, lens = inputs.make_decode(w)
        lens = np.array([n if d == 128 else 2 * d - 1], dtype=np.int32)
        args = [dev(q, "bf16"), dev(kc, "bf16"), dev(vc, "bf16"), torch.from_numpy(lens).cuda()]
        nbytes = L.lla_decode_workspace_bytes(B, H, n, d, d, L.LLA_BF16, splits)
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")

        def run(call, **kw):
            out = torch.full((B, H, d), float("nan"), dtype=torch.float32, device="cuda")
            try:
                call(*args, out, B, H, n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32, splits=splits, stream=stream_ptr(), **kw)
                status = 0
            except L.LlaError as e:
                status = e.status
            torch.cuda.synchronize()
            return status, out.cpu().numpy()

        for call, kw in ((L.lla_decode_ex, dict(workspace=ws, workspace_bytes=nbytes)), (L.lla_decode_noalloc, {})):
            status, got = run(call, **kw)
            if d == 128:
                assert status == 0
                err = row_err(got, oracle.decode(q, kc, vc, lens, w.scale, w.lam))
                assert err.max() <= TOL_BF16, float(err.max())
            else:
                assert status == 1 and np.isnan(got).all()          # invalid argument, and no kernel has written


def _decode_d128(seed):
    B, H, n, d = 4, 4, 1100, 128
    w = inputs.CONFIGS[5].shrink(B=B, H=H, n=n, d=d, dv=d, len_min=10, len_max=n, seed=seed)
    q, kc, vc, _ = inputs.make_decode(w)
    lens = np.array([100, 2 * d, 385, n], dtype=np.int32)
    return w, (q, kc, vc, lens), [dev(q, "bf16"), dev(kc, "bf16"), dev(vc, "bf16"), torch.from_numpy(lens).cuda()]


def test_captured_calls_allocate_nothing(oracle):
    """d = 128 without a buffer for the records, captured: the graph holds no allocation (a clone of it can be made) and its
    replays are right."""
    w, (q, kc, vc, lens), args = _decode_d128(450)
    d = w.d
    ref = oracle.decode(q, kc, vc, lens, w.scale, w.lam)
    for splits in (0, 1):
        out = torch.empty((w.B, w.H, d), dtype=torch.float32, device="cuda")
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph):
            L.lla_decode_ex(*args, out, w.B, w.H, w.n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32, splits=splits, stream=stream_ptr())
        cuda, clone = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
        assert cuda.cuGraphClone(ctypes.byref(clone), ctypes.c_void_p(graph.raw_cuda_graph())) == 0
        assert cuda.cuGraphDestroy(clone) == 0
        for _ in range(3):
            out.fill_(float("nan"))
            graph.replay()
            torch.cuda.synchronize()
            err = row_err(out.cpu().numpy(), ref)
            assert np.isfinite(err).all() and err.max() <= TOL_BF16, float(err.max())


def test_the_default_pool_is_left_alone():
    """d = 128 without a buffer for the records: they come from a pool of the library's own (in a process of its own, for
    other entry points do set the default pool's threshold)."""
    code = """
import ctypes, torch
from tests.test_decode_tensor_gpu import L, _decode_d128, stream_ptr
w, _, args = _decode_d128(451)
cuda, pool, value = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_uint64(77)
def threshold():
    assert cuda.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert cuda.cuMemPoolGetAttribute(pool, 4, ctypes.byref(value)) == 0
    return value.value
before = threshold()
out = torch.empty((w.B, w.H, w.d), dtype=torch.float32, device="cuda")
L.lla_decode_ex(*args, out, w.B, w.H, w.n, w.d, w.d, w.scale, w.lam, out_dtype=L.LLA_F32, stream=stream_ptr())
torch.cuda.synchronize()
print("thresholds", before, threshold())
"""
    res = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]
    _, before, after = res.stdout.split()[-3:]
    assert before == after
