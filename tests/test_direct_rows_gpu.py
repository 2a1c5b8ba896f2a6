"""The fp64 direct rows at the edges of their chunks of keys, of the rows of a block and of the two forms of the system:
every row of a problem with fp32 inputs or d = 16, and the short rows of the backward.  Each forward row is checked against
the oracle's single-query routine over exactly its visible keys."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2510_01450_b200 import binding as L, inputs
from tests.gpu_util import LLA_DT, dev, row_err, stream_ptr
from tests.test_backward_gpu import TOL, grad_err, run_backward
from tests.test_parity_gpu import TOL_BF16, TOL_F32

pytestmark = pytest.mark.gpu


# n around the chunk (64 keys at d = 16; 128, in longer blocks 64, at d = 64; 136, in longer blocks 128, at d = 128), one row,
# rows that do not fill a block's teams
@pytest.mark.parametrize("dtype,d,n,nq,H,Hkv,window,causal,mode", [
    ("f32", 16, 1, 1, 1, 1, 0, True, ""), ("f32", 16, 64, 64, 2, 2, 0, True, ""), ("f32", 16, 65, 65, 3, 1, 0, True, ""),
    ("bf16", 16, 131, 70, 2, 1, 0, True, ""), ("f32", 16, 193, 193, 1, 1, 40, True, ""), ("f32", 16, 97, 30, 2, 2, 0, False, ""),
    ("f32", 64, 127, 127, 1, 1, 0, True, ""), ("f32", 64, 128, 128, 2, 1, 0, True, ""), ("f32", 64, 129, 129, 1, 1, 0, True, ""),
    ("f32", 64, 132, 132, 1, 1, 0, True, ""), ("f32", 64, 193, 193, 1, 1, 0, True, ""), ("f32", 128, 136, 136, 1, 1, 0, True, ""),
    ("f32", 64, 72, 72, 2, 2, 0, True, ""), ("f32", 64, 73, 73, 1, 1, 0, True, ""), ("f32", 64, 217, 75, 4, 2, 0, True, ""),
    ("f32", 64, 300, 300, 1, 1, 131, True, ""), ("f32", 64, 145, 9, 2, 1, 0, False, ""), ("f32", 64, 310, 40, 2, 2, 0, True, "late_max"),
    ("f32", 64, 64, 33, 1, 1, 0, False, ""), ("f32", 128, 137, 137, 1, 1, 0, True, ""), ("f32", 128, 300, 70, 2, 1, 0, True, "late_max"),
    ("f32", 128, 129, 3, 2, 2, 0, False, ""), ("f32", 128, 300, 45, 1, 1, 256, True, "")])
def test_every_row_direct(oracle, dtype, d, n, nq, H, Hkv, window, causal, mode):
    B = 2
    w = inputs.CONFIGS[2].shrink(B=B, H=H, n=n, d=d, dv=d, dtype=dtype, seed=700 + d + n)
    q, _, _ = inputs.make_prefill(w)
    _, k, v = inputs.make_prefill(w.shrink(H=Hkv, seed=701 + n))
    qc = np.ascontiguousarray(q[:, :, n - nq:])
    if mode == "late_max":       # the first 100 keys score about e^-700 below the rest: the reference of the weights moves
        u = np.ones(d, dtype=np.float32) / np.sqrt(d)
        qc = qc - (qc @ u)[..., None] * u + 4 * u
        k = k - (k @ u)[..., None] * u
        k[:, :, :100] -= (175.0 / w.scale) * u
    rnd = inputs.round_to_bf16 if dtype == "bf16" else (lambda x: x.astype(np.float32))
    qc, k, v = rnd(qc), rnd(k), rnd(v)
    out = torch.full((B, H, nq, d), float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
    iters = torch.full((B, H, nq), -7, dtype=torch.int32, device="cuda")
    L.lla_forward_ex(dev(qc, dtype), dev(k, dtype), dev(v, dtype), out, B, H, n, d, d, w.scale, w.lam, causal=causal,
                     in_dtype=LLA_DT[dtype], out_dtype=L.LLA_F32, q_rows=nq, kv_heads=Hkv, window=window, iters=iters,
                     device_status=status, stream=stream_ptr())
    torch.cuda.synchronize()
    assert status.cpu().numpy()[L.STATUS_BAD_PIVOT] == 0
    it = iters.cpu().numpy()
    seen = np.array([n - nq + r + 1 if causal else n for r in range(nq)])
    head_rows = 2 * d if dtype == "f32" else d + d // 2
    assert (it == np.where(seen < head_rows, -1, 0)).all()
    kk, vv = np.repeat(k, H // Hkv, axis=1), np.repeat(v, H // Hkv, axis=1)
    lo = np.maximum(0, seen - window) if causal and window else np.zeros(nq, dtype=int)
    cnt = (seen - lo).astype(np.int32)
    for b in range(B):
        kc = np.zeros((nq, H, cnt.max(), d), dtype=np.float32)
        vc = np.zeros_like(kc)
        for r in range(nq):
            kc[r, :, :cnt[r]], vc[r, :, :cnt[r]] = kk[b, :, lo[r]:seen[r]], vv[b, :, lo[r]:seen[r]]
        ref = oracle.decode(np.ascontiguousarray(qc[b].transpose(1, 0, 2)), kc, vc, cnt, w.scale, w.lam)
        err = row_err(out.cpu().numpy()[b].transpose(1, 0, 2), ref)
        assert np.isfinite(err).all() and err.max() <= (TOL_F32 if dtype == "f32" else TOL_BF16), (b, float(err.max()), int(err.argmax()))


# lengths at which every row is direct (up to 1.5 d - 1 keys) or nearly, and which leave part of a block's rows empty
@pytest.mark.parametrize("d,n,H", [(64, 2, 1), (64, 5, 3), (64, 64, 1), (64, 65, 2), (64, 95, 1), (64, 97, 2), (128, 3, 1),
                                   (128, 128, 2), (128, 130, 1), (128, 191, 1), (128, 193, 1)])
def test_backward_short_rows(backward_oracle, d, n, H):
    w = inputs.CONFIGS[2].shrink(B=1, H=H, n=n, d=d, dv=d, seed=800 + d + n)
    q, k, v = inputs.make_prefill(w)
    g = inputs.make_upstream_grad(w)
    ref = backward_oracle.backward(q, k, v, g, w.scale, w.lam)
    for name, a, b in zip(("dq", "dk", "dv"), run_backward(w, q, k, v, g), ref):
        assert np.isfinite(a).all(), name
        err = grad_err(a, b)
        assert err.max() <= TOL, (name, float(err.max()), int(err.argmax()))


# calls large enough that the rows with many keys go to the conjugate gradients instead: part of the rows of a causal call,
# every row of a non-causal one
@pytest.mark.parametrize("n,nq,B,H,causal", [(1500, 1500, 2, 8, True), (1100, 1100, 2, 8, False), (2000, 700, 2, 8, True)])
def test_direct_and_iterative_rows_side_by_side(oracle, n, nq, B, H, causal):
    d = 128
    w = inputs.CONFIGS[2].shrink(B=B, H=H, n=n, d=d, dv=d, dtype="f32", seed=900 + n)
    q, k, v = inputs.make_prefill(w)
    qc = np.ascontiguousarray(q[:, :, n - nq:])
    out = torch.full((B, H, nq, d), float("nan"), dtype=torch.float32, device="cuda")
    iters = torch.full((B, H, nq), -7, dtype=torch.int32, device="cuda")
    L.lla_forward_ex(dev(qc, "f32"), dev(k, "f32"), dev(v, "f32"), out, B, H, n, d, d, w.scale, w.lam, causal=causal,
                     in_dtype=L.LLA_F32, out_dtype=L.LLA_F32, q_rows=nq, iters=iters, stream=stream_ptr())
    torch.cuda.synchronize()
    assert torch.isfinite(out).all()
    it = iters.cpu().numpy()
    assert (it >= -1).all() and (it[:, :, -1] > 0).all()
    cut = int(np.argmax(it[0, 0] > 0))                       # the first row of the iterative kernel
    assert (it[:, :, cut:] > 0).all() and (it[:, :, :cut] <= 0).all()
    rows = np.unique(np.clip([0, cut - 1, cut, cut + 1, nq // 2, nq - 1], 0, nq - 1))
    cnt = np.array([n - nq + r + 1 if causal else n for r in rows], dtype=np.int32)
    for b in range(B):
        kc = np.repeat(k[b][None], len(rows), axis=0)
        vc = np.repeat(v[b][None], len(rows), axis=0)
        ref = oracle.decode(np.ascontiguousarray(qc[b][:, rows].transpose(1, 0, 2)), kc, vc, cnt, w.scale, w.lam)
        err = row_err(out.cpu().numpy()[b][:, rows].transpose(1, 0, 2), ref)
        assert err.max() <= TOL_F32, (b, float(err.max()), int(err.argmax()))


def _scores_far_from_zero(dtype, d, n, mode):
    """Raw scores far below zero, where the systems' diagonal lambda e^{-s_j} is beyond 1e154: of every key ("low") or
    of every other key ("mixed"); or pairs of keys that equal the query, whose diagonal is lambda e^{-s} below 1e-154 ("high")."""
    rng = np.random.default_rng(950 + d + n)
    scale = np.float32(d ** -0.5)
    u = np.ones(d, dtype=np.float32) / np.float32(np.sqrt(d))
    a = np.float32(np.sqrt({"low": 520.0, "mixed": 520.0, "high": 600.0}[mode] / scale))
    noise = lambda: rng.standard_normal((1, 2, n, d)).astype(np.float32) * scale
    q, k, v = a * u + noise(), noise(), noise() * np.float32(np.sqrt(d))
    if mode == "low":
        k -= a * u
    if mode == "mixed":
        k[:, :, ::2] -= a * u
    if mode == "high":
        q[:] = a * u
        k[:, :, :2] = a * u
    rnd = inputs.round_to_bf16 if dtype == "bf16" else (lambda x: x.astype(np.float32))
    return (*map(rnd, (q, k, v)), float(scale))


FAR_SIZES = [("bf16", 64, 95), ("f32", 16, 130), ("f32", 64, 200), ("bf16", 128, 140), ("f32", 128, 150)]


@pytest.mark.parametrize("dtype,d,n,mode", [(*size, mode) for size in FAR_SIZES for mode in ("low", "mixed", "high")])
def test_scores_far_from_zero(oracle, dtype, d, n, mode):
    q, k, v, scale = _scores_far_from_zero(dtype, d, n, mode)
    if mode == "high":
        # every row sees the two keys at its query: z = 0 for both, the others weigh e^-600 -- the mean of the two values
        # (rows with more than d keys are left out: e^-600 of the identity is no ridge in the explicit form)
        n = d
        q, k, v = (np.ascontiguousarray(x[:, :, :n]) for x in (q, k, v))
        ref = np.repeat(v[:, :, :2].astype(np.float64).mean(axis=2, keepdims=True), n, axis=2)
        ref[:, :, 0] = v[:, :, 0]
    else:
        ref = oracle.forward(q, k, v, scale, 1e-3)
    out = torch.full(q.shape, float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
    L.lla_forward_ex(dev(q, dtype), dev(k, dtype), dev(v, dtype), out, 1, 2, n, d, d, scale, 1e-3, in_dtype=LLA_DT[dtype],
                     out_dtype=L.LLA_F32, device_status=status, stream=stream_ptr())
    torch.cuda.synchronize()
    assert status.cpu().numpy()[L.STATUS_BAD_PIVOT] == 0
    err = row_err(out.cpu().numpy(), ref)
    assert np.isfinite(err).all() and err.max() <= (TOL_F32 if dtype == "f32" else TOL_BF16), (float(np.nanmax(err)), int(np.isnan(err).sum()))


@pytest.mark.parametrize("mode", ["low", "mixed"])
def test_backward_scores_far_from_zero(backward_oracle, mode):
    d, n = 64, 95
    q, k, v, scale = _scores_far_from_zero("bf16", d, n, mode)
    w = inputs.CONFIGS[2].shrink(B=1, H=2, n=n, d=d, dv=d)
    assert abs(w.scale - scale) < 1e-6
    g = inputs.make_upstream_grad(w)
    ref = backward_oracle.backward(q, k, v, g, w.scale, w.lam)
    for name, a, b in zip(("dq", "dk", "dv"), run_backward(w, q, k, v, g), ref):
        assert np.isfinite(a).all(), name
        err = grad_err(a, b)
        assert err.max() <= TOL, (name, float(err.max()), int(err.argmax()))


# (up to 2 d - 1 keys: the rows whose systems are ill-conditioned)
@pytest.mark.parametrize("d,n,nq", [(16, 31, 31), (64, 127, 127), (64, 110, 41), (128, 255, 255)])
def test_fp32_inputs_far_from_the_origin(oracle, d, n, nq):
    """Keys and queries around a common point 1000 times as far away as they are spread: squares of the coordinates leave
    1e-10 of a double beside a ridge of 1e-8, so the systems must be formed from differences."""
    rng = np.random.default_rng(970 + d + n)
    u = np.ones(d, dtype=np.float32) / np.float32(np.sqrt(d))
    q, k = ((1000.0 * u + rng.standard_normal((1, 2, m, d)) / np.sqrt(d)).astype(np.float32) for m in (nq, n))
    v = rng.standard_normal((1, 2, n, d)).astype(np.float32)
    scale, lam = 1e-5, 1e-3
    out = torch.full((1, 2, nq, d), float("nan"), dtype=torch.float32, device="cuda")
    rho = torch.full_like(out, float("nan"))
    L.lla_forward_ex(dev(q, "f32"), dev(k, "f32"), dev(v, "f32"), out, 1, 2, n, d, d, scale, lam, in_dtype=L.LLA_F32,
                     out_dtype=L.LLA_F32, q_rows=nq, rho=rho, stream=stream_ptr())
    torch.cuda.synchronize()
    cnt = np.arange(n - nq + 1, n + 1, dtype=np.int32)
    ref = oracle.decode(np.ascontiguousarray(q[0].transpose(1, 0, 2)), np.repeat(k, nq, axis=0), np.repeat(v, nq, axis=0), cnt, scale, lam)
    err = row_err(out.cpu().numpy()[0].transpose(1, 0, 2), ref)
    assert np.isfinite(err).all() and err.max() <= TOL_F32, (float(err.max()), int(err.argmax()))
    if n == nq:
        _, rref, _, _ = oracle.forward_rows(q, k, v, scale, lam, want_aux=True)
        assert row_err(rho.cpu().numpy(), rref)[1:].max() <= TOL_F32


# more blocks of rows than the second dimension of a grid holds (65535 blocks of four rows, two at d = 128)
@pytest.mark.parametrize("d,n,window", [(16, 262200, 64), (128, 131100, 384)])
def test_long_windowed_sequences(oracle, d, n, window):
    rng = np.random.default_rng(980 + d)
    q, k, v = (rng.standard_normal((1, 1, n, d), dtype=np.float32) / np.float32(s) for s in (d ** 0.5, d ** 0.5, 1.0))
    out = torch.full((1, 1, n, d), float("nan"), dtype=torch.float32, device="cuda")
    iters = torch.full((1, 1, n), -7, dtype=torch.int32, device="cuda")
    scale, lam = d ** -0.5, 1e-3
    L.lla_forward_ex(dev(q, "f32"), dev(k, "f32"), dev(v, "f32"), out, 1, 1, n, d, d, scale, lam, in_dtype=L.LLA_F32,
                     out_dtype=L.LLA_F32, window=window, iters=iters, stream=stream_ptr())
    torch.cuda.synchronize()
    assert torch.isfinite(out).all()
    last = 65535 * (2 if d == 128 else 4)
    assert (iters[0, 0, 2 * d:last] == 0).all() and (iters[0, 0, last:] > 0).all()
    rows = np.unique(np.concatenate([np.arange(4), [last - 1, last, last + 1], rng.integers(0, n, 30), [n - 2, n - 1]]))
    lo = np.maximum(0, rows + 1 - window)
    cnt = (rows + 1 - lo).astype(np.int32)
    kc, vc = (np.zeros((len(rows), 1, window, d), dtype=np.float32) for _ in range(2))
    for s, (r, l, c) in enumerate(zip(rows, lo, cnt)):
        kc[s, 0, :c], vc[s, 0, :c] = k[0, 0, l:r + 1], v[0, 0, l:r + 1]
    ref = oracle.decode(np.ascontiguousarray(q[0, :, rows].reshape(len(rows), 1, d)), kc, vc, cnt, scale, lam)
    err = row_err(out.cpu().numpy()[0, 0, rows], ref)
    assert err.max() <= TOL_F32, (float(err.max()), int(err.argmax()))


def _gradients(w, q, k, v, g, head_rows=0):
    """dq, dk, dv of a forward and a backward pass, whatever the status words say."""
    t = [dev(x, "bf16") for x in (q, k, v)]
    out, rho, dq, dk, dv_ = (torch.full(q.shape, float("nan"), dtype=torch.float32, device="cuda") for _ in range(5))
    stats = torch.empty((w.B, w.H, w.n, 3), dtype=torch.float32, device="cuda")
    nbytes = L.lla_backward_workspace_bytes(w.B, w.H, w.n, w.d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    L.lla_forward_ex(*t, out, w.B, w.H, w.n, w.d, w.d, w.scale, w.lam, out_dtype=L.LLA_F32, head_rows=head_rows, rho=rho, stats=stats,
                     stream=stream_ptr())
    L.lla_backward_ex(*t, out, dev(g, "f32"), rho, stats, dq, dk, dv_, w.B, w.H, w.n, w.d, w.scale, w.lam, head_rows=head_rows,
                      workspace=ws, workspace_bytes=nbytes, stream=stream_ptr())
    torch.cuda.synchronize()
    return [x.cpu().numpy().astype(np.float64) for x in (dq, dk, dv_)]


# head_rows raised beyond the default: rows with more than 2 d keys solved directly in both passes, part of a sequence or all of
# it, up to the most keys that the backward takes
@pytest.mark.parametrize("d,n,head_rows", [(64, 129, 130), (64, 300, 200), (64, 300, 301), (128, 262, 270), (128, 400, 324), (64, 1222, 1223)])
def test_backward_with_more_direct_rows(backward_oracle, d, n, head_rows):
    H = 1 if n > 1000 else 2
    w = inputs.CONFIGS[2].shrink(B=1, H=H, n=n, d=d, dv=d, seed=860 + d + n)
    q, k, v = inputs.make_prefill(w)
    g = inputs.make_upstream_grad(w)
    ref = backward_oracle.backward(q, k, v, g, w.scale, w.lam)
    # fp64 throughout where every row is direct: the gradients' own fp32 rounding and sums
    tol = 1e-5 if head_rows > n else TOL
    for name, a, b in zip(("dq", "dk", "dv"), _gradients(w, q, k, v, g, head_rows), ref):
        err = grad_err(a, b)
        assert np.isfinite(err).all() and err.max() <= tol, (name, float(err.max()), int(err.argmax()))


@pytest.mark.parametrize("dtype,d,n", [("bf16", 128, 180), ("f32", 128, 250)])
def test_reference_far_below_the_maximum(oracle, dtype, d, n):
    """The first 130 keys score near -740, the others near -160: the weights' reference is the former's maximum, where
    lambda e^-m has no double, the row's ridge is the latter's."""
    rng = np.random.default_rng(985 + n)
    scale = np.float32(d ** -0.5)
    u = np.ones(d, dtype=np.float32) / np.float32(np.sqrt(d))
    a = np.float32(np.sqrt(740.0 / scale))
    noise = lambda: rng.standard_normal((1, 2, n, d)).astype(np.float32) * scale
    q, k, v = a * u + noise() * np.float32(0.01), noise() * np.float32(0.1), noise() * np.float32(np.sqrt(d))
    k[:, :, :130] -= a * u
    k[:, :, 130:] -= np.float32(160.0 / 740.0) * a * u
    rnd = inputs.round_to_bf16 if dtype == "bf16" else (lambda x: x.astype(np.float32))
    q, k, v = map(rnd, (q, k, v))
    ref = oracle.forward(q, k, v, float(scale), 1e-3)[:, :, 140:]
    out = torch.full(q.shape, float("nan"), dtype=torch.float32, device="cuda")
    L.lla_forward_ex(dev(q, dtype), dev(k, dtype), dev(v, dtype), out, 1, 2, n, d, d, float(scale), 1e-3, in_dtype=LLA_DT[dtype],
                     out_dtype=L.LLA_F32, stream=stream_ptr())
    torch.cuda.synchronize()
    err = row_err(out.cpu().numpy()[:, :, 140:], ref)
    assert np.isfinite(err).all() and err.max() <= (TOL_F32 if dtype == "f32" else TOL_BF16), float(np.nanmax(err))


@pytest.mark.parametrize("dtype,d,n,window", [("bf16", 64, 95, 0), ("f32", 16, 100, 0), ("f32", 16, 100, 33), ("f32", 64, 150, 0),
                                              ("f32", 64, 300, 131), ("bf16", 128, 150, 0), ("f32", 128, 140, 0), ("f32", 128, 400, 258)])
@pytest.mark.parametrize("where", ["q", "k", "v"])
def test_infinities_stay_in_the_rows_that_see_them(dtype, d, n, window, where):
    """A query row that is not finite spoils its own output, a key or value those of the rows that see it: the rows beside them
    in a block come out as without it."""
    w = inputs.CONFIGS[2].shrink(B=1, H=1, n=n, d=d, dv=d, dtype=dtype, seed=990 + d + n)
    x = dict(zip("qkv", (dev(a, dtype) for a in inputs.make_prefill(w))))

    def run():
        out, rho = (torch.full((1, 1, n, d), 7.0, dtype=torch.float32, device="cuda") for _ in range(2))
        stats = torch.full((1, 1, n, 3), 7.0, dtype=torch.float32, device="cuda")
        L.lla_forward_ex(x["q"], x["k"], x["v"], out, 1, 1, n, d, d, w.scale, w.lam, in_dtype=LLA_DT[dtype],
                         out_dtype=L.LLA_F32, window=window, rho=rho, stats=stats, stream=stream_ptr())
        torch.cuda.synchronize()
        return out[0, 0], rho[0, 0], stats[0, 0]

    clean = run()
    assert all(torch.isfinite(c).all() for c in clean)
    for j in (0, 1, 4, 41, 43, 66, n - 2):
        for bad in (float("inf"), float("nan")):
            keep = x[where][0, 0, j, 3].clone()
            x[where][0, 0, j, 3] = bad
            got = run()
            x[where][0, 0, j, 3] = keep
            rows = torch.arange(n, device="cuda")
            seen = rows == j if where == "q" else (rows >= j) & ((rows < j + window) if window else (rows >= 0))
            assert not torch.isfinite(got[0][seen]).all(dim=1).any(), (j, bad)
            if where != "v":
                assert not torch.isfinite(got[1][seen]).all(dim=1).any() and not torch.isfinite(got[2][seen]).all(dim=1).any()
            # (the frame or the form of a row's matrix may be another beside it: fp32 rounding)
            for a, b in zip(got, clean):
                assert torch.allclose(a[~seen], b[~seen], rtol=1e-5, atol=1e-6 * float(b.abs().max())), (j, bad)


@pytest.mark.parametrize("d,n", [(64, 95), (128, 150)])
def test_backward_infinities_stay_in_the_rows_that_see_them(d, n):
    w = inputs.CONFIGS[2].shrink(B=1, H=1, n=n, d=d, dv=d, seed=995 + d)
    q, k, v = inputs.make_prefill(w)
    g = inputs.make_upstream_grad(w)
    clean = _gradients(w, q, k, v, g)
    same = lambda a, b: np.abs(a - b).max() <= 1e-5 * np.abs(b).max()      # (fp32 sums in another order)
    for j in (4, 40, 42):
        gb = g.copy()
        gb[0, 0, j, 3] = np.nan
        dq, dk, dv = _gradients(w, q, k, v, gb)
        rest = np.arange(n) != j
        assert np.isnan(dq[0, 0, j]).any() and same(dq[0, 0, rest], clean[0][0, 0, rest])
        for a, b in ((dk, clean[1]), (dv, clean[2])):         # keys up to j get a share of row j
            assert np.isnan(a[0, 0, : j + 1]).any(axis=1).all() and same(a[0, 0, j + 1:], b[0, 0, j + 1:])
        for which in (1, 2):
            bad = [q, k.copy(), v.copy()]
            bad[which][0, 0, j, 3] = np.nan
            dq = _gradients(w, *bad, g)[0]
            assert same(dq[0, 0, :j], clean[0][0, 0, :j]) and np.isnan(dq[0, 0, j:]).any(axis=1).all()
