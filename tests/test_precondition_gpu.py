"""The solver that a call with default settings gets: conjugate gradients preconditioned per group of key blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2510_01450_b200 import binding as L, inputs
from tests.gpu_util import dev, row_err, stream_ptr
from tests.test_parity_gpu import TOL_BF16

pytestmark = pytest.mark.gpu


def _case(d, n, nq, H, Hkv, spread, seed):
    w = inputs.CONFIGS[2].shrink(B=1, H=H, n=n, d=d, dv=d, seed=seed)
    q, _, _ = inputs.make_prefill(w)
    _, k, v = inputs.make_prefill(w.shrink(H=Hkv, seed=seed + 1))
    return w, inputs.round_to_bf16(q[:, :, n - nq:] * np.float32(spread)), k, v


@pytest.mark.parametrize("d,n,nq,H,Hkv,window,causal,spread", [
    (64, 97, 97, 2, 2, 0, True, 1.0),          # two rows beyond the directly solved ones
    (64, 129, 129, 2, 2, 0, True, 1.0),        # a second block of one key
    (128, 193, 193, 2, 2, 0, True, 1.0),
    (64, 2305, 2305, 1, 1, 0, True, 1.0),      # pairs of blocks share a matrix, the last group has one block of one key
    (128, 1177, 300, 4, 2, 0, True, 1.0),      # a chunk of queries: heads packed, pairs of thread blocks
    (64, 1000, 257, 4, 1, 0, True, 12.0),      # the same with sharply peaked weights
    (64, 1400, 1400, 2, 2, 333, True, 1.0),    # window
    (64, 700, 700, 2, 2, 0, False, 1.0),       # every row sees every key
])
def test_default_solver_against_explicit_solves(d, n, nq, H, Hkv, window, causal, spread):
    """Both solvers stop at a residual of 1e-4; the default one may not be further from the float64 solution than the plain
    one is, beyond the half that two stopping points below the same bound can differ by."""
    w, q, k, v = _case(d, n, nq, H, Hkv, spread, 700 + n)
    nbytes = L.lla_forward_workspace_bytes(1, H, n, d, d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    args = [dev(x, "bf16") for x in (q, k, v)]
    outs = []
    for kw in ({}, {"max_iters": 64}):
        out = torch.full((1, H, nq, d), float("nan"), dtype=torch.float32, device="cuda")
        status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
        L.lla_forward_ex(*args, out, 1, H, n, d, d, w.scale, w.lam, causal=causal, out_dtype=L.LLA_F32, q_rows=nq, kv_heads=Hkv,
                         window=window, device_status=status, workspace=ws, workspace_bytes=nbytes, stream=stream_ptr(), **kw)
        torch.cuda.synchronize()
        st = status.cpu().tolist()
        assert st[L.STATUS_TIMEOUT] == 0 and st[L.STATUS_ROWS_AT_CAP] == 0
        outs.append((out.cpu().numpy()[0].astype(np.float64), st[L.STATUS_ITER_SUM]))
    assert np.isfinite(outs[0][0]).all()
    rows = np.unique(np.concatenate([np.arange(0, nq, max(1, nq // 40)), [nq - 1]]))
    errs = [[], []]
    for h in range(H):
        K, V = k[0, h * Hkv // H].astype(np.float64), v[0, h * Hkv // H].astype(np.float64)
        for r in rows:
            c = n - nq + r + 1 if causal else n
            lo = max(0, c - window) if window else 0
            s = w.scale * K[lo:c] @ q[0, h, r].astype(np.float64)
            wt, z = np.exp(s - s.max()), K[lo:c] - q[0, h, r]
            rho = np.linalg.solve((wt[:, None] * z).T @ z + w.lam * np.exp(-s.max()) * np.eye(d), wt @ z)
            a = wt * (1 - z @ rho)
            ref = a @ V[lo:c] / a.sum()
            for e, (o, _) in zip(errs, outs):
                e.append(row_err(o[h, r], ref[None])[0])
    default, plain = (np.asarray(e) for e in errs)
    assert default.max() <= TOL_BF16
    assert np.sqrt(np.mean(default ** 2)) <= 1.5 * np.sqrt(np.mean(plain ** 2)) + 1e-6
    if spread == 1.0:
        assert outs[0][1] < outs[1][1]            # fewer iterations: it is the preconditioned solver that ran


def test_an_input_outside_the_fp16_range_turns_the_matrices_off():
    # an entry of k beyond 6e4, in a key that no row sees: the copies, and with them the preconditioner, are off on the
    # device, and what runs is the plain solver on operand pairs
    n, nq = 300, 100
    w, q, k, v = _case(64, n, nq, 1, 1, 1.0, 31)
    nbytes = L.lla_forward_workspace_bytes(1, 1, n, 64, 64)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    sums = []
    for entry in (1.0, 70000.0):
        k[0, 0, 7, 5] = entry
        out = torch.full((1, 1, nq, 64), float("nan"), dtype=torch.float32, device="cuda")
        status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
        L.lla_forward_ex(dev(q, "bf16"), dev(k, "bf16"), dev(v, "bf16"), out, 1, 1, n, 64, 64, w.scale, w.lam, out_dtype=L.LLA_F32,
                         q_rows=nq, window=150, device_status=status, workspace=ws, workspace_bytes=nbytes, stream=stream_ptr())
        torch.cuda.synchronize()
        sums.append((out.cpu().numpy(), status.cpu().tolist()[L.STATUS_ITER_SUM]))
    assert sums[0][1] < sums[1][1]
    assert row_err(sums[0][0], sums[1][0].astype(np.float64)).max() <= 4e-4      # two stopping points below 1e-4 each


def _solve(w, q, k, v, nq, Hkv, **kw):
    """Output (float64 numpy), iterations per row, rows at the cap; the cap as in a default call."""
    nbytes = L.lla_forward_workspace_bytes(1, w.H, w.n, w.d, w.d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    out = torch.full((1, w.H, nq, w.d), float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
    iters = torch.full((1, w.H, nq), -1, dtype=torch.int32, device="cuda")
    L.lla_forward_ex(dev(q, "bf16"), dev(k, "bf16"), dev(v, "bf16"), out, 1, w.H, w.n, w.d, w.d, w.scale, w.lam, out_dtype=L.LLA_F32,
                     q_rows=nq, kv_heads=Hkv, device_status=status, iters=iters, workspace=ws, workspace_bytes=nbytes, stream=stream_ptr(),
                     **{"max_iters": 64, **kw})
    torch.cuda.synchronize()
    st = status.cpu().tolist()
    assert st[L.STATUS_TIMEOUT] == 0
    return out.cpu().numpy()[0].astype(np.float64), iters.cpu().numpy()[0], st[L.STATUS_ROWS_AT_CAP]


def _exact(w, q, k, v, h, hk, rows, nq, window=0):
    ref = []
    K, V = k[0, hk].astype(np.float64), v[0, hk].astype(np.float64)
    for r in rows:
        c = w.n - nq + r + 1
        lo = max(0, c - window) if window else 0
        s = w.scale * K[lo:c] @ q[0, h, r].astype(np.float64)
        wt, z = np.exp(s - s.max()), K[lo:c] - q[0, h, r]
        rho = np.linalg.solve((wt[:, None] * z).T @ z + w.lam * np.exp(-s.max()) * np.eye(w.d), wt @ z)
        a = wt * (1 - z @ rho)
        ref.append(a @ V[lo:c] / a.sum())
    return np.asarray(ref)


@pytest.mark.parametrize("d,n,nq,H,Hkv,window,spread", [
    (64, 2637, 2637, 2, 2, 96, 1.0),       # the narrowest window: a tile's windows lie in two blocks of keys
    (64, 2500, 2500, 2, 2, 128, 1.0),
    (64, 2637, 1111, 4, 2, 160, 1.0),      # a chunk whose tiles do not start at a block of keys, grouped heads
    (128, 2500, 2500, 2, 2, 192, 1.0),
    (128, 2637, 2637, 2, 2, 256, 1.0),
    (128, 2637, 2637, 2, 2, 224, 8 * 2 ** 0.5),      # scores of unit variance
    (64, 2500, 2500, 2, 2, 333, 8.0),
    (64, 4900, 4900, 2, 2, 2100, 1.0),     # two tiles share a matrix past 2048 keys; the last one has its own
    (64, 4900, 2300, 4, 2, 2050, 1.0),
    (64, 2600, 700, 4, 2, 600, 1.0),       # grouped heads in common tiles: the matrix of the tile's middle row
    (64, 5000, 1300, 4, 2, 2100, 1.0),
])
def test_the_matrices_of_a_window_are_made_of_the_keys_that_its_rows_see(d, n, nq, H, Hkv, window, spread):
    """Past 2048 keys and below it: fewer iterations than plain conjugate gradients in the first and in the second tile of every
    256 rows, no more rows that run into the cap, and no larger error (two stopping points below one bound: half)."""
    w, q, k, v = _case(d, n, nq, H, Hkv, 1.0, 900 + n + window)
    s = np.float32(d ** 0.5 if spread > 1 else 1.0)      # (q and k ~ N(0, 1): q . k / sqrt(d) of unit variance)
    q, k = inputs.round_to_bf16(q * s), inputs.round_to_bf16(k * s)
    rows = np.unique(np.concatenate([np.linspace(max(0, d + d // 2 - (n - nq)), nq - 1, 30).astype(int), [nq - 129, nq - 1]]))
    got = [_solve(w, q, k, v, nq, Hkv, window=window, **kw) for kw in ({"cg_precondition": 1}, {})]
    ref = _exact(w, q, k, v, H - 1, Hkv - 1, rows, nq, window)
    rms = [np.sqrt(np.mean(row_err(o[H - 1, rows], ref) ** 2)) for o, _, _ in got]
    assert rms[0] <= 1.5 * rms[1] + 1e-6
    assert got[0][2] <= got[1][2]
    for part in (0, 1):
        its = [i[:, (np.arange(nq) // 128 % 2) == part] for _, i, _ in got]
        its = [i[i >= 0].mean() for i in its]
        assert its[0] < 0.9 * its[1], (part, its)


@pytest.mark.parametrize("d,n,rank,distinct", [(64, 1700, 32, 0), (64, 2500, 60, 0), (128, 2500, 124, 0), (128, 1300, 64, 0), (64, 1300, 64, 40)])
def test_keys_that_do_not_span_the_space(d, n, rank, distinct):
    """Keys (and queries) in a subspace, up to their rounding to bf16, or few different keys: an inverse covariance that is all
    ridge outside the subspace must not drown what it says inside.  Not more iterations than plain conjugate gradients,
    nor rows at the cap, nor a larger error."""
    H = 2
    w, q, k, v = _case(d, n, n, H, H, 1.0, 1200 + n + rank)
    rng = np.random.default_rng(7)
    basis = np.linalg.qr(rng.standard_normal((d, d)))[0][:, :rank]
    proj = (basis @ basis.T * (d / rank) ** 0.5).astype(np.float32)
    if distinct:
        k = k[:, :, rng.integers(0, distinct, n)]
    else:
        q, k = inputs.round_to_bf16(q @ proj), inputs.round_to_bf16(k @ proj)
    rows = np.linspace(d + d // 2, n - 1, 40).astype(int)
    got = [_solve(w, q, k, v, n, H, **kw) for kw in ({"cg_precondition": 1}, {})]
    ref = _exact(w, q, k, v, H - 1, H - 1, rows, n)
    rms = [np.sqrt(np.mean(row_err(o[H - 1, rows], ref) ** 2)) for o, _, _ in got]
    its = [i[i >= 0].mean() for _, i, _ in got]
    assert its[0] < its[1] and got[0][2] <= got[1][2], (its, got[0][2], got[1][2])
    assert rms[0] <= 1.5 * rms[1] + 1e-6, rms


@pytest.mark.parametrize("d,scale_k,n", [(64, 1e-3, 700), (64, 1e-2, 1500), (128, 1e-2, 1300)])
def test_solutions_beyond_the_fp16_range(d, scale_k, n):
    """Small keys under ordinary queries: the solution grows with the inverse of the ridge, beyond 65504, and the coefficients
    formed from it must not."""
    w, q, k, v = _case(d, n, n, 1, 1, 1.0, 1300 + n)
    k = inputs.round_to_bf16(k * np.float32(scale_k))
    rows = np.linspace(d + d // 2, n - 1, 30).astype(int)
    ref = _exact(w, q, k, v, 0, 0, rows, n)
    for kw in ({"max_iters": 0}, {}, {"cg_precondition": 1}):
        out, _, _ = _solve(w, q, k, v, n, 1, **kw)
        assert row_err(out[0, rows], ref).max() <= TOL_BF16, kw


@pytest.mark.parametrize("d,n,kw", [(64, 500, dict(head_rows=-1)), (128, 500, dict(head_rows=40)), (64, 2600, dict(head_rows=16, window=48)),
                                    (128, 700, dict(head_rows=-1, window=20))])
def test_rows_of_few_keys_run_plain_conjugate_gradients(d, n, kw):
    """With head_rows below 1.5 d the solver gets rows whose covariance is not the tile's: by default the call is plain, and where the
    preconditioner is asked for it leaves those rows alone."""
    w, q, k, v = _case(d, n, n, 2, 2, 1.0, 1400 + n)
    plain, default, asked = (_solve(w, q, k, v, n, 2, **s, **kw) for s in ({}, {"max_iters": 0}, {"cg_precondition": 1}))
    assert np.array_equal(plain[0], default[0], equal_nan=True)
    few = np.arange(n) + 1 < d + d // 2 if "window" not in kw else np.ones(n, dtype=bool)
    at_cap = [(r[1][:, few] >= 64).sum() for r in (plain, asked)]
    assert at_cap[1] <= 1.1 * at_cap[0] + 2, at_cap


@pytest.mark.parametrize("d,n,nq", [(64, 700, 700), (128, 900, 400)])
def test_asking_for_iteration_counts_changes_nothing(d, n, nq):
    """The same bits with and without `iters`, and counts that are those of the solver that ran."""
    w, q, k, v = _case(d, n, nq, 2, 2, 1.0, 1500 + n)
    args = [dev(x, "bf16") for x in (q, k, v)]
    nbytes = L.lla_forward_workspace_bytes(1, 2, n, d, d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    outs = []
    iters = torch.full((1, 2, nq), -1, dtype=torch.int32, device="cuda")
    for it in (None, iters):
        out = torch.full((1, 2, nq, d), float("nan"), dtype=torch.float32, device="cuda")
        status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
        L.lla_forward_ex(*args, out, 1, 2, n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32, q_rows=nq, device_status=status, iters=it,
                         workspace=ws, workspace_bytes=nbytes, stream=stream_ptr())
        torch.cuda.synchronize()
        outs.append((out, status.cpu().tolist()[L.STATUS_ITER_SUM]))
    assert torch.equal(outs[0][0], outs[1][0]) and outs[0][1] == outs[1][1]
    it = iters.cpu().numpy()
    assert it[it > 0].sum() == outs[1][1]


def test_a_block_mask_runs_plain_conjugate_gradients():
    """The matrices are those of all keys, a masked row sees some: by default the call is the plain one, bit for bit."""
    n, d = 1500, 64
    w, q, k, v = _case(d, n, n, 2, 2, 1.0, 1600)
    mask = (np.random.default_rng(3).random(((n + 127) // 128, (n + 63) // 64)) < 0.2).astype(np.uint8)
    m = torch.from_numpy(mask).cuda()
    plain, default = (_solve(w, q, k, v, n, 2, block_mask=m, **s) for s in ({}, {"max_iters": 0}))
    assert np.array_equal(plain[0], default[0]) and np.array_equal(plain[1], default[1])


@pytest.mark.parametrize("d,n,nq,window,unit", [(64, 500, 460, 0, False), (64, 500, 439, 0, False), (128, 700, 580, 0, False),
                                                (64, 1500, 1500, 120, False), (128, 1500, 1500, 250, False), (64, 500, 460, 0, True)])
def test_rows_of_few_keys_go_on_to_half_the_residual(d, n, nq, window, unit):
    """Whatever tile a row of at most 2 d keys falls into: in a chunk whose tiles start elsewhere, and under a window.  The residual
    is that of the saved solution, in float64: y = rho / (1 - b . rho) solves C y = b to half of 1e-4; nine rows in ten
    within another quarter of the tolerance for what rounding adds to the solver's own residual (operand pairs in every iteration:
    of the order of 1e-5)."""
    H = 4
    w, q, k, v = _case(d, n, nq, H, H, 1.0, 1700 + nq)
    if unit:      # scores of unit variance: weights far from uniform, such rows stop at the tolerance itself
        q, k = (inputs.round_to_bf16(x * np.float32(d ** 0.5)) for x in (q, k))
    seen = np.arange(n - nq, n) + 1
    seen = np.minimum(seen, window) if window else seen
    rows = np.flatnonzero((seen >= d + d // 2) & (seen <= 2 * d))
    rows = rows[:: max(1, len(rows) // 40)]
    rho = torch.zeros((1, H, nq, d), dtype=torch.float32, device="cuda")
    _solve(w, q, k, v, nq, H, window=window, cg_precondition=1, cg_precise_iters=64, rho=rho)
    rho = rho.cpu().numpy()[0].astype(np.float64)
    res = []
    for h in range(H):
        K = k[0, h].astype(np.float64)
        for r in rows:
            c = n - nq + r + 1
            kk = K[max(0, c - window) if window else 0:c]
            sc = w.scale * kk @ q[0, h, r].astype(np.float64)
            wt = np.exp(sc - sc.max())
            kb = wt @ kk / wt.sum()
            b = kb - q[0, h, r]
            y = rho[h, r] / (1 - b @ rho[h, r])
            cy = (wt * ((kk - kb) @ y)) @ (kk - kb) / wt.sum() + w.lam * np.exp(-sc.max()) / wt.sum() * y
            res.append(np.linalg.norm(b - cy) / np.linalg.norm(b))
    res = np.asarray(res)
    stop = 1e-4 if unit else 0.5e-4
    assert np.quantile(res, 0.5) <= stop and np.quantile(res, 0.9) <= stop + 0.25e-4, np.sort(res)[::8]
    assert not unit or np.quantile(res, 0.5) > 0.5e-4, np.sort(res)[::8]


@pytest.mark.parametrize("d,size_q,size_k", [(64, 1e-4, 1e-4), (128, 1e-4, 1e-4), (64, 1.0, 3e-4), (64, 3e-4, 1.0), (64, 1e-3, 1e-3),
                                              (64, 3e-5, 2.0), (128, 1e-4, 100.0), (64, 1e-3, 0.3)])
def test_small_inputs_keep_their_bits(d, size_q, size_k):
    """Entries of q and k far below the fp16 range's middle: rho against float64 within the tolerance, whatever the solver.  (In fp16
    an entry of 1e-5 is off by up to 0.3 %.)"""
    n = 600
    w, q, k, v = _case(d, n, n, 1, 1, 1.0, 1800 + d)
    q, k = inputs.round_to_bf16(q * np.float32(size_q)), inputs.round_to_bf16(k * np.float32(size_k))
    rows = np.linspace(d + d // 2, n - 1, 30).astype(int)
    for lam in (1e-3, 1e-2 * size_k ** 2):
        w = w.shrink(lam=lam)
        K = k[0, 0].astype(np.float64)
        for kw in ({"max_iters": 0}, {}):
            rho = torch.zeros((1, 1, n, d), dtype=torch.float32, device="cuda")
            _solve(w, q, k, v, n, 1, rho=rho, **kw)
            for r in rows:
                z = K[:r + 1] - q[0, 0, r]
                s = w.scale * K[:r + 1] @ q[0, 0, r].astype(np.float64)
                wt = np.exp(s - s.max())
                ref = np.linalg.solve((wt[:, None] * z).T @ z + lam * np.exp(-s.max()) * np.eye(d), wt @ z)
                assert np.linalg.norm(rho[0, 0, r].cpu().numpy() - ref) <= 4e-4 * np.linalg.norm(ref), (lam, kw, r)


@pytest.mark.parametrize("d,n", [(64, 2500), (128, 2500)])
def test_many_keys_of_small_weight(d, n):
    """Eight keys of weight 2^-7.7 and thousands of about 2^-20, none larger (the weights are taken in the frame of a zero score where the
    largest lies within 2^+-8): in fp16 the small ones are multiples of 2^-24.  The queries lie far from the keys, which makes the
    systems sensitive to them; no larger an error than with bf16 operand pairs, whose bits are relative, and a quarter."""
    w, q, k, v = _case(d, n, n, 1, 1, 1.0, 1900 + d)
    rng = np.random.default_rng(11)
    u = np.zeros(d, dtype=np.float32)
    u[: d // 2] = (2.0 / d) ** 0.5
    away = rng.standard_normal((n, d)) * 0.5
    away -= np.outer(away @ u, u)
    k = (away + np.outer(-13.9 / 6 + 0.05 * rng.standard_normal(n), u)).astype(np.float32)
    k[:8] += (13.9 - 5.3) / 6 * u
    q = np.broadcast_to(6 * d ** 0.5 * u, (n, d)) + 0.1 * rng.standard_normal((n, d)).astype(np.float32)
    q, k = (inputs.round_to_bf16(x[None, None].astype(np.float32)) for x in (q, k))
    rows = np.linspace(d + d // 2, n - 1, 40).astype(int)
    ref = _exact(w, q, k, v, 0, 0, rows, n)
    rms = []
    for kw in ({"cg_precise_iters": L.LLA_CG_PRECISE_ALL}, {}, {"max_iters": 0}):
        out, _, _ = _solve(w, q, k, v, n, 1, **kw)
        rms.append(np.sqrt(np.mean(row_err(out[0, rows], ref) ** 2)))
    assert max(rms[1:]) <= 1.25 * rms[0], rms


@pytest.mark.parametrize("d,B,n,nq,H,Hkv", [(64, 1, 300, 300, 4, 1), (128, 2, 4500, 1300, 4, 1), (64, 1, 5000, 1257, 8, 2), (128, 1, 700, 129, 2, 2)])
def test_the_pre_pass_reads_any_layout_of_q_and_any_number_of_heads(d, B, n, nq, H, Hkv):
    """Few key/value heads cut their keys into more chunks (one block of keys a chunk, two and more; 4500 keys: a last chunk of one
    block), and q is looked at a tile of rows at a time: the same output bits for [B, H, nq, d] and [B, nq, H, d], and one entry
    beyond the fp16 range in the last row of the last head turns the fp16 sweeps off either way."""
    w = inputs.CONFIGS[2].shrink(B=B, H=H, n=n, d=d, dv=d, seed=2000 + n)
    q, _, _ = inputs.make_prefill(w)
    _, k, v = inputs.make_prefill(w.shrink(H=Hkv, seed=2001 + n))
    q = np.ascontiguousarray(q[:, :, n - nq:])
    nbytes = L.lla_forward_workspace_bytes(B, H, n, d, d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    kd, vd = dev(k, "bf16"), dev(v, "bf16")
    sums = []
    for big in (False, True):
        if big:
            q[-1, -1, -1, -1] = 65536.0
        outs = []
        for strided in (False, True):
            qd = dev(np.ascontiguousarray(q.transpose(0, 2, 1, 3)) if strided else q, "bf16")
            out = torch.full((B, H, nq, d), float("nan"), dtype=torch.float32, device="cuda")
            status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
            L.lla_forward_ex(qd, kd, vd, out, B, H, n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32, q_rows=nq, kv_heads=Hkv,
                             q_strides=(nq * H * d, d, H * d) if strided else None, device_status=status, workspace=ws,
                             workspace_bytes=nbytes, cg_precondition=1, stream=stream_ptr())
            torch.cuda.synchronize()
            outs.append(out[:, :, :-1])
            sums.append(status.cpu().tolist()[L.STATUS_ITER_SUM])
        assert torch.isfinite(outs[0]).all()
        # (packed rows of grouped heads need q in one piece; unpacked tiles end where other rows are)
        assert row_err(outs[0].cpu().numpy(), outs[1].cpu().numpy().astype(np.float64)).max() <= 4e-4
    assert max(sums[:2]) < min(sums[2:])
    for h in (0, H - 1):
        rows = np.linspace(max(0, d + d // 2 - (n - nq)), nq - 2, 12).astype(int)
        ref = _exact(w, q[-1:], k[-1:], v[-1:], h, h * Hkv // H, rows, nq)
        assert row_err(outs[0][-1, h].cpu().numpy()[rows], ref).max() <= TOL_BF16


@pytest.mark.parametrize("d,n,nq", [(64, 700, 700), (128, 1000, 300)])
def test_a_preconditioned_block_whose_waits_run_out_leaves_cleanly(d, n, nq):
    """No copy is issued, the matrix's neither, so every wait expires; the blocks leave, are counted, and the next call is right."""
    w, q, k, v = _case(d, n, nq, 2, 2, 1.0, 2100 + n)
    args = [dev(x, "bf16") for x in (q, k, v)]
    nbytes = L.lla_forward_workspace_bytes(1, 2, n, d, d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")

    def run(**kw):
        out = torch.full((1, 2, nq, d), float("nan"), dtype=torch.float32, device="cuda")
        status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
        L.lla_forward_ex(*args, out, 1, 2, n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32, q_rows=nq, device_status=status, workspace=ws,
                         workspace_bytes=nbytes, cg_precondition=1, stream=stream_ptr(), **kw)
        torch.cuda.synchronize()
        return out, status.cpu().tolist()

    good, st = run()
    assert st[L.STATUS_TIMEOUT] == 0 and torch.isfinite(good).all()
    _, st = run(debug_wait_clocks=1 << 20, debug_flags=L.LLA_DEBUG_NO_LOADS)
    assert st[L.STATUS_TIMEOUT] > 0
    again, st = run()
    assert st[L.STATUS_TIMEOUT] == 0 and torch.equal(good, again)
