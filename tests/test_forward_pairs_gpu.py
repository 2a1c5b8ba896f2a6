"""The tensor-core forward on grids that leave SMs idle: pairs of blocks per query tile (each sweeps half of the keys), and
the rows of grouped heads cut into tiles together.  Every sampled row is checked against the oracle's single-query routine
over exactly its visible keys; tolerance as in the other bf16 parity tests on an fp32 output buffer."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2510_01450_b200 import binding as L, inputs
from tests.gpu_util import dev, row_err, stream_ptr
from tests.test_parity_gpu import TOL_BF16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver", [{}, {"max_iters": 64}, {"cg_precondition": 1}], ids=["default", "plain", "preconditioned"])
@pytest.mark.parametrize("d,H,Hkv,n,nq,window,causal", [
    (64, 4, 4, 900, 300, 0, True),         # pairs, a ragged last tile
    (64, 8, 2, 700, 129, 0, True),         # packed rows of four heads: tiles that run over a head's end; pairs
    (128, 8, 2, 1000, 200, 0, True),
    (128, 4, 1, 1500, 257, 700, True),     # packed, window: a tile's first block comes from the next head's first row
    (64, 2, 2, 1000, 1000, 0, False),      # non-causal pairs
    (128, 6, 3, 600, 1, 0, True),          # one query per head: two rows in a tile
    (64, 16, 4, 2000, 700, 0, True),       # packed tiles, more of them than half the SMs
])
def test_pairs_and_packed_rows(oracle, d, H, Hkv, n, nq, window, causal, solver):
    B = 2
    w = inputs.CONFIGS[2].shrink(B=B, H=H, n=n, d=d, dv=d, seed=500 + d + n)
    q, _, _ = inputs.make_prefill(w)
    _, k, v = inputs.make_prefill(w.shrink(H=Hkv, seed=501 + n))
    qc = np.ascontiguousarray(q[:, :, n - nq:]) * np.float32(2.0)          # (exact in bf16; weights further from uniform)
    out = torch.full((B, H, nq, d), float("nan"), dtype=torch.float32, device="cuda")
    rho, stats = torch.empty_like(out), torch.empty((B, H, nq, 3), dtype=torch.float32, device="cuda")
    iters = torch.full((B, H, nq), -7, dtype=torch.int32, device="cuda")
    status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
    nbytes = L.lla_forward_workspace_bytes(B, H, n, d, d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        L.lla_forward_ex(dev(qc, "bf16"), dev(k, "bf16"), dev(v, "bf16"), out, B, H, n, d, d, w.scale, w.lam, causal=causal,
                         out_dtype=L.LLA_F32, q_rows=nq, kv_heads=Hkv, window=window, rho=rho, stats=stats, iters=iters,
                         device_status=status, workspace=ws, workspace_bytes=nbytes, stream=stream_ptr(), **solver)
    torch.cuda.synchronize()
    assert status.cpu().numpy()[L.STATUS_TIMEOUT] == 0
    assert (iters.cpu().numpy() >= -1).all()
    got = out.cpu().numpy().astype(np.float64)
    rows = np.unique(np.concatenate([np.arange(min(nq, 12)), np.random.default_rng(3).integers(0, nq, 40), [nq - 1]]))
    lo = [max(0, n - nq + r + 1 - window) if causal and window else 0 for r in rows]
    cnt = np.array([(n - nq + r + 1 if causal else n) - l for r, l in zip(rows, lo)], dtype=np.int32)
    kk, vv = np.repeat(k, H // Hkv, axis=1), np.repeat(v, H // Hkv, axis=1)
    for b in range(B):
        kc = np.zeros((len(rows), H, cnt.max(), d), dtype=np.float32)
        vc = np.zeros_like(kc)
        for s, (l, c) in enumerate(zip(lo, cnt)):
            kc[s, :, :c], vc[s, :, :c] = kk[b, :, l:l + c], vv[b, :, l:l + c]
        ref = oracle.decode(np.ascontiguousarray(qc[b][:, rows].transpose(1, 0, 2)), kc, vc, cnt, w.scale, w.lam)
        err = row_err(got[b][:, rows].transpose(1, 0, 2), ref)
        assert np.isfinite(err).all() and err.max() <= TOL_BF16, (b, float(err.max()), int(err.argmax()))
    # o = sum_j w_j (1 - z_j . rho) v_j / delta with the saved tensors, for one row of the last head
    r = int(rows[len(rows) // 2])
    l, c = lo[len(rows) // 2], int(cnt[len(rows) // 2])
    qr, kr, vr = qc[1, -1, r].astype(np.float64), kk[1, -1, l:l + c].astype(np.float64), vv[1, -1, l:l + c].astype(np.float64)
    m, om, dl = stats.cpu().numpy()[1, -1, r].astype(np.float64)
    wt = np.exp(w.scale * kr @ qr - m)
    assert abs(wt.sum() / om - 1) < 1e-4
    o = (wt * (1 - (kr - qr) @ rho.cpu().numpy()[1, -1, r])) @ vr / dl
    assert np.linalg.norm(o - got[1, -1, r]) <= 2e-3 * np.linalg.norm(o)


def test_a_pair_whose_waits_run_out_leaves_cleanly():
    """No copy is issued, so every wait expires; both blocks of every pair leave, are counted, and the next call is right."""
    B, H, n, d, nq = 1, 2, 1200, 64, 256
    w = inputs.CONFIGS[2].shrink(B=B, H=H, n=n, d=d, dv=d, seed=520)
    q, k, v = inputs.make_prefill(w)
    args = [dev(np.ascontiguousarray(q[:, :, n - nq:]), "bf16"), dev(k, "bf16"), dev(v, "bf16")]

    def run(**kw):
        out = torch.full((B, H, nq, d), float("nan"), dtype=torch.float32, device="cuda")
        status = torch.zeros(L.LLA_STATUS_WORDS, dtype=torch.int32, device="cuda")
        L.lla_forward_ex(*args, out, B, H, n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32, q_rows=nq, device_status=status,
                         stream=stream_ptr(), **kw)
        torch.cuda.synchronize()
        return out.cpu().numpy(), status.cpu().numpy()

    good, st = run()
    assert st[L.STATUS_TIMEOUT] == 0 and np.isfinite(good).all()
    _, st = run(debug_wait_clocks=1 << 20, debug_flags=L.LLA_DEBUG_NO_LOADS)
    assert st[L.STATUS_TIMEOUT] == 2 * B * H * (nq // 128)
    again, st = run()
    assert st[L.STATUS_TIMEOUT] == 0 and np.array_equal(good, again)


@pytest.mark.parametrize("d,H,n,nq", [(64, 4, 3000, 500), (128, 4, 2500, 400)])
def test_pairs_repeat_exactly(d, H, n, nq):
    """The two blocks of a pair leave their sums in each other's operand tiles; who reads and who overwrites them when must
    not show: every run gives the same bits (weights far from uniform, so that the rows take many iterations)."""
    w = inputs.CONFIGS[2].shrink(B=1, H=H, n=n, d=d, dv=d, seed=540 + d)
    q, k, v = inputs.make_prefill(w)
    s = np.float32(d ** 0.5)
    args = [dev(inputs.round_to_bf16(x), "bf16") for x in (np.ascontiguousarray(q[:, :, n - nq:]) * s, k * s, v)]
    nbytes = L.lla_forward_workspace_bytes(1, H, n, d, d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    first = None
    for _ in range(25):
        out = torch.full((1, H, nq, d), float("nan"), dtype=torch.float32, device="cuda")
        L.lla_forward_ex(*args, out, 1, H, n, d, d, w.scale, w.lam, out_dtype=L.LLA_F32, q_rows=nq, workspace=ws,
                         workspace_bytes=nbytes, stream=stream_ptr())
        assert torch.isfinite(out).all()
        first = out if first is None else first
        assert torch.equal(out, first)


@pytest.mark.parametrize("d,n,nq", [(64, 700, 600), (128, 1100, 908), (64, 560, 463)])
def test_packed_heads_keep_the_early_rows_precision(d, n, nq):
    """Rows of grouped heads cut into tiles together: the first rows of every head, which converge slowly, get as many
    iterations with operand pairs as the same rows of heads that are not grouped.  Their errors against the explicit
    solve may differ by how the other rows of the tile steer its iterations, not by the coarser operands' factor of two."""
    B, H, Hkv, rows = 1, 8, 2, 48
    w = inputs.CONFIGS[2].shrink(B=B, H=H, n=n, d=d, dv=d, seed=560 + n)
    q, _, _ = inputs.make_prefill(w)
    _, k, v = inputs.make_prefill(w.shrink(H=Hkv, seed=561 + n))
    kk, vv = np.repeat(k, H // Hkv, axis=1), np.repeat(v, H // Hkv, axis=1)
    qc = np.ascontiguousarray(q[:, :, n - nq:])
    nbytes = L.lla_forward_workspace_bytes(B, H, n, d, d)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    got = []
    for kx, vx, hkv in ((k, v, Hkv), (kk, vv, H)):
        out = torch.full((B, H, nq, d), float("nan"), dtype=torch.float32, device="cuda")
        L.lla_forward_ex(dev(qc, "bf16"), dev(kx, "bf16"), dev(vx, "bf16"), out, B, H, n, d, d, w.scale, w.lam,
                         out_dtype=L.LLA_F32, q_rows=nq, kv_heads=hkv, workspace=ws, workspace_bytes=nbytes, stream=stream_ptr())
        torch.cuda.synchronize()
        got.append(out.cpu().numpy()[0, :, :rows].astype(np.float64))
    errs = [[], []]
    for h in range(H):
        K, V = kk[0, h].astype(np.float64), vv[0, h].astype(np.float64)
        for r in range(rows):
            c = n - nq + r + 1
            s = w.scale * K[:c] @ qc[0, h, r].astype(np.float64)
            wt, z = np.exp(s - s.max()), K[:c] - qc[0, h, r]
            rho = np.linalg.solve((wt[:, None] * z).T @ z + w.lam * np.exp(-s.max()) * np.eye(d), wt @ z)
            a = wt * (1 - z @ rho)
            ref = a @ V[:c] / a.sum()
            for e, g in zip(errs, got):
                e.append(np.linalg.norm(g[h, r] - ref) / np.linalg.norm(ref))
    packed, alone = (np.sqrt(np.mean(np.square(e))) for e in errs)
    assert packed <= 1.25 * alone, (packed, alone)
