"""GPU parity, kernel by kernel, through the C ABI against the CPU oracle on the same seeded inputs.

Bars: kept masks, T_nbr / T_worker / T_round, b and theta are bit-exact (only comparisons touch
the times); parameters after the fp32 mix agree to 1e-5 per row (max-norm relative), which
leaves two orders of magnitude over the fp32 rounding of a <= 40-term weighted sum.
"""
import numpy as np
import pytest

from oracle import dbw_oracle as orc
from workloads import configs as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _dbw():
    import paper_2102_06280_b200 as p
    return p


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def row_rel_err(got, ref):
    got = np.asarray(got, dtype=np.float64)
    num = np.abs(got - ref).max(axis=1)
    den = np.maximum(np.abs(ref).max(axis=1), 1e-30)
    return float((num / den).max())


GRAPHS = {
    "ring8": lambda: wl.ring(8),
    "path2": lambda: wl.path(2),
    "complete40": lambda: wl.complete(40),          # degree 39 > one warp
    "complete70": lambda: wl.complete(70),          # degree 69: three 32-neighbour chunks
    "reg4_32": lambda: wl.random_regular(32, 4, 2),
    "er64": lambda: wl.erdos_renyi_connected(64, 0.2, 3),
    "reg32_256": lambda: wl.random_regular(256, 32, 11),
    "star_like": lambda: wl._csr_from_edges(6, [(0, 1), (0, 2), (0, 3), (0, 4), (0, 5)]),  # degree-1 leaves
}


def _select_gpu(h, n, nnz, t, b):
    kept = torch.zeros(nnz, dtype=torch.uint8, device="cuda")
    Tw = torch.zeros(n, dtype=torch.float64, device="cuda")
    Tn = torch.zeros(n, dtype=torch.float64, device="cuda")
    Tr = torch.zeros(1, dtype=torch.float64, device="cuda")
    h.select(dev(t), dev(b.astype(np.int32)), kept, Tw, Tn, Tr)
    torch.cuda.synchronize()
    return kept.cpu().numpy(), Tw.cpu().numpy(), Tn.cpu().numpy(), float(Tr.cpu()[0])


@pytest.mark.parametrize("name", list(GRAPHS))
def test_selection_bit_exact(name):
    p = _dbw()
    rowptr, col = GRAPHS[name]()
    n = len(rowptr) - 1
    deg = np.diff(rowptr)
    h = p.Dbw(rowptr, col, d=4)
    rng = np.random.default_rng(5)
    cases = []
    for trial in range(6):
        t = 1.0 + rng.exponential(1.0, size=n)
        if trial % 2:                                  # engineered ties
            t = np.round(t * 2) / 2
        cases.append((t, rng.integers(0, deg + 1)))
    cases.append((1.0 + rng.exponential(1.0, size=n), np.zeros(n, dtype=np.int64)))   # b = 0
    cases.append((1.0 + rng.exponential(1.0, size=n), deg.copy()))                     # b = deg
    cases.append((np.ones(n), rng.integers(0, deg + 1)))                               # all times equal
    for t, b in cases:
        kept, Tw, Tn, Tr = _select_gpu(h, n, len(col), t, b)
        ref = orc.select_fastest(rowptr, col, t, b)
        assert np.array_equal(kept, ref)
        rTn, rTw, rTr = orc.round_times(rowptr, col, t, b, ref)
        assert np.array_equal(Tn, rTn) and np.array_equal(Tw, rTw) and Tr == rTr
    assert h.status() == 0
    h.close()


def test_selection_flags_bad_inputs():
    p = _dbw()
    rowptr, col = wl.ring(8)
    h = p.Dbw(rowptr, col, d=4)
    t = np.arange(8, dtype=np.float64)
    b = np.array([0, 5, 0, -2, 0, 0, 0, 0])
    kept, *_ = _select_gpu(h, 8, len(col), t, b)
    assert h.status() & p.STATUS_BAD_B
    ref = orc.select_fastest(rowptr, col, t, np.clip(b, 0, 2))      # clamped, not trapped
    assert np.array_equal(kept, ref)
    t[3] = np.nan
    kept, *_ = _select_gpu(h, 8, len(col), t, np.ones(8, dtype=np.int64))
    assert h.status() & p.STATUS_NAN_TIME
    t[3] = np.inf                                                    # NaN is ordered last
    assert np.array_equal(kept, orc.select_fastest(rowptr, col, t, np.ones(8, dtype=np.int64)))
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("name,d", [("ring8", 7850), ("reg4_32", 1000), ("er64", 4100), ("complete40", 260),
                                     ("reg32_256", 3000)])
@pytest.mark.parametrize("rule", ["metropolis", "uniform"])
@pytest.mark.parametrize("order", ["local_then_mix", "mix_then_correct"])
def test_mix_matches_oracle(name, d, rule, order):
    p = _dbw()
    rowptr, col = GRAPHS[name]()
    n = len(rowptr) - 1
    deg = np.diff(rowptr)
    ld = (d + 3) // 4 * 4
    flags = (p.WEIGHT_UNIFORM if rule == "uniform" else 0) | (p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    h = p.Dbw(rowptr, col, d=d, ld=ld, flags=flags)
    rng = np.random.default_rng(8)
    X = np.zeros((n, ld), dtype=np.float32)
    G = np.zeros((n, ld), dtype=np.float32)
    X[:, :d] = rng.standard_normal((n, d), dtype=np.float32)
    G[:, :d] = rng.standard_normal((n, d), dtype=np.float32)
    t = 1.0 + rng.exponential(1.0, size=n)
    b = rng.integers(0, deg + 1)
    b[0] = deg[0]                                         # one worker waits for nobody
    kept = orc.select_fastest(rowptr, col, t, b)
    ws, we = orc.mixing_weights(rowptr, col, b, kept, rule)
    ref = orc.mix_update(rowptr, col, X, G, ws, we, 0.05, order)
    Xd, Gd, kd, bd = dev(X), dev(G), dev(kept), dev(b.astype(np.int32))
    for panel in (0, 1, 2, 16, 32, 64, 128, 256, -1):
        h.set_mix_panel(panel)
        out = torch.full_like(Xd, float("nan"))
        h.mix(Xd, Gd, kd, bd, 0.05, out)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        assert row_rel_err(got, ref) <= 1e-5, panel
        assert not np.any(got[:, d:])                      # padding stays zero
        if panel != -1 and h.mix_in_place_ok():
            inpl = Xd.clone()
            h.mix(inpl, Gd, kd, bd, 0.05, inpl)
            torch.cuda.synchronize()
            assert np.array_equal(inpl.cpu().numpy(), got)  # in place == out of place, bit for bit
    # per-worker learning rates (eta_j of Eq. 4)
    lrw = (0.01 + 0.1 * rng.random(n)).astype(np.float32)
    h.set_mix_panel(0)
    out = torch.empty_like(Xd)
    h.mix(Xd, Gd, kd, bd, 0.0, out, lr_per_worker=dev(lrw))
    torch.cuda.synchronize()
    ref = orc.mix_update(rowptr, col, X, G, ws, we, lrw.astype(np.float64), order)
    assert row_rel_err(out.cpu().numpy(), ref) <= 1e-5
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("n,deg,d,order", [(320, 16, 1000, "local_then_mix"), (700, 16, 1300, "mix_then_correct"),
                                           (1000, 32, 2052, "local_then_mix"), (512, 8, 516, "local_then_mix"),
                                           (514, 8, 260, "mix_then_correct")])
@pytest.mark.parametrize("panel,kernel", [(2, "mix_tc_kernel"), (3, "mix_sp_kernel")])
def test_mix_tensor_core_kernel_matches_oracle(n, deg, d, order, panel, kernel):
    """The 0/1-selection product on the tensor cores (three exact BF16 pieces per fp32 value), dense and with the
    selection matrix 2:4 structured-sparse in the graph's worker order: worker counts that leave ragged row tiles
    and K chunks, widths that leave a ragged last panel, both update orders, per-worker learning rates, in place
    where one CTA pair owns a panel, run-to-run reproducible."""
    p = _dbw()
    rowptr, col = wl.random_regular(n, deg, 21)
    degs = np.diff(rowptr)
    flags = p.WEIGHT_UNIFORM | (p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    h = p.Dbw(rowptr, col, d=d, ld=d, flags=flags)
    h.set_mix_panel(panel)
    assert h.mix_kernel() == kernel
    assert h.mix_in_place_ok() == (n <= 512)
    rng = np.random.default_rng(12)
    X = rng.standard_normal((n, d), dtype=np.float32) * np.float32(3.0)
    X[:, ::7] *= np.float32(1e-4)                          # small and large magnitudes side by side
    G = rng.standard_normal((n, d), dtype=np.float32)
    t = 1.0 + rng.exponential(1.0, size=n)
    b = rng.integers(0, np.minimum(degs, 8) + 1)
    b[0] = degs[0]
    kept = orc.select_fastest(rowptr, col, t, b)
    ws, we = orc.mixing_weights(rowptr, col, b, kept, "uniform")
    lrw = (0.01 + 0.1 * rng.random(n)).astype(np.float32)
    Xd, Gd, kd, bd = dev(X), dev(G), dev(kept), dev(b.astype(np.int32))
    for lr, lr_pw in ((0.05, None), (0.0, lrw)):
        ref = orc.mix_update(rowptr, col, X, G, ws, we, lr if lr_pw is None else lr_pw.astype(np.float64), order)
        out = torch.full_like(Xd, float("nan"))
        h.mix(Xd, Gd, kd, bd, lr, out, lr_per_worker=None if lr_pw is None else dev(lr_pw))
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        assert row_rel_err(got, ref) <= 1e-5
        for _ in range(3):                                   # reproducible: staging buffers are reused between stores
            again = torch.zeros_like(Xd)
            h.mix(Xd, Gd, kd, bd, lr, again, lr_per_worker=None if lr_pw is None else dev(lr_pw))
            torch.cuda.synchronize()
            assert np.array_equal(again.cpu().numpy(), got)
        if h.mix_in_place_ok():
            inpl = Xd.clone()
            h.mix(inpl, Gd, kd, bd, lr, inpl, lr_per_worker=None if lr_pw is None else dev(lr_pw))
            torch.cuda.synchronize()
            assert np.array_equal(inpl.cpu().numpy(), got)
        else:
            with pytest.raises(p.DbwError):
                h.mix(Xd, Gd, kd, bd, lr, Xd)
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("order", ["local_then_mix", "mix_then_correct"])
def test_mix_staged_kernel_with_metropolis_weights(order):
    """The paper's weight rule (Assumption 1) on a graph with many kept neighbours per worker: the persistent
    tensor-memory staged kernel is selected by itself, carries the weights as 6-bit codes in its neighbour lists,
    and adds in the same order as the shared-memory panel kernel: same bits, same bar against the oracle."""
    p = _dbw()
    n, deg, d = 1000, 32, 2052
    rowptr, col = wl.random_regular(n, deg, 7)
    degs = np.diff(rowptr)
    h = p.Dbw(rowptr, col, d=d, ld=d, flags=p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    assert h.mix_kernel() == "mix_staged_kernel" and h.mix_in_place_ok()
    rng = np.random.default_rng(2)
    X = rng.standard_normal((n, d), dtype=np.float32)
    G = rng.standard_normal((n, d), dtype=np.float32)
    t = 1.0 + rng.exponential(1.0, size=n)
    b = rng.integers(0, np.minimum(degs, 9) + 1)
    b[0], b[1] = degs[0], 0
    kept = orc.select_fastest(rowptr, col, t, b)
    ws, we = orc.mixing_weights(rowptr, col, b, kept, "metropolis")
    ref = orc.mix_update(rowptr, col, X, G, ws, we, 0.05, order)
    Xd, Gd, kd, bd = dev(X), dev(G), dev(kept), dev(b.astype(np.int32))
    res = {}
    for panel in (0, 16):
        h.set_mix_panel(panel)
        out = torch.full_like(Xd, float("nan"))
        h.mix(Xd, Gd, kd, bd, 0.05, out)
        torch.cuda.synchronize()
        res[panel] = out.cpu().numpy()
        assert row_rel_err(res[panel], ref) <= 1e-5, panel
    assert h.mix_kernel() == "mix_panel_kernel"
    assert np.array_equal(res[0], res[16])
    h.set_mix_panel(0)
    inpl = Xd.clone()
    h.mix(inpl, Gd, kd, bd, 0.05, inpl)
    torch.cuda.synchronize()
    assert np.array_equal(inpl.cpu().numpy(), res[0])
    assert h.status() == 0
    h.close()


def test_mix_large_worker_count_uses_the_l2_kernel():
    """More workers than a shared-memory panel of even 16 columns can hold: neighbour rows are re-read through L2
    (row-fastest work order inside column panels), out of place only, same bar."""
    p = _dbw()
    n, d = 4200, 1100
    rowptr, col = wl.random_regular(n, 4, 5)
    deg = np.diff(rowptr)
    for rule, order in (("metropolis", "local_then_mix"), ("uniform", "mix_then_correct")):
        flags = (p.WEIGHT_UNIFORM if rule == "uniform" else 0) | (p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
        h = p.Dbw(rowptr, col, d=d, ld=d, flags=flags)
        assert h.mix_kernel() == "mix_direct_kernel" and not h.mix_in_place_ok()
        rng = np.random.default_rng(3)
        X = rng.standard_normal((n, d), dtype=np.float32)
        G = rng.standard_normal((n, d), dtype=np.float32)
        t = 1.0 + rng.exponential(1.0, size=n)
        b = rng.integers(0, deg + 1)
        kept = orc.select_fastest(rowptr, col, t, b)
        ws, we = orc.mixing_weights(rowptr, col, b, kept, rule)
        ref = orc.mix_update(rowptr, col, X, G, ws, we, 0.05, order)
        Xd = dev(X)
        out = torch.full_like(Xd, float("nan"))
        h.mix(Xd, dev(G), dev(kept), dev(b.astype(np.int32)), 0.05, out)
        torch.cuda.synchronize()
        assert row_rel_err(out.cpu().numpy(), ref) <= 1e-5
        with pytest.raises(p.DbwError):
            h.mix(Xd, dev(G), dev(kept), dev(b.astype(np.int32)), 0.05, Xd)
        assert h.status() == 0
        h.close()


def test_mix_rejects_bad_aliasing():
    p = _dbw()
    rowptr, col = wl.ring(8)
    h = p.Dbw(rowptr, col, d=64)
    X = torch.zeros(8 * 64 + 64, device="cuda")
    G = torch.zeros(8 * 64, device="cuda")
    kept = torch.ones(16, dtype=torch.uint8, device="cuda")
    b = torch.zeros(8, dtype=torch.int32, device="cuda")
    with pytest.raises(p.DbwError):
        h.mix(X[:512], G, kept, b, 0.1, X[32:544])          # partial overlap
    with pytest.raises(p.DbwError):
        h.mix(X[:512], G, kept, b, 0.1, G)                  # output over the gradients
    h.set_mix_panel(-1)
    with pytest.raises(p.DbwError):
        h.mix(X[:512], G, kept, b, 0.1, X[:512])            # direct kernel cannot run in place
    h.close()


@pytest.mark.parametrize("name", ["ring8", "reg4_32", "er64", "complete40"])
def test_update_backups_bit_exact_and_resume(name):
    p = _dbw()
    rowptr, col = GRAPHS[name]()
    n = len(rowptr) - 1
    h = p.Dbw(rowptr, col, d=4)
    assert np.array_equal(h.links(), np.array(orc.spanning_links(rowptr, col)))
    ref = orc.Dtur(rowptr, col)
    rng = np.random.default_rng(3)
    b_d = torch.zeros(n, dtype=torch.int32, device="cuda")
    th_d = torch.zeros(1, dtype=torch.float64, device="cuda")
    rounds = 2 * (n - 1) + 3
    times = 1.0 + rng.exponential(1.0, size=(rounds, n))
    times[1] = np.round(times[1])                            # ties between links
    blob = None
    for k in range(rounds):
        if k == n // 2:
            blob = h.state_export()
            saved = (list(ref.covered), ref.step)
        h.update_backups(dev(times[k]), b_d, th_d)
        torch.cuda.synchronize()
        rb, rtheta = ref.update_backups(times[k])
        assert np.array_equal(b_d.cpu().numpy(), rb) and float(th_d.cpu()[0]) == rtheta
    # resume from the saved state reproduces the same sequence
    h.state_import(blob)
    ref.covered, ref.step = saved
    for k in range(n // 2, n // 2 + 5):
        h.update_backups(dev(times[k]), b_d, th_d)
        rb, rtheta = ref.update_backups(times[k])
        assert np.array_equal(b_d.cpu().numpy(), rb) and float(th_d.cpu()[0]) == rtheta
    h.reset_backups()
    fresh = orc.Dtur(rowptr, col)
    h.update_backups(dev(times[0]), b_d, th_d)
    assert np.array_equal(b_d.cpu().numpy(), fresh.update_backups(times[0])[0])
    with pytest.raises(p.DbwError):
        h.state_import(blob[:-4])
    h.close()


@pytest.mark.parametrize("dims,batch,n", [([784, 10], 32, 8), ([20, 13, 7], 5, 3), ([100, 70, 33, 10], 19, 4),
                                           ([784, 200, 10], 64, 6),
                                           ([64, 48, 24], 12, 3),     # 24 classes: the 32-class instance of the last-layer kernels
                                           ([256, 128], 40, 3),       # one layer of more than 32 classes: GEMM + loss kernel
                                           ([8, 5, 8, 4], 6, 3),      # last layer's weights not 16-byte aligned in the row: GEMM path
                                           ([128, 64, 64, 12], 256, 5)])  # whole tiles of the 128-bit GEMM, 8 x 4 outputs per thread
def test_grad_fp32_matches_oracle(dims, batch, n):
    p = _dbw()
    rowptr, col = wl.ring(max(n, 3)) if n >= 3 else wl.path(n)
    n = len(rowptr) - 1
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m)
    rng = np.random.default_rng(0)
    S = 3 * batch
    feat = rng.random((n, S, dims[0]), dtype=np.float32)
    labels = rng.integers(0, dims[-1], size=(n, S)).astype(np.int32)
    Xl = (rng.standard_normal((n, m.d)) * 0.2).astype(np.float32)
    idx = np.stack([rng.permutation(S)[:batch] for _ in range(n)]).astype(np.int32)
    h.set_dataset(dev(feat), dev(labels), S)
    G = torch.zeros(n, m.ld, device="cuda")
    loss = torch.zeros(n, device="cuda")
    h.grad(dev(m.pack(Xl)), dev(idx), G, loss)
    torch.cuda.synchronize()
    got = m.unpack(G.cpu().numpy())
    for i in range(n):
        g, l = orc.mlp_grad(Xl[i], dims, feat[i][idx[i]], labels[i][idx[i]])
        assert np.abs(got[i] - g).max() <= 1e-5 * max(np.abs(g).max(), 1e-30)
        assert abs(float(loss[i]) - l) <= 1e-5 * max(abs(l), 1.0)
    Gp = G.cpu().numpy()
    assert np.count_nonzero(Gp) == np.count_nonzero(got)      # padding untouched
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("dims,batch,n", [([256, 128, 128, 10], 128, 3),      # whole tiles
                                           ([3072, 512, 256, 10], 128, 2),     # config 2's model
                                           ([72, 200, 136, 10], 40, 3),        # ragged M, N and K tails
                                           ([320, 264, 24], 264, 2),           # two layers, three row tiles
                                           ([256, 256, 256, 10], 1024, 2),     # the paper's 2NN, batch 1024: 16 K-blocks in dW
                                           ([64, 10], 16, 3)])                 # softmax regression: no tensor-core layer
def test_grad_bf16_tensor_cores_match_oracle(dims, batch, n):
    """BF16 operands, fp32 accumulate.  Two references side by side:
    (1) tests/bf16_reference.py: the same gradient in double on operands rounded to bf16 at the points where
        the CUDA path rounds them.  Per layer block: every entry within 5e-3 of the block's max-norm and the
        block's 2-norm error within 1e-3 (measured on these shapes: at most 5e-4 and 4.5e-4); ReLU decisions on
        pre-activations that fp32 accumulation cannot tell from zero are inferred from the GPU's own output
        (see gradient_agrees).  A dropped K block, a wrong bias gradient scale or a wrong ReLU mask on a few
        percent of the entries is orders of magnitude above these bars.
    (2) the double-precision oracle on the fp32 master weights: bf16 rounding (2^-8 per operand, three chained
        GEMM stages for the first layer's dW, ReLU masks that flip where a pre-activation is within rounding
        of zero) is what separates them: 0.15 of each block's max-norm and a cosine above 0.995."""
    from bf16_reference import gradient_agrees
    p = _dbw()
    rowptr, col = wl.ring(n) if n >= 3 else wl.path(n)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m, flags=p.GEMM_BF16)
    rng = np.random.default_rng(1)
    S = 2 * batch
    feat = rng.random((n, S, dims[0]), dtype=np.float32)
    labels = rng.integers(0, dims[-1], size=(n, S)).astype(np.int32)
    parts = []
    for l in range(len(dims) - 1):
        parts.append(rng.standard_normal((n, dims[l] * dims[l + 1])) * np.sqrt(2.0 / dims[l]))
        parts.append(rng.standard_normal((n, dims[l + 1])) * 0.1)
    Xl = np.concatenate(parts, axis=1).astype(np.float32)
    idx = np.stack([rng.permutation(S)[:batch] for _ in range(n)]).astype(np.int32)
    h.set_dataset(dev(feat), dev(labels), S)
    G = torch.zeros(n, m.ld, device="cuda")
    loss = torch.zeros(n, device="cuda")
    Xd = dev(m.pack(Xl))
    for rep in range(2):                                   # second call reuses the rings and tensor memory
        G.zero_()
        h.grad(Xd, dev(idx), G, loss)
        torch.cuda.synchronize()
    got = m.unpack(G.cpu().numpy())
    assert h.status() == 0
    worst = 0.0
    for i in range(n):
        g, l = orc.mlp_grad(Xl[i], dims, feat[i][idx[i]], labels[i][idx[i]])
        # (a ReLU decision on a pre-activation that fp32 accumulation cannot tell from zero may go either way:
        # see gradient_agrees for how those are treated)
        ok, rep = gradient_agrees(got[i].astype(np.float64), Xl[i], dims, feat[i][idx[i]], labels[i][idx[i]])
        worst = max(worst, rep["l2"])
        assert ok, (i, rep)
        le = rep["loss"]
        off = 0
        for lay in range(len(dims) - 1):
            for size in (dims[lay] * dims[lay + 1], dims[lay + 1]):
                a, r = got[i, off:off + size], g[off:off + size]
                assert np.abs(a - r).max() <= 0.15 * np.abs(r).max() + 1e-7, (i, lay, size)
                off += size
        cos = float(got[i] @ g / (np.linalg.norm(got[i]) * np.linalg.norm(g)))
        assert cos > 0.995, cos
        assert abs(float(loss[i]) - le) <= 1e-4 * max(abs(le), 1.0)
        assert abs(float(loss[i]) - l) <= 2e-2 * max(abs(l), 1.0)
    print("bf16 gradient vs bf16-point reference: worst block 2-norm error %.2e" % worst)
    assert np.count_nonzero(G.cpu().numpy()) <= m.d * n     # padding untouched
    h.close()


@pytest.mark.parametrize("classes,batch,n", [(2, 8, 3), (8, 32, 2), (9, 40, 2), (12, 72, 3), (13, 24, 2), (16, 264, 2), (17, 16, 2)])
def test_bf16_last_layer_at_the_edges_of_its_class_counts(classes, batch, n):
    """Logits are summed over the lanes with samples and classes halved in turn: class counts on both sides of every halving and
    of the kernel's variants, with the references and bars of the test above."""
    test_grad_bf16_tensor_cores_match_oracle([128, 72, classes], batch, n)


@pytest.mark.parametrize("flag", [0, 4])
def test_label_out_of_range_is_clamped_and_reported(flag):
    """A label outside [0, classes) must not become an out-of-bounds read: it is clamped, the status word
    says so, and the loss stays finite."""
    p = _dbw()
    rowptr, col = wl.ring(3)
    dims, batch = [64, 32, 10], 16
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m, flags=flag)
    rng = np.random.default_rng(2)
    S = 32
    feat = rng.random((3, S, dims[0]), dtype=np.float32)
    labels = rng.integers(0, 10, size=(3, S)).astype(np.int32)
    labels[1, 5] = 1 << 30
    labels[2, 7] = -3
    idx = np.stack([np.arange(batch) for _ in range(3)]).astype(np.int32)
    Xl = (rng.standard_normal((3, m.d)) * 0.1).astype(np.float32)
    h.set_dataset(dev(feat), dev(labels), S)
    G = torch.zeros(3, m.ld, device="cuda")
    loss = torch.zeros(3, device="cuda")
    h.grad(dev(m.pack(Xl)), dev(idx), G, loss)
    torch.cuda.synchronize()
    assert h.status() & p.STATUS_BAD_INDEX
    assert torch.isfinite(loss).all() and torch.isfinite(G).all()
    # the clamped labels are what the gradient was computed with
    fixed = np.clip(labels, 0, 9)
    got = m.unpack(G.cpu().numpy())
    for i in range(3):
        g, _ = orc.mlp_grad(Xl[i], dims, feat[i][idx[i]], fixed[i][idx[i]])
        tol = 1e-5 if flag == 0 else 0.15
        assert np.abs(got[i] - g).max() <= tol * np.abs(g).max()
    h.close()


def test_expired_pipeline_wait_is_reported_and_drains():
    """The bounded wait every tensor-core pipeline uses: a barrier that nothing completes makes the wait give
    up after its poll limit, sets DBW_STATUS_WAIT_TIMEOUT, and every later wait of the thread block returns
    at once instead of spinning its own limit; the context stays usable."""
    import time
    p = _dbw()
    rowptr, col = wl.ring(4)
    h = p.Dbw(rowptr, col, d=4)
    out = torch.zeros(3, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    t0 = time.time()
    h.debug_wait_probe(2000, out)
    torch.cuda.synchronize()
    took = time.time() - t0
    o = out.cpu().numpy()
    assert o[0] == 1 and o[1] == 1
    assert o[2] < 20000                       # the second wait did not poll: a few hundred clocks
    assert took < 5.0
    assert h.status() & p.STATUS_WAIT_TIMEOUT
    assert h.status() == 0                    # cleared by the read; the context still works
    kept, *_ = _select_gpu(h, 4, len(col), np.arange(4.0), np.zeros(4, dtype=np.int64))
    assert kept.all()
    h.close()


@pytest.mark.parametrize("rule", ["uniform", "metropolis"])
def test_mix_with_a_mask_that_disagrees_with_b(rule):
    """dbw_mix on its own takes kept and b from the caller.  With uniform weights the weight is
    1 / (1 + entries set in the row), so rows stay stochastic whatever b says; the mismatch is reported."""
    p = _dbw()
    rowptr, col = GRAPHS["reg4_32"]()
    n, d = 32, 64
    h = p.Dbw(rowptr, col, d=d, flags=p.WEIGHT_UNIFORM if rule == "uniform" else 0)
    rng = np.random.default_rng(3)
    X = rng.standard_normal((n, d)).astype(np.float32)
    G = rng.standard_normal((n, d)).astype(np.float32)
    b = np.ones(n, dtype=np.int32)
    kept = orc.select_fastest(rowptr, col, 1.0 + rng.random(n), b)
    kept2 = kept.copy()
    e0 = int(rowptr[5])
    kept2[e0: e0 + 4] = [1, 0, 0, 0]          # worker 5 keeps one neighbour although b says three
    out = torch.empty(n, d, device="cuda")
    h.mix(dev(X), dev(G), dev(kept2), dev(b), 0.1, out)
    torch.cuda.synchronize()
    assert h.status() & p.STATUS_BAD_B
    got = out.cpu().numpy().astype(np.float64)
    if rule == "uniform":
        b_eff = b.copy()
        b_eff[5] = 3                          # the weights follow the mask
        ws, we = orc.mixing_weights(rowptr, col, b_eff, kept2, orc.UNIFORM)
        assert row_rel_err(got, orc.mix_update(rowptr, col, X, G, ws, we, 0.1)) <= 1e-5
    else:                                     # Assumption 1 on the nominal counts; w_ii = 1 - sum keeps the row stochastic
        ws, we = orc.mixing_weights(rowptr, col, b, kept2, orc.METROPOLIS)
        assert abs(ws[5] + we[e0: e0 + 4].sum() - 1.0) < 1e-12
        assert row_rel_err(got, orc.mix_update(rowptr, col, X, G, ws, we, 0.1)) <= 1e-5
    h.close()


@pytest.mark.parametrize("kernel,graph,panel", [("mix_panel_kernel", "reg4_32", 0), ("mix_staged_kernel", "reg32_256", 1),
                                                ("mix_direct_kernel", "reg4_32", -1), ("mix_tc_kernel", "reg32_256", 2),
                                                ("mix_sp_kernel", "reg32_256", 3)])
@pytest.mark.parametrize("order", ["local_then_mix", "mix_then_correct"])
def test_consensus_only_mix_reads_no_gradient(kernel, graph, panel, order):
    """G == NULL (Section 3.2.1's truncated model: gradients zero after K) gives the bits of a mix with an
    all-zero gradient matrix, in every mix kernel and both update orders."""
    p = _dbw()
    rowptr, col = GRAPHS[graph]()
    n, d = len(rowptr) - 1, 1000
    deg = np.diff(rowptr)
    flags = p.WEIGHT_UNIFORM | (p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    h = p.Dbw(rowptr, col, d=d, flags=flags)
    h.set_mix_panel(panel)
    assert h.mix_kernel() == kernel
    rng = np.random.default_rng(4)
    X = dev(rng.standard_normal((n, d)).astype(np.float32))
    t = dev(1.0 + rng.random(n))
    b = dev(rng.integers(0, deg // 2 + 1).astype(np.int32))
    kept = torch.zeros(len(col), dtype=torch.uint8, device="cuda")
    out0, out1 = torch.empty_like(X), torch.empty_like(X)
    h.round(X, t, b, 0.1, out0, kept, G_ext=torch.zeros_like(X))
    h.round(X, t, b, 0.1, out1, kept)                         # neither batches nor gradients: G = 0
    torch.cuda.synchronize()
    assert torch.equal(out0, out1)
    out2 = torch.empty_like(X)
    h.mix(X, None, kept, b, 0.1, out2)
    torch.cuda.synchronize()
    assert torch.equal(out0, out2)
    assert h.status() == 0
    h.close()


def test_consensus_only_rounds_converge_to_the_initial_mean():
    """Corollary 1 / the truncated model of Section 3.2.1 with G = 0 and b = 0 (Metropolis weights doubly
    stochastic): every round agrees with the oracle to 1e-5 (teacher-forced from the GPU's own fp32 state),
    the network mean is preserved and the rows contract geometrically onto it."""
    p = _dbw()
    rowptr, col = GRAPHS["reg4_32"]()
    n, d = 32, 1536
    h = p.Dbw(rowptr, col, d=d)
    rng = np.random.default_rng(6)
    X0 = rng.standard_normal((n, d)).astype(np.float32)
    mean0 = X0.astype(np.float64).mean(axis=0)
    X = dev(X0)
    b = np.zeros(n, dtype=np.int32)
    kept = torch.zeros(len(col), dtype=torch.uint8, device="cuda")
    spread = []
    X_orc = X0.astype(np.float64)
    rounds = 120
    for k in range(rounds):
        t = 1.0 + rng.random(n)
        before = X.cpu().numpy()
        h.round(X, dev(t), dev(b), 0.05, X, kept)             # in place, no gradients
        torch.cuda.synchronize()
        r = orc.dbw_round(rowptr, col, before, t, b, 0.05, G=np.zeros((n, d)))
        assert row_rel_err(X.cpu().numpy(), r["X"]) <= 1e-5, k
        X_orc = orc.dbw_round(rowptr, col, X_orc, t, b, 0.05, G=np.zeros((n, d)))["X"]
        spread.append(float(np.abs(X.cpu().numpy().astype(np.float64) - mean0).max()))
    got = X.cpu().numpy().astype(np.float64)
    assert np.abs(got.mean(axis=0) - mean0).max() <= 1e-5     # mean preserved (fp32 rounding only)
    assert spread[59] < 1e-2 * spread[0] and spread[-1] < 1e-4 * spread[0]
    rate = (spread[59] / spread[9]) ** (1.0 / 50)
    assert rate < 0.95                                        # geometric contraction
    assert np.abs(got - X_orc).max() <= 1e-5
    assert h.status() == 0
    h.close()


def test_degenerate_sizes():
    """One worker (no links), two workers, and a padded leading dimension far above d."""
    p = _dbw()
    # N = 1: no neighbours, the round is a plain SGD step and lasts t_0
    rowptr, col = np.array([0, 0], dtype=np.int32), np.zeros(0, dtype=np.int32)
    h = p.Dbw(rowptr, col, d=10, ld=12)
    X = torch.arange(12, dtype=torch.float32, device="cuda").reshape(1, 12)
    G = torch.ones(1, 12, device="cuda")
    kept = torch.zeros(1, dtype=torch.uint8, device="cuda")
    Tw = torch.zeros(1, dtype=torch.float64, device="cuda")
    Tr = torch.zeros(1, dtype=torch.float64, device="cuda")
    out = torch.empty_like(X)
    t, b = dev(np.array([2.5])), dev(np.zeros(1, dtype=np.int32))
    h.round(X, t, b, 0.5, out, kept, G_ext=G, T_worker=Tw, T_round=Tr)
    torch.cuda.synchronize()
    assert torch.equal(out, X - 0.5 * G)
    assert float(Tw[0]) == 0.0 and float(Tr[0]) == 0.0         # nobody waits for anybody: no participant
    bo = torch.full((1,), 7, dtype=torch.int32, device="cuda")
    th = torch.zeros(1, dtype=torch.float64, device="cuda")
    h.update_backups(t, bo, th)                                   # no links: threshold +inf, b = deg = 0
    torch.cuda.synchronize()
    assert int(bo[0]) == 0 and np.isinf(float(th[0]))
    assert h.status() == 0
    h.close()
    # N = 2, ld much larger than d (the tail is padding and must stay zero)
    rowptr, col = wl.path(2)
    d, ld = 6, 512
    h = p.Dbw(rowptr, col, d=d, ld=ld)
    rng = np.random.default_rng(0)
    Xh = np.zeros((2, ld), dtype=np.float32); Gh = np.zeros((2, ld), dtype=np.float32)
    Xh[:, :d] = rng.standard_normal((2, d)); Gh[:, :d] = rng.standard_normal((2, d))
    Xd = dev(Xh)
    kept = torch.zeros(2, dtype=torch.uint8, device="cuda")
    tt, bb = np.array([1.0, 1.0]), np.zeros(2, dtype=np.int32)
    h.round(Xd, dev(tt), dev(bb), 0.1, Xd, kept, G_ext=dev(Gh))
    torch.cuda.synchronize()
    r = orc.dbw_round(rowptr, col, Xh, tt, bb, 0.1, G=Gh)
    assert row_rel_err(Xd.cpu().numpy()[:, :d], r["X"][:, :d]) <= 1e-5
    assert not np.any(Xd.cpu().numpy()[:, d:])
    assert np.array_equal(kept.cpu().numpy(), r["kept"])
    h.close()


@pytest.mark.parametrize("name", ["ring8", "complete40", "reg4_32", "er64", "reg32_256"])
def test_selection_with_per_link_times_bit_exact(name):
    p = _dbw()
    rowptr, col = GRAPHS[name]()
    n, nnz = len(rowptr) - 1, len(col)
    deg = np.diff(rowptr)
    h = p.Dbw(rowptr, col, d=8)
    rng = np.random.default_rng(31)
    X = rng.standard_normal((n, 8)).astype(np.float32)
    G = rng.standard_normal((n, 8)).astype(np.float32)
    for trial in range(4):
        t = 1.0 + rng.exponential(1.0, size=n)
        te = np.round(4 * (t[col] + rng.random(nnz))) / 4                 # link delays, with ties
        b = rng.integers(0, deg + 1)
        h.set_edge_times(dev(te))
        kept, Tw, Tn, Tr = _select_gpu(h, n, nnz, t, b)
        ref = orc.select_fastest(rowptr, col, t, b, t_edge=te)
        assert np.array_equal(kept, ref)
        rTn, rTw, rTr = orc.round_times(rowptr, col, t, b, ref, t_edge=te)
        assert np.array_equal(Tn, rTn) and np.array_equal(Tw, rTw) and Tr == rTr
        # the whole round follows the link-time selection
        out = torch.empty(n, 8, device="cuda")
        kd = torch.zeros(nnz, dtype=torch.uint8, device="cuda")
        h.round(dev(X), dev(t), dev(b.astype(np.int32)), 0.1, out, kd, G_ext=dev(G))
        torch.cuda.synchronize()
        ws, we = orc.mixing_weights(rowptr, col, b, ref)
        assert np.array_equal(kd.cpu().numpy(), ref)
        assert row_rel_err(out.cpu().numpy(), orc.mix_update(rowptr, col, X, G, ws, we, 0.1)) <= 1e-5
        h.set_edge_times(None)                                            # back to per-worker times
        kept0, *_ = _select_gpu(h, n, nnz, t, b)
        assert np.array_equal(kept0, orc.select_fastest(rowptr, col, t, b))
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("dims,batch,n", [([72, 200, 136, 10], 40, 10),      # 128-wide dW tiles, ragged on every side
                                          ([328, 264, 10], 24, 40),          # 256-wide dW tiles, ragged
                                          ([256, 128, 64, 10], 64, 150)])    # whole tiles; panels of fewer columns
@pytest.mark.parametrize("order", ["local_then_mix", "mix_then_correct"])
def test_round_with_few_participants_gives_the_bits_of_its_steps(dims, batch, n, order):
    """In a tensor-core round the dW GEMMs take the SGD step of the workers that take no part and the mix works on the
    others.  From no participant to all of them, around the count at which the round is mixed as a whole, in place and
    not, with and without parameter tracking, the round gives the bits of its steps called one by one (dbw_grad,
    dbw_select, dbw_mix), which the oracle tests pin."""
    p = _dbw()
    rowptr, col = wl.ring(n)
    deg = np.diff(rowptr)
    flags = p.GEMM_BF16 | (p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m, flags=flags)
    rng = np.random.default_rng(5)
    S = 2 * batch
    feat = dev(rng.standard_normal((n, S, dims[0]), dtype=np.float32))
    labels = dev(rng.integers(0, dims[-1], size=(n, S)).astype(np.int32))
    h.set_dataset(feat, labels, S)
    X0 = np.zeros((n, m.ld), dtype=np.float32)
    X0[:] = m.pack(0.1 * rng.standard_normal((n, m.d)).astype(np.float32))
    idx = dev(rng.integers(0, S, size=(n, batch)).astype(np.int32))
    lr_pw = dev(rng.uniform(0.01, 0.1, size=n).astype(np.float32))
    kept, kept2 = (torch.zeros(len(col), dtype=torch.uint8, device="cuda") for _ in range(2))
    G = torch.zeros(n, m.ld, device="cuda")
    for k in (0, 2, n // 2, n // 2 + 1, n):
        inside = np.arange(n) < k
        t = dev(np.where(inside, 1.0, 9.0) + rng.random(n))
        mates = np.array([inside[col[rowptr[i]:rowptr[i + 1]]].sum() for i in range(n)])
        b = dev(np.where(inside, deg - mates, deg).astype(np.int32))
        X = dev(X0)
        h.set_param_tracking(False)
        ref = torch.empty_like(X)
        h.grad(X, idx, G)
        h.select(t, b, kept)
        h.mix(X, G, kept, b, 0.05, ref, lr_per_worker=lr_pw)
        for track in (False, True):
            h.set_param_tracking(track)
            out = torch.full_like(X, float("nan"))
            h.round(X, t, b, 0.05, out, kept2, batch_idx=idx, lr_per_worker=lr_pw)
            assert torch.equal(out, ref) and torch.equal(kept, kept2), (k, track)
            Y = X.clone()
            h.round(Y, t, b, 0.05, Y, kept2, batch_idx=idx, lr_per_worker=lr_pw)
            assert torch.equal(Y, ref), (k, track)
        # the tracked bf16 copy is that of a cast after the fact: the next gradients agree
        G2 = torch.zeros_like(G)
        h.grad(Y, idx, G2)
        h.set_param_tracking(False)
        h.grad(Y, idx, G)
        assert torch.equal(G, G2), k
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("dims,batch,n", [([32, 10], 257, 3),           # two parts of the batch, the second of one sample
                                          ([40, 24, 32], 256, 3),       # one part, the most classes: the largest staging
                                          ([64, 48, 36, 10], 520, 4),   # three parts; a bias gradient out of a dW GEMM
                                          ([68, 36, 100, 12], 20, 3),   # GEMMs in slices of k: ragged tiles, a last slice of a few k
                                          ([260, 64, 32, 10], 64, 5),   # ... whole tiles, a slice of less than a step more
                                          ([128, 320, 64, 10], 64, 60),  # as many tiles as do without slices, and fewer
                                          ([132, 100, 12], 52, 40),     # one-warp forward tiles: ragged in every dimension
                                          ([128, 320, 64, 10], 20, 60),  # ... one row of them, k of whole steps
                                          ([64, 30, 36, 10], 18, 3)])   # widths and a batch without 128-bit accesses beside some with
def test_fp32_last_layer_in_parts_of_the_batch(dims, batch, n):
    """The last layer's backward step splits a large batch into parts whose sums are added in a fixed order.  Gradients and
    losses against the oracle (hidden units are far on one side of zero, so no ReLU decision is a matter of rounding), and
    the single-launch round against the step-by-step one, bit for bit."""
    p = _dbw()
    rowptr, col = wl.ring(n)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m)
    rng = np.random.default_rng(2)
    S = batch + 40
    feat = rng.random((n, S, dims[0]), dtype=np.float32)
    labels = rng.integers(0, dims[-1], size=(n, S)).astype(np.int32)
    X = m.pack((0.05 * rng.standard_normal((n, m.d))).astype(np.float32))
    for l in range(len(dims) - 2):
        X[:, m.b_off[l]: m.b_off[l] + dims[l + 1]] = np.where(np.arange(dims[l + 1]) % 3 == 0, -9.0, 9.0) * 0.5 ** l
    idx = np.stack([rng.permutation(S)[:batch] for _ in range(n)]).astype(np.int32)
    h.set_dataset(dev(feat), dev(labels), S)
    G, loss = torch.zeros(n, m.ld, device="cuda"), torch.zeros(n, device="cuda")
    h.grad(dev(X), dev(idx), G, loss)
    got = m.unpack(G.cpu().numpy())
    for i in range(n):
        g, l = orc.mlp_grad(m.unpack(X[i:i + 1])[0], dims, feat[i][idx[i]], labels[i][idx[i]])
        assert np.abs(got[i] - g).max() <= 1e-5 * np.abs(g).max()
        assert abs(float(loss[i]) - l) <= 1e-5 * max(abs(l), 1.0)
    t, b = dev(1.0 + rng.random(n)), torch.ones(n, dtype=torch.int32, device="cuda")
    outs = []
    for fused in (True, False):
        h.set_fused_round(fused)
        assert h.round_is_fused() == fused
        Y, kept = dev(X), torch.zeros(len(col), dtype=torch.uint8, device="cuda")
        h.round(Y, t, b, 0.05, Y, kept, batch_idx=dev(idx), loss=loss)
        outs.append((Y, loss.clone()))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("n", [1, 2, 127, 512, 513, 4097, 6016, 6100])  # strides of the loads, the last size with its times in shared memory
def test_threshold_rule_and_times_at_the_edges_of_the_worker_count(n):
    p = _dbw()
    rowptr, col = wl.ring(n) if n >= 3 else wl.path(n)
    h = p.Dbw(rowptr, col, d=4)
    ref = orc.Dtur(rowptr, col) if n > 1 else None
    rng = np.random.default_rng(n)
    b, kept = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(max(len(col), 1), dtype=torch.uint8, device="cuda")
    Tw, Tn, Tr, theta = (torch.zeros(k, dtype=torch.float64, device="cuda") for k in (n, n, 1, 1))
    for k in range(3):
        t = 1.0 + np.round(rng.exponential(1.0, size=n), 2)      # with ties
        h.update_backups(dev(t), b, theta)
        h.select(dev(t), b, kept, Tw, Tn, Tr)
        if n == 1:
            assert int(b[0]) == 0 and float(Tr[0]) == 0.0
            continue
        rb, rt = ref.update_backups(t)
        assert np.array_equal(b.cpu().numpy(), rb) and float(theta[0]) == rt
        rk = orc.select_fastest(rowptr, col, t, rb)
        assert np.array_equal(kept.cpu().numpy(), np.asarray(rk, dtype=np.uint8))
        rTn, rTw, rTr = orc.round_times(rowptr, col, t, rb, rk)
        assert np.array_equal(Tn.cpu().numpy(), rTn) and np.array_equal(Tw.cpu().numpy(), rTw) and float(Tr[0]) == rTr
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("n,deg", [(960, 32), (1024, 6), (1025, 30), (2048, 8), (2049, 14), (4096, 8)])
@pytest.mark.parametrize("rule,order", [("uniform", "local_then_mix"), ("metropolis", "mix_then_correct"), ("metropolis", "local_then_mix")])
def test_staged_kernel_at_the_edges_of_its_panel_widths(n, deg, rule, order):
    """Panels of 32, 16 and 8 columns by the worker count, the largest degrees whose weight codes and lists still fit, rows
    that keep nobody, a ragged last panel, in place: against the oracle, and with the paper's weights bit for bit against the
    kernel that gathers through L2."""
    p = _dbw()
    d = 1036
    rowptr, col = wl.random_regular(n, deg, 3)
    flags = (p.WEIGHT_UNIFORM if rule == "uniform" else 0) | (p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    h = p.Dbw(rowptr, col, d=d, flags=flags)
    h.set_mix_panel(1)
    assert h.mix_kernel() == "mix_staged_kernel" and h.mix_in_place_ok()
    rng = np.random.default_rng(4)
    X, G = (rng.standard_normal((n, d), dtype=np.float32) for _ in range(2))
    b = rng.integers(0, deg + 1, size=n)
    b[:40] = 0
    t = 1.0 + rng.exponential(1.0, size=n)
    kept = orc.select_fastest(rowptr, col, t, b)
    ws, we = orc.mixing_weights(rowptr, col, b, kept, rule)
    args = (dev(G), dev(kept), dev(b.astype(np.int32)), 0.05)
    Y = dev(X)
    h.mix(Y, *args, Y)
    assert row_rel_err(Y.cpu().numpy(), orc.mix_update(rowptr, col, X, G, ws, we, 0.05, order)) <= 1e-5
    if rule == "metropolis":
        h.set_mix_panel(-1)
        Z = torch.empty_like(Y)
        h.mix(dev(X), *args, Z)
        assert torch.equal(Y, Z)
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("between", ["grad", "round_of_another_matrix"])
def test_tracked_copy_is_forgotten_when_other_parameters_pass_through(between):
    """With parameter tracking the bf16 copy belongs to the X_out of the call before.  Gradients of another matrix Z in between
    (an averaged model, say) overwrite it: gradients of the tracked matrix Y afterwards are those without tracking, bit for bit."""
    p = _dbw()
    dims, batch, n = [128, 72, 64, 10], 32, 6
    rowptr, col = wl.ring(n)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m, flags=p.GEMM_BF16)
    rng = np.random.default_rng(8)
    S = 2 * batch
    feat, labels = dev(rng.standard_normal((n, S, dims[0]), dtype=np.float32)), dev(rng.integers(0, dims[-1], size=(n, S)).astype(np.int32))
    h.set_dataset(feat, labels, S)
    X, Z = (dev(m.pack(0.1 * rng.standard_normal((n, m.d)).astype(np.float32))) for _ in range(2))
    idx = dev(rng.integers(0, S, size=(n, batch)).astype(np.int32))
    t = dev(1.0 + rng.random(n))
    kept = torch.zeros(len(col), dtype=torch.uint8, device="cuda")
    for backups in (1, 2):  # everybody mixes / the dW GEMMs take everybody's step
        b = torch.full((n,), backups, dtype=torch.int32, device="cuda")
        h.set_param_tracking(True)
        Y, other = torch.empty_like(X), torch.empty_like(X)
        h.round(X, t, b, 0.05, Y, kept, batch_idx=idx)
        G, G_ref = torch.zeros_like(X), torch.zeros_like(X)
        if between == "grad":
            h.grad(Z, idx, G)
        else:
            h.round(Z, t, b, 0.05, other, kept, batch_idx=idx)
        h.grad(Y, idx, G)
        h.set_param_tracking(False)
        h.grad(Y, idx, G_ref)
        assert torch.equal(G, G_ref), backups
    assert h.status() == 0
    h.close()


def test_bias_gradient_of_a_layer_of_one_unit():
    """One unit: its dW GEMM has unit stride along k on both sides and no slices, and its bias gradient is summed in the same order,
    step by step and in one launch."""
    p = _dbw()
    dims, batch, n = [64, 1, 10], 128, 3
    rowptr, col = wl.ring(n)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m)
    rng = np.random.default_rng(12)
    feat, labels = dev(rng.random((n, batch, dims[0]), dtype=np.float32)), dev(rng.integers(0, 10, size=(n, batch)).astype(np.int32))
    h.set_dataset(feat, labels, batch)
    X = m.pack((0.3 * rng.standard_normal((n, m.d))).astype(np.float32))
    X[:, m.w_off[0]: m.w_off[0] + dims[0]] = np.abs(X[:, m.w_off[0]: m.w_off[0] + dims[0]])  # every sample passes the ReLU
    X[:, m.b_off[0]] = 0.0  # its step is all that is left of it
    idx = dev(np.stack([rng.permutation(batch) for _ in range(n)]).astype(np.int32))
    t, b = dev(1.0 + rng.random(n)), torch.full((n,), 2, dtype=torch.int32, device="cuda")
    outs = []
    for fused in (True, False):
        h.set_fused_round(fused)
        Y, kept = dev(X), torch.zeros(len(col), dtype=torch.uint8, device="cuda")
        h.round(Y, t, b, 0.05, Y, kept, batch_idx=idx)
        outs.append(Y)
    assert torch.equal(outs[0], outs[1])
    assert h.status() == 0
    h.close()


# both sides measured where the lines were drawn (csrc/round_fused.cu)
@pytest.mark.parametrize("dims,batch,n,single", [([784, 10], 32, 8, True), ([784, 10], 64, 16, True), ([256, 10], 128, 20, True), ([256, 10], 129, 20, False),
                                                 ([121, 10], 16, 4, True), ([121, 10], 17, 4, False),
                                                 ([256, 64, 10], 128, 8, True), ([64, 40, 10], 24, 21, False), ([64, 40, 10], 102, 20, True),
                                                 ([64, 41, 10], 32, 16, True), ([64, 41, 10], 33, 16, False), ([64, 41, 41, 10], 4, 50, True),
                                                 ([784, 200, 10], 64, 32, False), ([784, 320, 10], 128, 4, False)])
def test_which_rounds_are_one_launch(dims, batch, n, single):
    p = _dbw()
    rowptr, col = wl.ring(n)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m)
    feat, labels = torch.zeros(n, batch, dims[0], device="cuda"), torch.zeros(n, batch, dtype=torch.int32, device="cuda")
    h.set_dataset(feat, labels, batch)
    assert h.round_is_fused() == single
    h.close()


@pytest.mark.parametrize("n,deg,d,flags,kernel,in_place", [
    (1019, 48, 10_653, 0, "mix_panel_kernel", True), (1000, 32, 10_653, 0, "mix_staged_kernel", True),    # lists that crowd L1 out
    (922, 48, 13_110, 0, "mix_staged_kernel", True),
    (2652, 8, 1507, 0, "mix_panel_kernel", True), (2652, 8, 1507, 1, "mix_staged_kernel", True),          # weighted lists, a matrix in L2
    (3049, 20, 11_692, 1, "mix_panel_kernel", True), (2500, 8, 30_000, 0, "mix_staged_kernel", True),
    (3700, 6, 20_000, 0, "mix_staged_kernel", False), (3700, 6, 20_000, 2, "mix_direct_kernel", False)])   # no panel of all rows fits
def test_which_kernel_mixes_many_workers(n, deg, d, flags, kernel, in_place):
    p = _dbw()
    h = p.Dbw(*wl.random_regular(n, deg, 7), d=d, flags=flags)
    assert h.mix_kernel() == kernel and h.mix_in_place_ok() == in_place
    h.close()


@pytest.mark.parametrize("order", ["local_then_mix", "mix_then_correct"])
def test_kernel_by_the_kept_count_where_no_panel_fits(order):
    """Out of place the L2 kernel takes the rounds of fewer than six kept neighbours a worker (in Eq. 3's order, and without
    gradients, every round) and the staged kernel the others; in place it is the staged kernel's alone.  Uniform weights, which
    the two apply at different places of the sum, tell them apart by their bits."""
    p = _dbw()
    n, deg, d = 3640, 8, 19_000
    rowptr, col = wl.random_regular(n, deg, 3)
    flags = p.WEIGHT_UNIFORM | (p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    h = p.Dbw(rowptr, col, d=d, flags=flags)
    gen = torch.Generator(device="cuda").manual_seed(5)
    X, G = (torch.randn(n, h.ld, device="cuda", generator=gen) for _ in range(2))
    X[:, d:] = 0
    G[:, d:] = 0
    kept = torch.zeros(len(col), dtype=torch.uint8, device="cuda")
    t = dev(1.0 + np.random.default_rng(2).random(n))
    out, direct, staged = (torch.empty_like(X) for _ in range(3))
    for total in (0, 6 * n - 1, 6 * n, deg * n):
        p_i = np.full(n, total // n) + (np.arange(n) < total % n)
        b = dev((deg - p_i).astype(np.int32))
        h.select(t, b, kept)
        for g in (G, None):
            for panel, to in ((-1, direct), (1, staged), (0, out)):
                h.set_mix_panel(panel)
                h.mix(X, g, kept, b, 0.05, to)
            assert total == 0 or not torch.equal(direct, staged)
            wants = direct if total < 6 * n or g is None or order == "mix_then_correct" else staged
            assert torch.equal(out, wants), (total, g is None)
            Y = X.clone()
            h.mix(Y, g, kept, b, 0.05, Y)  # in place: accepted, by the staged kernel
            assert torch.equal(Y, staged), (total, g is None)
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("n,cols", [(10, 16), (10, 32), (10, 64), (10, 256), (80, 0), (80, 16)])  # 80 workers: four and five dW tiles to an SM
def test_stepping_rounds_with_merged_panels_of_every_width(n, cols):
    """Rounds whose dW GEMMs step, on a matrix wide enough that several panels of the participants are staged together, the last
    group of a block a ragged one, with every panel width, and with several dW tiles to an SM: the bits of the round's steps.  One
    launch more than with a mix that cannot leave rows out says that this is the path."""
    p = _dbw()
    from paper_2102_06280_b200 import binding
    dims, batch = [1024, 264, 10], 64
    rowptr, col = wl.ring(n)
    deg = np.diff(rowptr)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m, flags=p.GEMM_BF16)
    gen = torch.Generator(device="cuda").manual_seed(3)
    feat, labels = torch.randn(n, batch, dims[0], device="cuda", generator=gen), torch.randint(0, 10, (n, batch), dtype=torch.int32, device="cuda", generator=gen)
    h.set_dataset(feat, labels, batch)
    X = torch.zeros(n, m.ld, device="cuda")
    for l in range(2):
        X[:, m.w_off[l]: m.w_off[l] + dims[l] * dims[l + 1]].normal_(0.0, 0.05, generator=gen)
    idx = torch.stack([torch.randperm(batch, device="cuda", generator=gen) for _ in range(n)]).int()
    rng = np.random.default_rng(1)
    kept, kept2 = (torch.zeros(len(col), dtype=torch.uint8, device="cuda") for _ in range(2))
    G, ref, out = (torch.zeros_like(X) for _ in range(3))

    def launches(f):
        before = binding.launch_count()
        f()
        return binding.launch_count() - before

    for k in (0, 2, 3, n // 2):
        inside = np.arange(n) < k
        t = dev(np.where(inside, 1.0, 9.0) + rng.random(n))
        mates = np.array([inside[col[rowptr[i]:rowptr[i + 1]]].sum() for i in range(n)])
        b = dev(np.where(inside, deg - mates, deg).astype(np.int32))
        h.set_mix_panel(cols)
        h.grad(X, idx, G)
        h.select(t, b, kept)
        h.mix(X, G, kept, b, 0.05, ref)
        for track in (False, True):
            h.set_param_tracking(track)
            out.fill_(float("nan"))
            stepping = launches(lambda: h.round(X, t, b, 0.05, out, kept2, batch_idx=idx))
            assert torch.equal(out, ref) and torch.equal(kept, kept2), (k, track)
            Y = X.clone()
            h.set_param_tracking(track)
            h.round(Y, t, b, 0.05, Y, kept2, batch_idx=idx)
            assert torch.equal(Y, ref), (k, track)
            h.set_param_tracking(False)
            h.set_mix_panel(-1)
            assert stepping == launches(lambda: h.round(X, t, b, 0.05, out, kept2, batch_idx=idx)) + 1
            h.set_mix_panel(cols)
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("kind", ["fp32_steps", "bf16", "bf16_tracked", "mix_only", "consensus_only", "one_launch"])
@pytest.mark.parametrize("dynamic", [False, True])
def test_round_host_on_two_streams_gives_the_bits_of_dbw_round(kind, dynamic):
    """dbw_round_host with its copies beside the gradients and the mix: several rounds queued without a wait in between, each with host
    buffers of its own, with given backup counts and with the threshold rule's, against dbw_update_backups and dbw_round."""
    p = _dbw()
    n, rounds = 12, 5
    rowptr, col = wl.random_regular(n, 4, 1)
    rng = np.random.default_rng(6)
    model = kind in ("fp32_steps", "one_launch") or kind.startswith("bf16")
    if model:
        dims, batch, S = [136, 72, 10], 40, 90
        m = p.model_layout(dims, batch)
        handles = [p.Dbw(rowptr, col, d=m.d, model=m, flags=p.GEMM_BF16 if kind.startswith("bf16") else 0) for _ in range(2)]
        feat, labels = dev(rng.random((n, S, dims[0]), dtype=np.float32)), dev(rng.integers(0, 10, size=(n, S)).astype(np.int32))
        X0 = dev(m.pack((0.1 * rng.standard_normal((n, m.d))).astype(np.float32)))
        for h in handles:
            h.set_dataset(feat, labels, S)
            h.set_fused_round(kind == "one_launch")
            h.set_param_tracking(kind == "bf16_tracked")
        G = None
    else:
        handles = [p.Dbw(rowptr, col, d=5000) for _ in range(2)]
        X0 = dev(rng.standard_normal((n, 5000), dtype=np.float32))
        G = dev(0.1 * rng.standard_normal((n, 5000), dtype=np.float32)) if kind == "mix_only" else None
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
    times = [pin(1.0 + rng.exponential(1.0, size=n)) for _ in range(rounds)]
    counts = [pin(rng.integers(0, 5, size=n).astype(np.int32)) for _ in range(rounds)]
    idx = [pin(np.stack([rng.permutation(90)[:40] for _ in range(n)]).astype(np.int32)) for _ in range(rounds)] if model else [None] * rounds

    def results():
        return {"kept": torch.zeros(len(col), dtype=torch.uint8), "T_worker": torch.zeros(n, dtype=torch.float64), "T_round": torch.zeros(1, dtype=torch.float64),
                "loss": torch.zeros(n), "b_out": torch.zeros(n, dtype=torch.int32)}

    # on the host's buffers
    h, X, got = handles[0], X0.clone(), []
    for k in range(rounds):
        r = {name: v.pin_memory() for name, v in results().items()}
        h.round_host(X, times[k], None if dynamic else counts[k], 0.05, X, h_batch_idx=idx[k], G_ext=G, h_kept=r["kept"], h_T_worker=r["T_worker"],
                     h_T_round=r["T_round"], h_loss=r["loss"] if model else None, h_b_out=r["b_out"])
        got.append(r)
    torch.cuda.current_stream().synchronize()
    # on the device's
    h, Y = handles[1], X0.clone()
    for k in range(rounds):
        r = {name: v.cuda() for name, v in results().items()}
        t = times[k].cuda()
        if dynamic:
            h.update_backups(t, r["b_out"])
        else:
            r["b_out"].copy_(counts[k])
        h.round(Y, t, r["b_out"], 0.05, Y, r["kept"], batch_idx=None if idx[k] is None else idx[k].cuda(), G_ext=G, T_worker=r["T_worker"],
                T_round=r["T_round"], loss=r["loss"] if model else None)
        for name, v in r.items():
            assert torch.equal(v.cpu(), got[k][name]), (k, name)
    assert torch.equal(X, Y)
    for h in handles:
        assert h.status() == 0
        h.close()


@pytest.mark.parametrize("dims,batch,n", [([129, 127, 65, 10], 97, 40),   # nothing a multiple of four: rows at every shift, partial tiles one short and one over
                                          ([132, 128, 64, 10], 128, 64),  # whole tiles, more of them than SMs, and dW with four columns over
                                          ([784, 64, 10], 64, 20),        # dW alone, two steps, no more tiles than SMs: the deep ring
                                          ([36, 256, 10], 128, 60),       # dW of 36 columns
                                          ([31, 301, 10], 100, 40),       # dW of three steps and four samples
                                          ([300, 201, 10], 33, 20),       # dW of a step and one sample
                                          ([65, 500, 130, 10], 250, 12)])
def test_fp32_gemms_on_the_tensor_cores(dims, batch, n):
    """fp32 GEMMs of three bf16 pieces per value: gradients and losses against the oracle within 1e-5 of the largest entry (fp32 sums;
    hidden units far from zero, so no ReLU decision is a matter of rounding), single launch and steps bit for bit, and an infinite
    weight that stays its worker's own and shows in its loss."""
    p = _dbw()
    rowptr, col = wl.ring(n)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m)
    rng = np.random.default_rng(4)
    S = batch + 11
    feat = rng.random((n, S, dims[0]), dtype=np.float32)
    labels = rng.integers(0, dims[-1], size=(n, S)).astype(np.int32)
    X = m.pack((0.05 * rng.standard_normal((n, m.d))).astype(np.float32))
    for l in range(len(dims) - 2):
        X[:, m.b_off[l]: m.b_off[l] + dims[l + 1]] = np.where(np.arange(dims[l + 1]) % 3 == 0, -9.0, 9.0) * 0.5 ** l
    idx = np.stack([rng.permutation(S)[:batch] for _ in range(n)]).astype(np.int32)
    h.set_dataset(dev(feat), dev(labels), S)
    G, loss = torch.zeros(n, m.ld, device="cuda"), torch.zeros(n, device="cuda")
    h.grad(dev(X), dev(idx), G, loss)
    got = m.unpack(G.cpu().numpy())
    for i in range(n):
        g, l = orc.mlp_grad(m.unpack(X[i:i + 1])[0], dims, feat[i][idx[i]], labels[i][idx[i]])
        assert np.abs(got[i] - g).max() <= 1e-5 * np.abs(g).max()
        assert abs(float(loss[i]) - l) <= 1e-5 * max(abs(l), 1.0)
    if n <= 64:
        t, b = dev(1.0 + rng.random(n)), torch.ones(n, dtype=torch.int32, device="cuda")
        outs = []
        for fused in (True, False):
            h.set_fused_round(fused)
            Y, kept = dev(X), torch.zeros(len(col), dtype=torch.uint8, device="cuda")
            h.round(Y, t, b, 0.05, Y, kept, batch_idx=dev(idx), loss=loss)
            outs.append((Y, loss.clone()))
        assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    X[1, m.w_off[0] + dims[0] + 1] = np.inf  # a unit that passes its ReLU
    G2, loss2 = torch.zeros_like(G), torch.zeros_like(loss)
    h.grad(dev(X), dev(idx), G2, loss2)
    others = [i for i in range(n) if i != 1]
    assert torch.equal(G2[others], G[others]) and not np.isfinite(float(loss2[1]))
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("dims,batch,n", [([33, 10], 65, 3),             # one layer, rows of the data set at every shift
                                          ([64, 131, 10], 72, 35),       # sixteen lanes to a feature group, a last group of three features
                                          ([64, 132, 12], 301, 30),      # ... aligned, two parts, four samples to a warp and one left over
                                          ([64, 35, 16], 258, 41),       # ... unaligned
                                          ([64, 130, 32], 50, 30),       # the most classes
                                          ([64, 132, 30], 90, 30),       # ... with sixteen lanes to a feature group, aligned
                                          ([64, 131, 20], 72, 35),       # ... and not
                                          ([20, 1, 3], 9, 4)])           # a single feature
def test_fp32_last_layer_of_any_width(dims, batch, n):
    """The last layer's two steps with rows that are not 16-byte aligned, and their variants by size: gradients and losses against the
    oracle within 1e-5 of the largest entry (fp32 sums; hidden units far from zero), single launch and steps bit for bit."""
    p = _dbw()
    rowptr, col = wl.ring(n)
    m = p.model_layout(dims, batch)
    h = p.Dbw(rowptr, col, d=m.d, model=m)
    rng = np.random.default_rng(8)
    S = batch + 5
    feat = rng.random((n, S, dims[0]), dtype=np.float32)
    labels = rng.integers(0, dims[-1], size=(n, S)).astype(np.int32)
    X = m.pack((0.05 * rng.standard_normal((n, m.d))).astype(np.float32))
    for l in range(len(dims) - 2):
        X[:, m.b_off[l]: m.b_off[l] + dims[l + 1]] = np.where(np.arange(dims[l + 1]) % 3 == 0, 9.0, -9.0)
    idx = np.stack([rng.permutation(S)[:batch] for _ in range(n)]).astype(np.int32)
    h.set_dataset(dev(feat), dev(labels), S)
    G, loss = torch.zeros(n, m.ld, device="cuda"), torch.zeros(n, device="cuda")
    h.grad(dev(X), dev(idx), G, loss)
    got = m.unpack(G.cpu().numpy())
    for i in range(n):
        g, l = orc.mlp_grad(m.unpack(X[i:i + 1])[0], dims, feat[i][idx[i]], labels[i][idx[i]])
        assert np.abs(got[i] - g).max() <= 1e-5 * np.abs(g).max()
        assert abs(float(loss[i]) - l) <= 1e-5 * max(abs(l), 1.0)
    assert np.count_nonzero(G.cpu().numpy()) == np.count_nonzero(got)  # padding untouched
    t, b = dev(1.0 + rng.random(n)), torch.ones(n, dtype=torch.int32, device="cuda")
    outs = []
    for fused in (True, False):
        h.set_fused_round(fused)
        Y, kept = dev(X), torch.zeros(len(col), dtype=torch.uint8, device="cuda")
        h.round(Y, t, b, 0.05, Y, kept, batch_idx=dev(idx), loss=loss)
        outs.append((Y, loss.clone()))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    assert h.status() == 0
    h.close()


# Workers, degree, columns; columns of a panel and blocks to an SM with gradients and without (tests/test_mix_pipe_cpu.py), 0: the plain kernel.
PIPE_SHAPES = [(5, 2, 4_200_001, (256, 2, 256, 2)), (17, 4, 1_250_000, (128, 2, 128, 2)), (33, 4, 640_003, (64, 2, 64, 2)),
               (70, 32, 300_000, (64, 2, 64, 2)),                              # a long plan
               (129, 8, 165_001, (32, 2, 64, 2)), (200, 6, 110_002, (32, 2, 64, 2)),
               (257, 8, 85_000, (32, 1, 32, 2)),                               # two boxes of rows
               (400, 6, 53_000, (32, 1, 64, 1)), (439, 6, 19_000, (0, 0, 32, 1)), (750, 4, 20_000, (0, 0, 32, 1))]


@pytest.mark.parametrize("n,deg,d", [c[:3] for c in PIPE_SHAPES])
@pytest.mark.parametrize("order", ["local_then_mix", "mix_then_correct"])
def test_pipelined_panel_mix_gives_the_bits_of_the_plain_one(n, deg, d, order):
    """The panel mix with its next panels on their way, at the edges of its panel widths: with and without gradients, with a learning rate per
    worker and in place, against the plain panel kernel (asked for by its width) bit for bit."""
    p = _dbw()
    rowptr, col = wl.ring(n) if deg == 2 else wl.random_regular(n, deg, 3)
    h = p.Dbw(rowptr, col, d=d, flags=p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    gen = torch.Generator(device="cuda").manual_seed(n)
    X, G = (torch.randn(n, h.ld, device="cuda", generator=gen) for _ in range(2))
    lr = torch.rand(n, device="cuda", generator=gen)
    t = torch.rand(n, device="cuda", generator=gen, dtype=torch.float64)
    b = torch.randint(0, deg, (n,), device="cuda", generator=gen, dtype=torch.int32)
    kept = torch.zeros(len(col), dtype=torch.uint8, device="cuda")
    h.select(t, b, kept)
    for g, rate in ((G, None), (G, lr), (None, None)):
        want, got = torch.empty_like(X), torch.empty_like(X)
        h.set_mix_panel(16)
        h.mix(X, g, kept, b, 0.05, want, lr_per_worker=rate)
        h.set_mix_panel(0)
        h.mix(X, g, kept, b, 0.05, got, lr_per_worker=rate)
        assert torch.equal(got, want)
        Y = X.clone()
        h.mix(Y, g, kept, b, 0.05, Y, lr_per_worker=rate)
        assert torch.equal(Y, want)
    assert h.status() == 0
    h.close()


def _bf16_pieces(x, count):
    """float64 sums of the first `count` bf16 pieces of fp32 values."""
    rest, out = torch.from_numpy(np.ascontiguousarray(x)), 0.0
    for _ in range(count):
        piece = rest.bfloat16().float()
        rest, out = rest - piece, out + piece.double()
    return out.numpy()


def _few_product_errors(got, Z, T, counts):
    """Per count of non-zero rows in T's column groups: the errors of `got` and of fp32 multiply-adds in ascending k against float64 Z^T T, relative to
    the sum of the products' magnitudes, and those magnitudes."""
    Z64, T64, cols = Z.astype(np.float64), T.astype(np.float64), T.shape[1] // len(counts)
    ref, size, acc = Z64.T @ T64, np.abs(Z64).T @ np.abs(T64), np.zeros((Z.shape[1], T.shape[1]), np.float32)
    for k in range(Z.shape[0]):
        at = T[k] != 0
        acc[:, at] = (acc[:, at].astype(np.float64) + np.outer(Z64[k], T64[k, at])).astype(np.float32)
    out = []
    for g in range(len(counts)):
        sl = slice(g * cols, (g + 1) * cols)
        there = size[:, sl] > 0
        out.append([np.abs(a[:, sl].astype(np.float64) - ref[:, sl])[there] / size[:, sl][there] for a in (got, acc)] + [size[:, sl][there]])
    return out


def _check_few_products(got, Z, T, counts):
    for n, (mine, theirs, size) in zip(counts, _few_product_errors(got, Z, T, counts)):
        normal = size > 2.0 ** -125  # not a subnormal number
        if n == 1:  # one rounding, of a sum whose smaller part (2^-8 of it) is truncated a few times
            assert (mine - 2.0 ** -149 / size).max() <= 2.0 ** -24 * (1 + 2.0 ** -5)
        assert np.sqrt((mine[normal] ** 2).mean()) <= 1.001 * np.sqrt((theirs[normal] ** 2).mean()), (n, mine.max(), theirs.max())


@pytest.mark.parametrize("batch,tests,out,n", [(128, 384, 128, 8),    # whole tiles, a block to an SM
                                               (64, 192, 160, 24),    # ... five k steps in dA
                                               (64, 192, 128, 60),    # two blocks to an SM
                                               (97, 158, 131, 30),    # rows at every shift
                                               (27, 302, 131, 40),    # ... and dW of less than a step
                                               (130, 300, 27, 40)])   # ... and dA
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -112, 2.0 ** 118])  # ... whose last pieces are below the smallest bf16 number; whose sums overflow when scaled
def test_fp32_tensor_core_gemms_sum_few_products_as_multiply_adds_do(batch, tests, out, n, scale):
    """Sums of one, two and four non-zero products, and dense ones, are no less exact than fp32 multiply-adds in the tensor-core GEMMs: dW through
    sparse features, dA through sparse weights.  The GEMMs' other operand is read back exactly through one-hot samples and hidden units."""
    p = _dbw()
    rng = np.random.default_rng(11)
    rowptr, col = wl.ring(n)
    labels = rng.integers(0, 10, size=(n, batch)).astype(np.int32)
    idx = np.tile(np.arange(batch, dtype=np.int32), (n, 1))

    def sparse(k, counts):
        t = np.zeros((k, tests // len(counts) * len(counts)), np.float32)
        for c in range(t.shape[1]):
            at = rng.permutation(k)[: counts[c // (tests // len(counts))]]
            t[at, c] = rng.standard_normal(len(at)) * scale
        return t

    def gradients(dims, X, feat):
        m = p.model_layout(dims, batch)
        h = p.Dbw(rowptr, col, d=m.d, model=m)
        rows = np.zeros((n, m.ld), np.float32)
        for l, W in enumerate(X):
            rows[:, m.w_off[l]: m.w_off[l] + W[0].size] = W.reshape(n, -1)
            if l:
                rows[:, m.b_off[l - 1]: m.b_off[l - 1] + W.shape[2]] = float(l == len(X) - 1)
        f, lab, G = dev(feat), dev(labels), torch.zeros(n, m.ld, device="cuda")
        h.set_dataset(f, lab, batch)
        h.grad(dev(rows), dev(idx), G)
        assert h.status() == 0
        g = G.cpu().numpy()
        h.close()
        return [g[:, m.w_off[l]: m.w_off[l] + W[0].size].reshape(W.shape) for l, W in enumerate(X)]

    top = (0.2 * rng.standard_normal((n, 10, out))).astype(np.float32)
    counts = (1, 2, 4, batch)
    T = [sparse(batch, counts) for _ in range(n)]
    wide = batch + T[0].shape[1]
    first = np.zeros((n, out, wide), np.float32)
    first[:, :, :batch] = 0.1 * rng.standard_normal((n, out, batch))
    feat = np.stack([np.concatenate([np.eye(batch, dtype=np.float32), t], 1) for t in T])
    g = gradients([wide, out, 10], [first, top], feat)[0]
    Z = g[0, :, :batch].T
    _check_few_products(g[0, :, batch:], Z, T[0], counts)
    with pytest.raises(AssertionError):  # two pieces would not do
        _check_few_products((Z.astype(np.float64).T @ _bf16_pieces(T[0], 2)).astype(np.float32), Z, T[0], counts)

    counts = (1, 2, 4, out)
    T = [sparse(out, counts) for _ in range(n)]
    wide = batch + T[0].shape[1]
    hidden = np.full((n, wide, batch), 2.0 ** -126, np.float32)  # units that are active and weigh next to nothing in the next layer
    hidden[:, :batch] = np.eye(batch)
    second = np.concatenate([0.1 * rng.standard_normal((n, out, batch)), np.stack(T)], 2).astype(np.float32)
    g = gradients([batch, wide, out, 10], [hidden, second, top], np.tile(np.eye(batch, dtype=np.float32), (n, 1, 1)))
    _check_few_products(g[0][0, batch:].T, g[1][0, :, :batch], T[0], counts)


def test_fp32_tensor_core_gemms_with_outputs_that_are_not_finite():
    """A NaN, an infinity and values that overflow make the outputs they reach what multiply-adds make of them, leave the others alone, and do not
    take many times as long (a network that has diverged)."""
    p = _dbw()
    n, batch, dims = 12, 128, [300, 256, 200, 10]
    rowptr, col = wl.ring(n)
    m = p.model_layout(dims, batch)
    rng = np.random.default_rng(21)
    h = p.Dbw(rowptr, col, d=m.d, model=m)
    feat, labels = rng.random((n, batch, dims[0]), dtype=np.float32) + 0.1, rng.integers(0, 10, size=(n, batch)).astype(np.int32)
    X = m.pack((0.05 * rng.standard_normal((n, m.d))).astype(np.float32))
    for l in range(2):  # every unit active
        X[:, m.b_off[l]: m.b_off[l] + dims[l + 1]] = 9.0
    idx = np.tile(np.arange(batch, dtype=np.int32), (n, 1))

    def gradients(feat, X):
        f, lab, G, loss = dev(feat), dev(labels), torch.zeros(n, m.ld, device="cuda"), torch.zeros(n, device="cuda")
        h.set_dataset(f, lab, batch)
        x, ix = dev(X), dev(idx)
        h.grad(x, ix, G, loss)
        best = 1e9
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(5):
                h.grad(x, ix, G, loss)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        g = G.cpu().numpy()
        return [g[:, m.w_off[l]: m.w_off[l] + dims[l] * dims[l + 1]].reshape(n, dims[l + 1], dims[l]) for l in range(3)], best

    plain, usual = gradients(feat, X)
    # a feature of one sample: the column of dW that it is multiplied into (its weights are zero, so nothing else is reached)
    X0, bad = X.copy(), feat.copy()
    X0[:, m.w_off[0]: m.w_off[0] + dims[0] * dims[1]].reshape(n, dims[1], dims[0])[:, :, 7] = 0.0
    want, _ = gradients(feat, X0)
    for value in (3e38, -1e35):  # above the largest bf16; scaled, infinite
        bad[2, 5, 7] = value
        got, _ = gradients(bad, X0)
        z = got[0][2, :, 7].astype(np.float64)
        ref = want[0][2, :, 7].astype(np.float64)
        assert np.isfinite(z).all() and np.abs(z - ref).max() > 1e30
        assert np.array_equal(got[0][[i for i in range(n) if i != 2]], want[0][[i for i in range(n) if i != 2]])
        others = np.arange(dims[0]) != 7
        assert np.abs(got[0][2][:, others] - want[0][2][:, others]).max() <= 1e-6 * np.abs(want[0][2]).max()
        dz = z / value  # dZ of that sample, up to the rounding of one product and the other samples' share
        bad[2, 5, 7] = value / 4
        again, _ = gradients(bad, X0)
        assert np.abs(again[0][2, :, 7] / (value / 4) - dz).max() <= 2.0 ** -22 * np.abs(dz).max()
    # a weight of the second layer, in dA (times every dZ) and, through NaN logits, in every dZ
    for value in (np.nan, np.inf):
        X1 = X.copy()
        X1[3, m.w_off[1] + 4] = value
        got, _ = gradients(feat, X1)
        if np.isinf(value):
            assert not np.isfinite(got[0][3]).any()
        else:  # a NaN is no activation, so it is in that one unit's dZ alone
            assert np.isnan(got[0][3][4]).all() and np.isfinite(np.delete(got[0][3], 4, 0)).all()
        assert all(np.array_equal(got[l][i], plain[l][i]) for l in range(3) for i in range(n) if i != 3)
    X1 = X.copy()
    X1[:, m.w_off[2]] = np.nan
    got, time = gradients(feat, X1)
    assert all(np.isnan(g[g0 != 0]).all() for g, g0 in zip(got, plain))
    assert time <= 4 * usual, (time, usual)
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("n,deg,d,order", [(24, 4, 3_800_000, "local_then_mix"), (65, 6, 1_500_003, "mix_then_correct"), (224, 4, 420_000, "local_then_mix")])
def test_pipelined_panel_mix_leaves_rounds_with_few_kept_neighbours_to_the_plain_one(n, deg, d, order):
    """Matrices large enough for both kernels to be launched: nothing kept, one neighbour less than the line, the line, everything; in place and
    out of place, against the plain panel kernel bit for bit."""
    p = _dbw()
    rowptr, col = wl.random_regular(n, deg, 3)
    h = p.Dbw(rowptr, col, d=d, flags=p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    assert n * h.ld * 12 >= 1 << 30
    gen = torch.Generator(device="cuda").manual_seed(n)
    X, G = (torch.randn(n, h.ld, device="cuda", generator=gen) for _ in range(2))
    want, got = torch.empty_like(X), torch.empty_like(X)
    kept = torch.zeros(len(col), dtype=torch.uint8, device="cuda")
    t = torch.rand(n, device="cuda", generator=gen, dtype=torch.float64)
    line = (n + 1) // 2
    for total in (0, line - 1, line, n * deg):
        b = torch.full((n,), deg, dtype=torch.int32, device="cuda")
        if total == n * deg:
            b.zero_()
        else:
            b[torch.randperm(n, device="cuda", generator=gen)[:total]] -= 1
        h.select(t, b, kept)
        assert int(kept.sum()) == total
        h.set_mix_panel(16)
        h.mix(X, G, kept, b, 0.05, want)
        h.set_mix_panel(0)
        got.zero_()
        h.mix(X, G, kept, b, 0.05, got)
        assert torch.equal(got, want), total
        got.copy_(X)
        h.mix(got, G, kept, b, 0.05, got)
        assert torch.equal(got, want), total
    assert h.status() == 0
    h.close()


@pytest.mark.parametrize("order", ["local_then_mix", "mix_then_correct"])
@pytest.mark.parametrize("n,dims", [(20, [3072, 304, 10]), (96, [3072, 64, 10]), (210, [1024, 120, 10])])  # panels of 128, 64 and 32 columns
def test_pipelined_panel_mix_in_tensor_core_rounds(n, dims, order):
    """Rounds whose mix is the pipeline's where more than half of the workers take part and another kernel's where fewer do, with the bf16 copy of
    the parameters that the next round reads: against rounds on the plain panel kernel bit for bit, in place and out of place."""
    p = _dbw()
    batch = 8
    rowptr, col = wl.ring(n)
    m = p.model_layout(dims, batch)
    flags = p.GEMM_BF16 | (p.ORDER_MIX_THEN_CORRECT if order == "mix_then_correct" else 0)
    assert 12 * n * m.ld >= 160 << 20
    gen = torch.Generator(device="cuda").manual_seed(n)
    feat = torch.rand(n, batch, dims[0], device="cuda", generator=gen)
    labels = torch.randint(0, 10, (n, batch), device="cuda", generator=gen, dtype=torch.int32)
    idx = torch.arange(batch, device="cuda", dtype=torch.int32).repeat(n, 1)
    t = 1.0 + torch.rand(n, device="cuda", generator=gen, dtype=torch.float64)
    everyone = torch.zeros(n, dtype=torch.int32, device="cuda")
    few = torch.where(torch.arange(n, device="cuda") < n // 6, 1, 2).int()
    X0 = torch.zeros(n, m.ld, device="cuda")
    for l in range(2):
        X0[:, m.w_off[l]: m.w_off[l] + dims[l] * dims[l + 1]].normal_(0.0, 0.03, generator=gen)
    outs = []
    for panel in (0, 16):
        h = p.Dbw(rowptr, col, d=m.d, model=m, flags=flags)
        h.set_dataset(feat, labels, batch)
        h.set_mix_panel(panel)
        h.set_param_tracking(True)
        kept, loss = torch.zeros(len(col), dtype=torch.uint8, device="cuda"), torch.zeros(n, device="cuda")
        X, Y, got = X0.clone(), torch.zeros_like(X0), []
        for b in (everyone, few, everyone, everyone):
            out = X if len(got) == 2 else Y
            h.round(X, t, b, 0.05, out, kept, batch_idx=idx, loss=loss)
            got.append((out.clone(), loss.clone()))
            X, Y = out, (Y if out is X else X)
        assert h.status() == 0
        h.close()
        outs.append(got)
    for (x, l), (y, k) in zip(*outs):
        assert torch.equal(x, y) and torch.equal(l, k)
