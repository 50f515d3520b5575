"""Kernels at the sizes and alignments where their tiles, chunks and vector
accesses end, against plain float64 results; the bounds follow from the
arithmetic (float32 chains, the FP16 split) and are stated with each test."""
import types

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cq():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_05836_gb300 import cutqc
    return cutqc


def _pair(oa, ob, k, qa=None):
    """Two subcircuits over k cuts, A measured and B initialised; qa: the
    uncut qubits of A's outputs (default: the highest)."""
    qa = list(range(ob, ob + oa)) if qa is None else list(qa)
    qb = [q for q in range(oa + ob) if q not in qa]
    e = list(range(k))
    a = types.SimpleNamespace(w=oa + k, in_local=[], out_local=list(range(oa, oa + k)), in_edge=[], out_edge=e, out_qubit=qa)
    b = types.SimpleNamespace(w=ob, in_local=list(range(k)), out_local=[], in_edge=e, out_edge=[], out_qubit=qb)
    return [a, b], qa, qb


def _place(p, qa, qb):
    """[2^oa, 2^ob] -> uncut qubit order."""
    def dep(qs):
        r = np.arange(1 << len(qs))
        return sum((((r >> j) & 1) << q for j, q in enumerate(qs)), np.zeros_like(r))
    out = np.empty(p.size)
    out[dep(qa)[:, None] | dep(qb)[None, :]] = p
    return out


def _operands(torch, oa, ob, k, seed, shift=0):
    """Random attributed tensors on the device, `shift` floats past a 16-byte
    boundary, and their float64 copies."""
    rng = np.random.default_rng(seed)
    dev, host = [], []
    for o in (oa, ob):
        x = rng.standard_normal((1 << o, 4 ** k)).astype(np.float32)
        buf = torch.empty(x.size + 4, dtype=torch.float32, device="cuda")
        t = buf[shift:shift + x.size].view(x.shape)
        t.copy_(torch.from_numpy(x))
        dev.append(t)
        host.append(x.astype(np.float64))
    return dev, host


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("oa,ob,k", [(10, 9, 1), (3, 16, 2), (9, 10, 3), (7, 13, 4), (14, 6, 4), (3, 16, 5), (11, 11, 1),
                                     (11, 11, 3)])
def test_fp32_gemm_tiles(cq, oa, ob, k, shift):
    """The FP32 GEMM (steps past the small one-launch kernel) with fewer rows
    or columns than a 64 x 64 and a 128 x 128 tile, fewer and more values than
    a 16-value chunk, few and many tiles (256 of 128 x 128 in the last two), aligned and unaligned operands and outputs (scalar loads and
    stores), Kronecker and interleaved orders.  Bound: the float32 chain of
    4^k terms, (4^k + 2) 2^-24 of the absolute terms, per output."""
    import torch
    dev, (A, B) = _operands(torch, oa, ob, k, 100 * oa + 10 * ob + k, shift)
    for qa in (None, range(0, 2 * oa, 2) if ob >= oa - 1 else None):
        if qa is None and k == 1 and oa + ob >= 22:
            continue                # row-major outputs of few terms take the outer-product kernel
        subs, la, lb = _pair(oa, ob, k, qa)
        assert sorted(la + lb) == list(range(oa + ob))
        buf = torch.full(((1 << (oa + ob)) + 8,), 7.0, dtype=torch.float32, device="cuda")
        out = buf[shift:shift + (1 << (oa + ob))]
        total = torch.zeros(1, dtype=torch.float64, device="cuda")
        cq.cutqc_reconstruct_fd(subs, dev, cq.ORDER_ORIGINAL, cq.PREC_FP32_SIMT, out=out, sum_out=total)
        torch.cuda.synchronize()
        ref = _place(A @ B.T * 2.0 ** -k, la, lb)
        tol = _place((4 ** k + 2) * 2.0 ** -24 * (np.abs(A) @ np.abs(B).T) * 2.0 ** -k, la, lb)
        got = out.cpu().numpy().astype(np.float64)
        assert (np.abs(got - ref) <= tol).all()
        # nothing written around the output
        assert bool((buf[:shift] == 7.0).all()) and bool((buf[shift + got.size:] == 7.0).all())
        # the float64 total of the written floats: 128 of them in float32 first
        assert abs(total.item() - got.sum()) <= 130 * 2.0 ** -24 * np.abs(got).sum()


def _mlp_setup(cq, torch, B, seed, shift=0):
    """Network, inputs and targets; shift: floats (and BF16 values) past a
    16-byte boundary of every array."""
    rng = np.random.default_rng(seed)
    flat = cq.init_params(seed) + (rng.standard_normal(82689) * 0.05).astype(np.float32)
    net = cq.MLP(flat)
    def moved(t):
        buf = torch.empty(t.numel() + 8, dtype=t.dtype, device="cuda")
        v = buf[shift:shift + t.numel()].view(t.shape)
        v.copy_(t)
        return v
    if shift:
        net.p, net.pb = moved(net.p), moved(net.pb)
    x = moved(torch.from_numpy(rng.standard_normal((B, 64)).astype(np.float32)).cuda())
    t = moved(torch.from_numpy(rng.standard_normal(B).astype(np.float32)).cuda())
    return net, x, t


@pytest.mark.parametrize("B,shift", [(7, 1), (95, 0), (97, 0), (300, 1), (1217, 0), (2500, 1), (6001, 0)])
def test_mlp_row_tiles_and_batch_slices(cq, B, shift):
    """Scores and gradients of batches that take 8, 16 and 32 rows per tile,
    one and several tiles per CTA, one and several batch slices, aligned and
    unaligned arrays, against the same rows taken 8 at a time or fewer (one
    tile, one slice: the form the oracle tests check).  Hidden values are the
    same fmaf chains in every form, so scores are equal up to nothing and the
    ReLU masks too; gradients differ by the order of a float32 sum over the
    batch: at most (B + 8) 2^-23 of the absolute terms."""
    import torch
    net, x, t = _mlp_setup(cq, torch, B, 40 + B, shift)
    y = net.forward(x)
    grad, loss = net.gradients(x, t)
    grad, loss = grad.double().cpu().numpy(), loss.item()
    acc, ref_loss = np.zeros_like(grad), 0.0
    for b in range(0, B, 8):
        xs, ts = x[b:b + 8].clone(), t[b:b + 8].clone()
        assert torch.equal(net.forward(xs), y[b:b + 8])
        g, l = net.gradients(xs, ts)
        acc += g.double().cpu().numpy() * (len(ts) / B)
        ref_loss += l.item() * len(ts) / B
    # absolute terms, in float64
    W1, b1, W2, b2, W3, b3 = [w.double() for w in _split(cq, net)]
    X = x.double()
    h1 = (X @ W1 + b1).clamp_min(0)
    h2 = (h1 @ W2 + b2).clamp_min(0)
    dy = ((h2 @ W3 + b3).reshape(-1) - t.double()).abs().reshape(-1, 1) * 2 / B
    g2 = dy @ W3.abs().T
    g1 = g2 @ W2.abs().T
    bound = torch.cat([q.reshape(-1) for q in (X.abs().T @ g1, g1.sum(0), h1.T @ g2, g2.sum(0), h2.T @ dy, dy.sum(0))])
    assert (np.abs(grad - acc) <= (B + 8) * 2.0 ** -23 * bound.cpu().numpy() + 1e-30).all()
    assert abs(loss - ref_loss) <= 1e-12 * ref_loss + 1e-30


def _split(cq, net):
    """Weights as the kernels read them (BF16 values), FP32 biases."""
    out, o = [], 0
    for a, b in ((64, 256), (256, 256), (256, 1)):
        out.append(net.pb[o:o + a * b].float().view(a, b))
        out.append(net.p[o + a * b:o + a * b + b])
        o += a * b + b
    return out


def _orders(oa, ob):
    """Uncut qubits of A's outputs: runs of 1, 2, 3 and 6 from either operand
    first, and two random splits."""
    n = oa + ob
    out = []
    for run in (1, 2, 3, 6):
        for first in (0, 1):
            a, b, q = [], [], 0
            side = first
            while q < n:
                mine, most = ((a, oa), (b, ob))[side]
                for _ in range(min(run, most - len(mine))):
                    mine.append(q)
                    q += 1
                side ^= 1
            out.append(a)
    rng = np.random.default_rng(n)
    out += [sorted(rng.permutation(n)[:oa].tolist()) for _ in range(2)]
    return [list(x) for x in sorted({tuple(x) for x in out})]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("oa,ob,k", [(9, 10, 2), (3, 16, 3), (10, 10, 4), (3, 17, 4), (16, 4, 4), (1, 19, 4), (9, 10, 5),
                                     (13, 5, 5), (4, 12, 6), (8, 14, 5), (13, 9, 5), (10, 12, 6)])
def test_tensor_core_outputs_in_any_qubit_order(cq, oa, ob, k, shift):
    """The tensor-core GEMMs (4^k <= 256 terms on SM pairs with A resident,
    more on single SMs or, from 2^22 outputs here, on pairs) storing in orders where the low output bits come from either operand
    or both: register stores of 8-column sectors, staged whole lines, fewer
    rows or columns than a tile, at 4-byte aligned outputs too.  Bound per output: the
    split's 3 2^-22 and the accumulation's truncations, together under 2^-18
    of the absolute terms, and 2^-39 of the subnormal low parts' terms
    (largest entry times the other row's absolute sum); doubled."""
    import torch
    dev, (A, B) = _operands(torch, oa, ob, k, 7 * oa + 11 * ob + k)
    A[1] *= 2.0 ** -12          # rows of different scales
    dev[0].copy_(torch.from_numpy(A.astype(np.float32)))
    P = A @ B.T * 2.0 ** -k
    L1a, L1b = np.abs(A).sum(1), np.abs(B).sum(1)
    tol = 2.0 ** -k * 2 * (2.0 ** -18 * (np.abs(A) @ np.abs(B).T) +
                           2.0 ** -39 * (L1a[:, None] * np.abs(B).max() + L1b[None, :] * np.abs(A).max()))
    for qa in _orders(oa, ob):
        subs, la, lb = _pair(oa, ob, k, qa)
        if shift and (la == list(range(ob, ob + oa)) or lb == list(range(oa, oa + ob))):
            continue        # row-major outputs start 16-byte aligned
        n = 1 << (oa + ob)
        buf = torch.full((n + 8,), 7.0, dtype=torch.float32, device="cuda")
        out = buf[shift:shift + n]
        total = torch.zeros(1, dtype=torch.float64, device="cuda")
        cq.cutqc_reconstruct_fd(subs, dev, cq.ORDER_ORIGINAL, cq.PREC_FP16X3_TC, out=out, sum_out=total)
        torch.cuda.synchronize()
        got = out.cpu().numpy().astype(np.float64)
        assert (np.abs(got - _place(P, la, lb)) <= _place(tol, la, lb)).all(), qa
        assert bool((buf[:shift] == 7.0).all()) and bool((buf[shift + n:] == 7.0).all())
        # float32 partial sums of at most 2048 outputs, then float64
        assert abs(total.item() - got.sum()) <= 2048 * 2.0 ** -24 * np.abs(got).sum()
    assert cq.cutqc_device_status() == 0


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("oa,ob,k", [(0, 1, 1), (1, 1, 1), (2, 3, 2), (4, 4, 3), (5, 4, 4), (3, 5, 5), (7, 8, 2), (8, 8, 4),
                                     (5, 12, 3), (12, 5, 5), (9, 9, 4)])
def test_small_steps_in_one_launch(cq, oa, ob, k, precision):
    """The one-launch kernel of small steps below, at and above its 16 x 16
    and 32 x 32 tiles and its 256- and 128-value chunks, in several qubit
    orders, whole and as row ranges.  Bound: float32 chains of 4^k terms in
    at most 16 groups, (4^k + 18) 2^-24 of the absolute terms."""
    import torch
    dev, (A, B) = _operands(torch, oa, ob, k, 5 * oa + 3 * ob + k, 1)
    P = A @ B.T * 2.0 ** -k
    tol = (4 ** k + 18) * 2.0 ** -24 * (np.abs(A) @ np.abs(B).T) * 2.0 ** -k
    n = 1 << (oa + ob)
    for qa in _orders(oa, ob)[:4]:
        subs, la, lb = _pair(oa, ob, k, qa)
        buf = torch.full((n + 8,), 7.0, dtype=torch.float32, device="cuda")
        total = torch.zeros(1, dtype=torch.float64, device="cuda")
        launches = cq.cutqc_kernel_launches()
        cq.cutqc_reconstruct_fd(subs, dev, cq.ORDER_ORIGINAL, precision, out=buf[4:4 + n], sum_out=total)
        assert cq.cutqc_kernel_launches() - launches == 1
        got = buf[4:4 + n].cpu().numpy().astype(np.float64)
        assert (np.abs(got - _place(P, la, lb)) <= _place(tol, la, lb)).all(), qa
        assert bool((buf[:4] == 7.0).all()) and bool((buf[4 + n:] == 7.0).all())
        assert abs(total.item() - got.sum()) <= 8 * 2.0 ** -24 * np.abs(got).sum()
    subs, _, _ = _pair(oa, ob, k)
    rows, cols = cq.cutqc_fd_shape(subs)
    for r0, r1 in ((0, rows // 2), (rows // 2, rows), (rows - 1, rows)):
        if r1 > r0:
            out, _ = cq.cutqc_reconstruct_fd(subs, dev, cq.ORDER_KRON, precision, r0, r1)
            got = out.view(-1, cols).cpu().numpy()
            assert (np.abs(got - P.reshape(rows, cols)[r0:r1]) <= tol.reshape(rows, cols)[r0:r1]).all()


@pytest.mark.parametrize("oa,ob,k", [(15, 7, 0), (14, 8, 1), (13, 9, 2), (12, 10, 1), (11, 11, 0), (10, 12, 1), (8, 14, 1),
                                     (7, 15, 2), (5, 17, 0)])
def test_outer_products_at_every_width(cq, oa, ob, k):
    """Row-major last steps over 1, 4 and 16 terms at 2^22 outputs: columns
    from one warp per row (128) over the widest tile (4096 columns, 1024 at
    16 terms) to many tiles, rows down to one group of 32, rows in order and
    permuted.  Bound: float32 chains, (4^k + 2) 2^-24 of the absolute terms."""
    import torch
    dev, (A, B) = _operands(torch, oa, ob, k, 13 * oa + k)
    P = A @ B.T * 2.0 ** -k
    tol = (4 ** k + 2) * 2.0 ** -24 * (np.abs(A) @ np.abs(B).T) * 2.0 ** -k
    subs, _, _ = _pair(oa, ob, k)
    for perm in (False, True):
        order = np.arange(oa)
        if perm:
            order = np.random.default_rng(oa).permutation(oa)
            subs[0].out_qubit = (ob + order).tolist()
        buf = torch.full(((1 << 22) + 8,), 7.0, dtype=torch.float32, device="cuda")
        total = torch.zeros(1, dtype=torch.float64, device="cuda")
        cq.cutqc_reconstruct_fd(subs, dev, cq.ORDER_ORIGINAL, cq.PREC_FP32_SIMT, out=buf[4:4 + (1 << 22)], sum_out=total)
        got = buf[4:4 + (1 << 22)].cpu().numpy().astype(np.float64)
        rows = np.arange(1 << oa)
        at = sum((((rows >> j) & 1) << int(order[j]) for j in range(oa)), np.zeros_like(rows))
        got = got.reshape(1 << oa, 1 << ob)[at]
        assert (np.abs(got - P) <= tol).all()
        assert bool((buf[:4] == 7.0).all()) and bool((buf[4 + (1 << 22):] == 7.0).all())
        # at most 512 outputs per float32 partial sum
        assert abs(total.item() - got.sum()) <= 512 * 2.0 ** -24 * np.abs(got).sum()


@pytest.mark.parametrize("kin,kout,w", [(1, 1, 2), (1, 1, 9), (1, 1, 12), (2, 2, 5), (3, 1, 8), (4, 2, 9), (4, 2, 11), (2, 3, 10),
                                        (1, 4, 6), (4, 4, 6), (5, 1, 7), (2, 0, 3), (3, 0, 9), (4, 0, 5), (4, 0, 10)])
def test_attribution_items_and_fibers(cq, kin, kout, w):
    """The measured side with several (state, row) items per thread (fewer
    and more rows than a CTA's items, whole blocks of states), and the
    initialised side in register steps (2 to 4 cuts on the lowest columns,
    fewer and more fibers than a CTA's) or along the columns (the edges the
    other way round), aligned and unaligned outputs.  Every entry written and
    within the float32 rounding of the sums (2^kout terms, then at most 4 per
    initialised cut) of the oracle."""
    import torch
    from oracle import attribution
    rng = np.random.default_rng(100 * kin + 10 * kout + w)
    o = w - kout
    var = rng.uniform(0.0, 1.0, size=(4 ** kin, 3 ** kout, 2 ** w))
    tol = (kout + 3 * kin + 2) * 2.0 ** (kout + 2 * kin - 24)
    for low in (True, False):
        out_local = list(range(o, w)) if low else sorted(rng.choice(w, size=kout, replace=False).tolist())
        in_local = sorted(rng.choice(w, size=min(kin, w), replace=False).tolist())
        if len(in_local) < kin:
            continue
        ein, eout = rng.permutation(kin), rng.permutation(kout)
        ein, eout = (ein, kin + eout) if low else (kout + ein, eout)
        sub = types.SimpleNamespace(w=w, in_local=in_local, out_local=out_local, in_edge=ein.tolist(),
                                    out_edge=eout.tolist(), out_qubit=list(range(o)))
        ref = attribution.attribute(var, w, in_local, out_local, sub.in_edge, sub.out_edge)
        for dtype, shift in ((torch.float64, 0), (torch.float32, 0), (torch.float64, 1)):
            buf = torch.full((ref.size + 8,), float("nan"), dtype=torch.float32, device="cuda")
            out = buf[shift:shift + ref.size].view(ref.shape)
            cq.cutqc_attribute(sub, torch.from_numpy(var).cuda().to(dtype), out=out)
            got = out.double().cpu().numpy()
            assert np.abs(got - ref).max() <= tol, (low, dtype, shift)
            assert torch.isnan(buf[:shift]).all() and torch.isnan(buf[shift + ref.size:]).all()


@pytest.mark.parametrize("n,M,T", [(90, 10, 4), (67, 7, 2), (128, 13, 3)])
def test_dd_children_beyond_64_qubits(cq, n, M, T):
    """Algorithm 1 down a chain of sparse subcircuits, with levels whose
    active qubits end at, straddle and start beyond qubit 64 (the zoom words
    meet there) and GEMM tiles of few rows and columns: the level-by-level
    and the one-launch records equal the float64 oracle's.  Bound of the
    bins: all terms are >= 0 and at most 5 % of 2^o, each sum one rounding
    per nonzero term, one sum per subcircuit, then 4 terms per cut."""
    import torch
    from oracle import dd
    rng = np.random.default_rng(n)
    o = [15] * (n // 15) + ([n % 15] if n % 15 else [])
    subs, A, q = [], [], 0
    for i, w in enumerate(o):
        edges = [e for e in (i - 1, i) if 0 <= e < len(o) - 1]
        x = np.exp(2.0 * rng.standard_normal((1 << w, 4 ** len(edges)))) * (rng.random((1 << w, 4 ** len(edges))) < 0.05)
        A.append((x / x.sum()).astype(np.float32).astype(np.float64))
        subs.append(types.SimpleNamespace(w=w + (i < len(o) - 1), in_local=[0] if i else [], in_edge=[i - 1] if i else [],
                                          out_local=[w] if i < len(o) - 1 else [], out_edge=[i] if i < len(o) - 1 else [],
                                          out_qubit=list(range(q, q + w)), edges=edges, o=w))
        q += w
    R = -(-n // M)
    ref = dd.run(A, [s.out_qubit for s in subs], [s.edges for s in subs], len(o) - 1, n, M, R, T, strategy="bfs")
    At = [torch.from_numpy(a.astype(np.float32)).cuda() for a in A]
    jobs, n_jobs, bins = cq.cutqc_dd_run_async(subs, At, n, M, R, T)
    run = cq.dd_batch_run(subs, At, n, M, R, T, max_jobs=len(ref) + 8)
    cq.cutqc_dd_batch_create([run]).launch()
    torch.cuda.synchronize()
    rel = (len(o) * 0.06 * 2 ** 15 + 4 * len(o)) * 2.0 ** -24
    for got, b in ((cq.dd_jobs_from_device(jobs, n_jobs), bins), (cq.dd_jobs_from_device(run["jobs"], run["n_jobs"]), run["bins"])):
        assert len(got) == len(ref)
        for J, r in zip(got, ref):
            assert list(J.active[:J.n_active]) == r["active"]
            assert J.zoom() == r["zoom"]
            x = b[J.bins_offset:J.bins_offset + (1 << J.n_active)].cpu().numpy().astype(np.float64)
            assert (np.abs(x - r["bins"]) <= rel * r["bins"] + 1e-37).all()
    assert cq.cutqc_device_status() == 0


def test_mlp_inputs_of_every_class(cq):
    """Rows of ordinary, subnormal, tiny, huge, infinite and NaN inputs, each
    alone among ordinary rows: finite scores within the float32 rounding of
    the layers' sums (64, 256 and 256 terms, twice over), the others of the
    class of the float32 formula with fmax as the ReLU; neighbours unchanged."""
    import torch
    net, x, _ = _mlp_setup(cq, torch, 40, 5, 0)
    plain = net.forward(x).clone()
    rows = {3: 1e-40, 9: 1e-30, 10: 2.0 ** 100, 17: float("inf"), 18: float("-inf"), 25: float("nan")}
    for r, v in rows.items():
        x[r, r % 7] = v
    x[30] = torch.linspace(-1, 1, 64, device="cuda") * 1e-38
    x[31] *= 2.0 ** 90
    y = net.forward(x)
    W1, b1, W2, b2, W3, b3 = [w.double() for w in _split(cq, net)]
    zero = torch.zeros((), dtype=torch.float64, device="cuda")
    X = x.double()
    ref = (torch.fmax(torch.fmax(X @ W1 + b1, zero) @ W2 + b2, zero) @ W3 + b3).reshape(-1)
    size = (((X.abs() @ W1.abs() + b1.abs()) @ W2.abs() + b2.abs()) @ W3.abs() + b3.abs()).reshape(-1)
    ok = torch.isfinite(size)
    assert int(ok.sum()) == 37
    assert bool(((y.double() - ref).abs() <= 2 * 576 * 2.0 ** -24 * size + 1e-30)[ok].all())
    for r in (17, 18, 25):
        a, b = y[r].item(), ref[r].item()
        assert np.isnan(a) == np.isnan(b) and np.isinf(a) == np.isinf(b) and (not np.isinf(a) or (a > 0) == (b > 0))
    same = [r for r in range(40) if r not in rows and r not in (30, 31)]
    assert torch.equal(y[same], plain[same])


@pytest.mark.parametrize("oa,ob,k", [(9, 12, 3), (10, 12, 4), (12, 13, 5)])
def test_dependent_launches_in_graphs_and_on_streams(cq, oa, ob, k):
    """The tensor-core step's launches (the column operand's max pass with the
    row operand's preparation beside it, dependent preparation and GEMM):
    replayed from a graph on new inputs, right behind the kernels that write
    them, and from two streams at once, each with its own buffers.  Equal to
    the eager result bit for bit."""
    import torch
    subs, _, _ = _pair(oa, ob, k)
    need = max(1, cq.cutqc_reconstruct_fd_workspace_size(subs, cq.PREC_FP16X3_TC))
    sets = []
    for seed in range(2):
        dev, _ = _operands(torch, oa, ob, k, 70 + seed)
        sets.append((dev, torch.empty(1 << (oa + ob), device="cuda"), torch.empty(need, dtype=torch.uint8, device="cuda")))

    def run(att, out, ws):
        cq.cutqc_reconstruct_fd(subs, att, cq.ORDER_KRON, cq.PREC_FP16X3_TC, out=out, ws=ws)

    eager = []
    for scale in (1.0, 3.0):
        for att, out, ws in sets:
            run([a * scale for a in att], out, ws)
            torch.cuda.synchronize()
            eager.append(out.clone())
    att, out, ws = sets[0]
    work = [torch.empty_like(a) for a in att]
    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        run(att, out, ws)
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        for w, a in zip(work, att):
            torch.mul(a, 3.0, out=w)
        run(work, out, ws)
    for _ in range(3):
        out.fill_(-1.0)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, eager[2])
    streams = [torch.cuda.Stream() for _ in sets]
    for rep in range(8):
        for st, (att, out, ws) in zip(streams, sets):
            with torch.cuda.stream(st):
                if rep == 0:
                    out.fill_(-1.0)
                run(att, out, ws)
    torch.cuda.synchronize()
    for i, (att, out, ws) in enumerate(sets):
        assert torch.equal(out, eager[i])
    assert cq.cutqc_device_status() == 0


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_whole_row_range_in_uncut_order(cq, precision):
    """The whole row range given by its end, for the operand of the highest
    output bit in the rows and (it holds output bit 0 too) in the columns of
    the last step: the result of row_end = -1."""
    import torch
    dev, _ = _operands(torch, 12, 10, 4, 3)
    for qa in (list(range(10, 22)), [0, 1, 2] + list(range(13, 22))):
        subs, _, _ = _pair(12, 10, 4, qa)
        rows, _ = cq.cutqc_fd_shape(subs)
        whole, _ = cq.cutqc_reconstruct_fd(subs, dev, cq.ORDER_ORIGINAL, precision)
        out = torch.full_like(whole, 7.0)
        cq.cutqc_reconstruct_fd(subs, dev, cq.ORDER_ORIGINAL, precision, 0, rows, out=out)
        assert torch.equal(out, whole)


def test_fp32_columns_past_the_row_limit_in_uncut_order(cq):
    """A row operand of few outputs that holds the lowest and the highest
    output bit against 2^24 columns (more than the FP32 GEMM takes as rows).
    Bound: the float32 chain, (4 + 2) 2^-24 of the absolute terms."""
    import torch
    dev, _ = _operands(torch, 3, 24, 1, 9)
    subs, _, _ = _pair(3, 24, 1, [0, 1, 26])
    out, _ = cq.cutqc_reconstruct_fd(subs, dev, cq.ORDER_ORIGINAL, cq.PREC_FP32_SIMT)
    A, B = (x.double() for x in dev)
    got = out.view(2, 1 << 24, 4)
    for top in range(2):
        a = A[4 * top:4 * top + 4]
        err = (got[top].double() - B @ a.T / 2).abs()
        assert bool((err <= 6 * 2.0 ** -24 * (B.abs() @ a.abs().T) / 2).all())


# Equal outputs: every add of a float32 chain then rounds the same way.
_EQUAL = (1.1, 1.3, 1.7, 0.7)


@pytest.mark.parametrize("oa,ob,k", [(14, 8, 0), (14, 8, 2), (12, 10, 1), (11, 11, 0), (10, 12, 1), (9, 14, 0), (8, 14, 1),
                                     (7, 15, 2)])
def test_outer_product_totals_of_equal_outputs(cq, oa, ob, k):
    """The float64 total of outer-product steps at every width of its tiles
    (one, two and four column groups per thread, one to sixteen rows at a
    time): at most 8 outputs are added in float32 (three roundings), the rest
    without rounding but for the float64 adds."""
    import torch
    subs, _, _ = _pair(oa, ob, k)
    for c in _EQUAL:
        A = torch.zeros((1 << oa, 4 ** k), device="cuda")
        B = torch.zeros((1 << ob, 4 ** k), device="cuda")
        A[:, 0], B[:, 0] = c, 2.0 ** k
        total = torch.zeros(1, dtype=torch.float64, device="cuda")
        out, _ = cq.cutqc_reconstruct_fd(subs, [A, B], cq.ORDER_KRON, cq.PREC_FP32_SIMT, sum_out=total)
        ref = out.double().sum().item()
        assert abs(ref - out.numel() * float(np.float32(c))) <= 1e-9 * ref
        assert abs(total.item() - ref) <= 3 * 2.0 ** -24 * ref, c


def _uneven(torch, oa, ob, k, big, small):
    """Operands whose product's rows are all 1 (where big(row)) or all
    `small`."""
    A = torch.zeros((1 << oa, 4 ** k), device="cuda")
    B = torch.zeros((1 << ob, 4 ** k), device="cuda")
    m = torch.arange(1 << oa, device="cuda")
    A[:, 0] = torch.where(big(m), 1.0, small)
    B[:, 0] = 2.0 ** k
    return A, B


@pytest.mark.parametrize("oa,ob,k,original,rounds", [(12, 11, 3, False, 3), (12, 11, 3, True, 3), (11, 12, 4, False, 3),
                                                     (13, 6, 4, False, 2), (6, 13, 4, True, 2)])
def test_fp32_gemm_totals_of_uneven_rows(cq, oa, ob, k, original, rounds):
    """The float64 total of FP32 steps in 128 x 128 tiles (16-byte and single
    stores) and 64 x 64 tiles, where the first of a thread's rows is 1 and the
    others are just below half the last place of four (or sixteen) ones: at
    most 8 and 4 outputs, of one row, are added in float32 (three and two
    roundings), the rest without rounding but for the float64 adds."""
    import torch
    n = oa + ob
    subs, _, _ = _pair(oa, ob, k, [2 * i + 1 for i in range(oa - 1)] + [n - 1] if original else None)
    A, B = _uneven(torch, oa, ob, k, lambda m: (m % 4 == 0) & (m // 64 % 2 == 0), 2.0 ** -24 * (1 - 2.0 ** -6))
    total = torch.zeros(1, dtype=torch.float64, device="cuda")
    out, _ = cq.cutqc_reconstruct_fd(subs, [A, B], cq.ORDER_ORIGINAL if original else cq.ORDER_KRON, cq.PREC_FP32_SIMT,
                                     sum_out=total)
    ref = (A[:, 0].double().sum() * 2.0 ** ob).item()
    assert abs(out.double().sum().item() - ref) <= 1e-12 * ref
    assert abs(total.item() - ref) <= rounds * 2.0 ** -24 * ref


@pytest.mark.parametrize("narrow", [-1, 16])
def test_dd_bin_totals_of_uneven_rows(cq, narrow):
    """The same for the bin totals of the level launches and of the persistent
    launch's 64 x 64 and 256 x 16 tiles: four bins of one row are added in
    float32 (two roundings), the rest without rounding but for the float64
    adds."""
    import torch
    subs, _, _ = _pair(8, 4, 1)
    A, B = _uneven(torch, 8, 4, 1, lambda m: m % 4 == 0, 2.0 ** -24 * (1 - 2.0 ** -6))
    run = cq.dd_batch_run(subs, [A, B], 12, 12, 1, 1, max_jobs=4)
    cq.cutqc_dd_batch_create([run], options={"narrow_max_n": narrow}).launch()
    jobs, n_jobs, bins = cq.cutqc_dd_run_async(subs, [A, B], 12, 12, 1, 1)
    torch.cuda.synchronize()
    ref = (A[:, 0].double().sum() * 2.0 ** 4).item()
    for J, b in ((cq.dd_jobs_from_device(run["jobs"], run["n_jobs"])[0], run["bins"]),
                 (cq.dd_jobs_from_device(jobs, n_jobs)[0], bins)):
        assert abs(b[:1 << 12].double().sum().item() - ref) <= 1e-12 * ref
        assert abs(J.bin_sum - ref) <= 2 * 2.0 ** -24 * ref


@pytest.mark.parametrize("original", [False, True])
def test_wide_gemm_totals_of_uneven_rows(cq, original):
    """The same for the paired GEMM over 1024 terms, the first eight of 32
    rows 1 and the others just below half the last place of sixteen ones: 32
    outputs of one row are added in float32, in a tree (five roundings)."""
    import torch
    qb = [0, 1, 2] + list(range(12, 21))
    subs, _, _ = _pair(12, 12, 5, [q for q in range(24) if q not in qb] if original else None)
    A, B = _uneven(torch, 12, 12, 5, lambda m: m % 32 < 8, 2.0 ** -20 * (1 - 2.0 ** -6))
    total = torch.zeros(1, dtype=torch.float64, device="cuda")
    out, _ = cq.cutqc_reconstruct_fd(subs, [A, B], cq.ORDER_ORIGINAL if original else cq.ORDER_KRON, cq.PREC_FP16X3_TC,
                                     sum_out=total)
    ref = (A[:, 0].double().sum() * 2.0 ** 12).item()
    assert abs(out.double().sum().item() - ref) <= 1e-12 * ref
    assert abs(total.item() - ref) <= 5 * 2.0 ** -24 * ref


@pytest.mark.parametrize("k", [5, 6])
@pytest.mark.parametrize("sign", ["one", "both"])
def test_many_term_sums(cq, k, sign):
    """Steps of 1024 and 4096 terms, all positive, and of falling size and
    both signs beside one positive column as in an attributed tensor: the
    paired GEMM (many tiles) is on average no further from float64 than the
    single-SM GEMM, which the same rows take as a row range of few tiles."""
    import torch
    rng = np.random.default_rng(k)
    ops = []
    for _ in range(2):
        if sign == "one":
            x = rng.uniform(0.01, 1.0, (1 << 12, 4 ** k))
        else:
            x = rng.standard_normal((1 << 12, 4 ** k))
            x *= 2.0 ** -np.array([sum(((c >> 2 * j) & 3) != 0 for j in range(k)) for c in range(4 ** k)])
            x[:, 0] = 1.0
        ops.append(torch.from_numpy(x.astype(np.float32)).cuda())
    A, B = ops
    subs, _, _ = _pair(12, 12, k)
    whole, _ = cq.cutqc_reconstruct_fd(subs, [A, B], cq.ORDER_KRON, cq.PREC_FP16X3_TC)
    rows, _ = cq.cutqc_reconstruct_fd(subs, [A, B], cq.ORDER_KRON, cq.PREC_FP16X3_TC, 512, 768)
    whole = whole.view(1 << 12, 1 << 12)[512:768]
    rows = rows.view(256, 1 << 12)
    assert not torch.equal(whole, rows)
    ref = A[512:768].double() @ B.double().T * 2.0 ** -k
    err = [(x.double() - ref).abs().sum().item() for x in (whole, rows)]
    assert err[0] <= err[1], err
    assert cq.cutqc_device_status() == 0


@pytest.mark.parametrize("oa,ob,k", [(9, 12, 3), (10, 12, 4), (8, 12, 5), (12, 13, 5), (8, 11, 6)])
def test_dependent_launches_from_poisoned_buffers(cq, oa, ob, k):
    """The tensor-core step's dependent launches where nothing right is left to
    read: before every pass the workspace holds 0xFF bytes (NaNs), the output
    -1 and the inputs another scale, all written right before on the same
    stream; eagerly on two streams at once and from a graph.  Every pass is
    compared on the device, and the eager result once with float64 (the bound
    of the split and the accumulation, 2^-16 of the absolute terms)."""
    import torch
    subs, _, _ = _pair(oa, ob, k)
    need = cq.cutqc_reconstruct_fd_workspace_size(subs, cq.PREC_FP16X3_TC)
    scales = (1.0, 3.0, 0.7)
    sets = []
    for seed in range(2):
        dev, (A, B) = _operands(torch, oa, ob, k, 170 + seed)
        s = dict(src=dev, att=[torch.empty_like(a) for a in dev], out=torch.empty(1 << (oa + ob), device="cuda"),
                 ws=torch.empty(need, dtype=torch.uint8, device="cuda"), bad=torch.zeros((), dtype=torch.int64, device="cuda"),
                 scale=torch.ones((), device="cuda"), stream=torch.cuda.Stream(), ref=[])
        for x in scales:
            att = [a * x for a in dev]
            out, _ = cq.cutqc_reconstruct_fd(subs, att, cq.ORDER_KRON, cq.PREC_FP16X3_TC)
            torch.cuda.synchronize()
            s["ref"].append(out.clone())
        P, terms = A @ B.T * 2.0 ** -k, np.abs(A) @ np.abs(B).T * 2.0 ** -k
        assert (np.abs(s["ref"][0].view(1 << oa, 1 << ob).double().cpu().numpy() - P) <= 2.0 ** -16 * terms).all()
        sets.append(s)

    def one(s):
        s["ws"].fill_(0xFF)
        s["out"].fill_(-1.0)
        for w, a in zip(s["att"], s["src"]):
            torch.mul(a, s["scale"], out=w)
        cq.cutqc_reconstruct_fd(subs, s["att"], cq.ORDER_KRON, cq.PREC_FP16X3_TC, out=s["out"], ws=s["ws"])

    for rep in range(9):
        for s in sets:
            with torch.cuda.stream(s["stream"]):
                s["scale"].fill_(scales[rep % 3])
                one(s)
                s["bad"] += (s["out"] != s["ref"][rep % 3]).sum()
    torch.cuda.synchronize()
    assert [int(s["bad"]) for s in sets] == [0, 0]
    s = sets[0]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s["stream"]):
        one(s)
    for rep in range(6):
        s["scale"].fill_(scales[(rep + 1) % 3])
        g.replay()
        s["bad"] += (s["out"] != s["ref"][(rep + 1) % 3]).sum()
    torch.cuda.synchronize()
    assert int(s["bad"]) == 0
    assert cq.cutqc_device_status() == 0


@pytest.mark.parametrize("oa,ob,k", [(17, 7, 0), (16, 8, 1), (15, 9, 0), (14, 10, 1), (13, 11, 0), (15, 7, 2), (14, 8, 2),
                                     (13, 10, 2), (10, 13, 2)])
def test_outer_products_in_groups_of_rows(cq, oa, ob, k):
    """Outer products whose CTAs take several groups of 32 rows (narrow tiles,
    and tiles of 1024 columns at 16 terms), rows in order and permuted, and
    their block maxima: every output within the float32 chain's (4^k + 2)
    2^-24 of the absolute terms, nothing written around them, the total (8
    outputs in float32, three roundings), and the largest bins of a
    dynamic-definition job of the same step, which come from the maxima."""
    import torch
    n = oa + ob
    g = torch.Generator(device="cuda")
    g.manual_seed(100 * oa + k)
    A = torch.randn((1 << oa, 4 ** k), device="cuda", generator=g)
    B = torch.randn((1 << ob, 4 ** k), device="cuda", generator=g)
    P = A.double() @ B.double().T * 2.0 ** -k
    tol = (4 ** k + 2) * 2.0 ** -24 * (A.double().abs() @ B.double().abs().T) * 2.0 ** -k
    subs, _, _ = _pair(oa, ob, k)
    for perm in (False, True):
        order = np.arange(oa)
        if perm:
            order = np.random.default_rng(oa).permutation(oa)
            subs[0].out_qubit = (ob + order).tolist()
        buf = torch.full(((1 << n) + 8,), 7.0, device="cuda")
        total = torch.zeros(1, dtype=torch.float64, device="cuda")
        out = buf[4:4 + (1 << n)]
        cq.cutqc_reconstruct_fd(subs, [A, B], cq.ORDER_ORIGINAL, cq.PREC_FP32_SIMT, out=out, sum_out=total)
        rows = torch.arange(1 << oa, device="cuda")
        at = sum((((rows >> j) & 1) << int(order[j]) for j in range(oa)), torch.zeros_like(rows))
        assert bool(((out.view(1 << oa, 1 << ob)[at].double() - P).abs() <= tol).all())
        assert bool((buf[:4] == 7.0).all()) and bool((buf[4 + (1 << n):] == 7.0).all())
        assert abs(total.item() - out.double().sum().item()) <= 3 * 2.0 ** -24 * out.double().abs().sum().item()
        jobs, n_jobs, bins = cq.cutqc_dd_run_async(subs, [A, B], n, n, 1, 4)
        torch.cuda.synchronize()
        J = cq.dd_jobs_from_device(jobs, n_jobs)[0]
        bins = bins[:1 << n]
        assert torch.equal(bins, out)
        v, i = torch.topk(bins, 4)
        assert list(J.top_idx[:4]) == i.tolist() and list(J.top_val[:4]) == v.tolist()
    assert cq.cutqc_device_status() == 0
