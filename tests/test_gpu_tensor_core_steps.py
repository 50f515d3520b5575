"""Tensor-core contraction steps at sizes past the one-launch kernel of small
steps (2^18 outputs, 2^27 products): dynamic range, chains with open digits,
late inputs, graphs, row ranges, pruned k-blocks, the launch after an expired
wait.  References in float64 on the device; launch counts show that the step
was not the one-launch kernel's."""
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


def _chain(outs, cuts):
    """Subcircuits of a chain, edges numbered along it, uncut qubits in chain
    order from the lowest."""
    subs, q, e, left = [], 0, 0, []
    for i, o in enumerate(outs):
        right = list(range(e, e + cuts[i])) if i < len(cuts) else []
        e += len(right)
        subs.append(types.SimpleNamespace(w=o + len(right), in_local=list(range(len(left))), in_edge=left,
                                          out_local=list(range(o, o + len(right))), out_edge=right,
                                          out_qubit=list(range(q, q + o)), o=o, k=len(left) + len(right)))
        q, left = q + o, right
    return subs


def _pair(oa, ob, k, qa=None):
    """Two subcircuits over k cuts; qa: the uncut qubits of the first's
    outputs (default: the highest)."""
    a, b = _chain([oa, ob], [k])
    a.out_qubit = list(range(ob, ob + oa)) if qa is None else list(qa)
    b.out_qubit = [q for q in range(oa + ob) if q not in a.out_qubit]
    return [a, b]


def _normal(subs, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return [torch.randn((1 << s.o, 4 ** s.k), device="cuda", generator=g) for s in subs]


def _chain64(subs, att):
    """Kronecker order, float64: the chain's tensors joined from the left."""
    x = None
    for s, a in zip(subs, att):
        kl = 4 ** len(s.in_edge)
        a = a.double().view(1 << s.o, -1, kl)          # [rows][right digits][left digits, lowest edges]
        if x is None:
            x = a[:, :, 0]
        else:
            x = (x.view(-1, kl) @ a.permute(2, 0, 1).reshape(kl, -1)).view(-1, a.shape[1])
    return x.view(-1) * 2.0 ** -sum(len(s.out_edge) for s in subs)


def _to_original(p, subs):
    """Kronecker order -> uncut qubit order."""
    import torch
    n = sum(s.o for s in subs)
    idx = torch.zeros(1, dtype=torch.int64, device=p.device)
    for s in subs:
        r = torch.arange(1 << s.o, device=p.device)
        d = sum((((r >> t) & 1) << q for t, q in enumerate(s.out_qubit)), torch.zeros_like(r))
        idx = (idx[:, None] | d[None, :]).view(-1)
    out = torch.empty_like(p)
    out[idx] = p
    assert out.numel() == 1 << n
    return out


def _wide_range(rng, rows, cols, decades):
    a = rng.choice([-1.0, 1.0], size=(rows, cols)) * 10.0 ** rng.uniform(-decades, 0, size=(rows, cols))
    a *= 10.0 ** rng.uniform(-4, 0, size=(rows, 1))
    a[rng.random((rows, cols)) < 0.05] = 0.0
    a[rng.random(rows) < 0.03] = 0.0
    return a.astype(np.float32)


@pytest.mark.parametrize("decades", [8, 10])
@pytest.mark.parametrize("oa,ob,k", [(8, 11, 4), (8, 11, 5), (10, 12, 5), (8, 11, 6), (11, 8, 6)])
def test_split_over_a_wide_dynamic_range(cq, oa, ob, k, decades):
    """Entries over 8 and 10 decades in a row and 4 more across rows, zeros and
    both signs, so that low parts fall into FP16's subnormals: every tensor-core
    GEMM, in the order where the first operand is the row operand (a scale per
    row) and in one where it may be the column operand (it holds output bit 0
    too: one scale in all).  Bound of the split, four times over:
        2^-16 sum_k |a_k b_k| + 2^-37 (|A_m|_1 max|B| + |B_n|_1 max|A|)  (times 2^-K)."""
    import torch
    rng = np.random.default_rng(100 * k + decades)
    att = [torch.from_numpy(_wide_range(rng, 1 << o, 4 ** k, decades)).cuda() for o in (oa, ob)]
    A, B = (a.double() for a in att)
    ref = (A @ B.T).view(-1) * 2.0 ** -k
    under = A.abs().sum(1)[:, None] * B.abs().max() + B.abs().sum(1)[None, :] * A.abs().max()
    bound = (2.0 ** -16 * (A.abs() @ B.abs().T) + 2.0 ** -37 * under).view(-1) * 2.0 ** -k
    for qa in (None, [0, 1, 2] + list(range(ob + 3, ob + oa))):
        subs = _pair(oa, ob, k, qa)
        n0 = cq.cutqc_kernel_launches()
        out, _ = cq.cutqc_reconstruct_fd(subs, att, cq.ORDER_ORIGINAL, cq.PREC_FP16X3_TC)
        assert cq.cutqc_kernel_launches() - n0 >= 3
        err = (out.double() - _to_original(ref, subs)).abs()
        assert bool((err <= _to_original(bound, subs)).all()), qa
        # zero rows of either operand give exact zeros
        zero = (A.abs().sum(1) == 0)[:, None] | (B.abs().sum(1) == 0)[None, :]
        assert not bool(out[_to_original(zero.view(-1), subs)].any())
    assert cq.cutqc_device_status() == 0


@pytest.mark.parametrize("order", [0, 1], ids=["kron", "original"])
@pytest.mark.parametrize("outs,cuts", [((8, 7, 6), (3, 3)), ((8, 8, 5), (3, 4)), ((8, 6, 5), (4, 3)), ((8, 7, 6), (3, 2)),
                                       ((6, 6, 6, 6), (2, 5, 2))])
def test_chains_with_open_digits(cq, outs, cuts, order):
    """Chains whose middle tensors are joined over their high digits first,
    the open ones lowest (transposing preparation, intermediates stored by
    columns of open digits; in the last, 2^22-entry intermediates on two
    streams and a last step of 1024 terms).  Bound: 2^-16 of the absolute
    terms (the split and two accumulations)."""
    import torch
    subs = _chain(outs, cuts)
    if order:
        perm = np.random.default_rng(sum(outs)).permutation(sum(outs))
        for s in subs:
            s.out_qubit = perm[s.out_qubit].tolist()
    att = _normal(subs, 3)
    ref, bound = _chain64(subs, att), _chain64(subs, [a.abs() for a in att])
    if order:
        ref, bound = _to_original(ref, subs), _to_original(bound, subs)
    total = torch.zeros(1, dtype=torch.float64, device="cuda")
    n0 = cq.cutqc_kernel_launches()
    out, _ = cq.cutqc_reconstruct_fd(subs, att, order, cq.PREC_FP16X3_TC, sum_out=total)
    assert cq.cutqc_kernel_launches() - n0 >= 3 * len(cuts)
    assert bool(((out.double() - ref).abs() <= 2.0 ** -16 * bound).all())
    assert abs(total.item() - out.double().sum().item()) <= 2.0 ** -20 * out.double().abs().sum().item()
    assert cq.cutqc_device_status() == 0


@pytest.mark.parametrize("graph", [False, True], ids=["eager", "graph"])
@pytest.mark.parametrize("late", [0, 1, 2, 3])
@pytest.mark.parametrize("precision", [1, 2], ids=["tc", "tc_prune"])
def test_late_inputs_of_tensor_core_steps(cq, precision, late, graph):
    """A reconstruction issued before one of its inputs (each in turn: row and
    column operands of steps on the caller's and on a side stream) is written,
    about a millisecond later on another stream, from NaNs: the bits of the
    reconstruction of the same tensors written beforehand, eagerly and from a
    graph whose inputs and workspace are poisoned before each replay."""
    import torch
    subs = _chain((6, 6, 6, 6), (2, 5, 2))
    src = _normal(subs, 5)
    ref, _ = cq.cutqc_reconstruct_fd(subs, src, 0, precision)
    att = [s.clone() for s in src]
    out = torch.empty_like(ref)
    ws = torch.empty(cq.cutqc_reconstruct_fd_workspace_size(subs, precision), dtype=torch.uint8, device="cuda")
    other = torch.cuda.Stream()

    def step():
        cur = torch.cuda.current_stream()
        other.wait_stream(cur)
        ev = [None] * len(subs)
        with torch.cuda.stream(other):
            torch.cuda._sleep(2_000_000)
            att[late].copy_(src[late])
            ev[late] = torch.cuda.Event()
            ev[late].record(other)
        cq.cutqc_reconstruct_fd(subs, att, 0, precision, out=out, ws=ws, input_events=ev)
        cur.wait_stream(other)

    def poison():
        att[late].fill_(float("nan"))
        out.fill_(float("nan"))
        ws.fill_(0xFF)
        torch.cuda.synchronize()

    if graph:
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=torch.cuda.Stream()):
            step()
    for _ in range(2):
        poison()
        g.replay() if graph else step()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    assert cq.cutqc_device_status() == 0


def test_row_ranges_of_a_tensor_core_step(cq):
    """Row ranges of 256-term steps written separately equal the whole, from a
    single row to ranges that end inside the 256-row tiles."""
    import torch
    subs = _pair(10, 11, 4)
    att = _normal(subs, 7)
    whole, _ = cq.cutqc_reconstruct_fd(subs, att, 0, cq.PREC_FP16X3_TC)
    rows, _ = cq.cutqc_fd_shape(subs)
    parts = []
    for r0, r1 in ((0, 1), (1, 3), (3, 260), (260, 773), (773, rows)):
        n0 = cq.cutqc_kernel_launches()
        parts.append(cq.cutqc_reconstruct_fd(subs, att, 0, cq.PREC_FP16X3_TC, r0, r1)[0])
        assert cq.cutqc_kernel_launches() - n0 >= 3
    assert torch.equal(torch.cat(parts), whole)
    assert cq.cutqc_device_status() == 0


@pytest.mark.parametrize("kept", [1, 40, 130, 300, 700, 1000])
@pytest.mark.parametrize("oa,ob", [(11, 12), (8, 11)])
def test_pruned_k_blocks_of_1024_terms(cq, oa, ob, kept):
    """1024 terms of which all but `kept` are negligible: the GEMMs on SM pairs
    (2^23 outputs) and on single SMs run 1, 3, 5, 11 and 16 k-blocks, a count
    read on the device, odd ones among them.  Bound: the split's and 2^-30."""
    import torch
    rng = np.random.default_rng(kept)
    scale = np.full(1024, 1e-24)
    scale[rng.choice(1024, size=kept, replace=False)] = 1.0
    a = (np.abs(rng.standard_normal((1 << oa, 1024))) / (1 << oa)).astype(np.float32)
    b = (rng.standard_normal((1 << ob, 1024)) / (1 << ob) * scale).astype(np.float32)
    att = [torch.from_numpy(x).cuda() for x in (a, b)]
    A, B = (x.double() for x in att)
    ref = (A @ B.T).view(-1) * 2.0 ** -5
    bound = (A.abs() @ B.abs().T).view(-1) * 2.0 ** -5
    for qa in (None, list(range(3, 3 + oa))):
        subs = _pair(oa, ob, 5, qa)
        full, _ = cq.cutqc_reconstruct_fd(subs, att, cq.ORDER_ORIGINAL, cq.PREC_FP16X3_TC)
        out, _ = cq.cutqc_reconstruct_fd(subs, att, cq.ORDER_ORIGINAL, cq.PREC_FP16X3_TC_PRUNE)
        r, c = _to_original(ref, subs), _to_original(bound, subs)
        assert bool(((full.double() - r).abs() <= 2.0 ** -16 * c).all())
        assert bool(((out.double() - r).abs() <= 2.0 ** -16 * c + cq.PRUNE_TOL).all())
    assert cq.cutqc_device_status() == 0


def test_tensor_core_step_after_an_expired_wait(cq):
    """After a device wait gave up and its status was read, the GEMMs on SM
    pairs and single SMs still run, with the bits of before."""
    import torch
    cases = [(_pair(8, 11, 4), 1), (_pair(10, 12, 5), 2), (_pair(8, 11, 5), 3)]
    att = [_normal(subs, seed) for subs, seed in cases]
    before = [cq.cutqc_reconstruct_fd(subs, a, 0, cq.PREC_FP16X3_TC)[0] for (subs, _), a in zip(cases, att)]
    waited = torch.zeros(1, dtype=torch.int32, device="cuda")
    cq.cutqc_selftest_wait_timeout(waited)
    assert cq.cutqc_device_status() == -4
    for (subs, _), a, ref in zip(cases, att, before):
        assert torch.equal(cq.cutqc_reconstruct_fd(subs, a, 0, cq.PREC_FP16X3_TC)[0], ref)
    assert cq.cutqc_device_status() == 0
