"""Degenerate and boundary cases of the solver through the C ABI, against the
oracle: a single node, an edgeless graph, one starting point, phases of zero
steps, a lift of three (Eq. 11 summed in order), complete graphs (closed-form
optimum), a graph near the shared-memory limit of the on-chip kernel, and the
bounded device waits giving up (failure detection without a GPU fault)."""
import numpy as np
import pytest

import graphgen as gg
from oracle import deco_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2509_18612_gb300 as deco  # noqa: E402

DEV = torch.device("cuda:0")


def _agree(a, b):
    return float(np.mean(np.asarray(a) == np.asarray(b)))


@pytest.mark.parametrize("n", [1, 2, 50])
def test_edgeless_graphs_cut_zero(n):
    g = gg.from_edges(n, [], [])
    for kern in (deco.DECO_KERNEL_GLOBAL, deco.DECO_KERNEL_AUTO):
        res, z, pc = deco.deco_solve(deco.graph_from(g), 8, [(1, 20, 0.01, 0.9), (2, 5, 0.001, 0.9)],
                                     deco.params(init=deco.DECO_INIT_IDI, kernel=kern), 3)
        assert res.best_cut == 0 and (pc == 0).all() and z.shape == (n,)


def test_one_starting_point_and_zero_step_phases():
    g = gg.er_graph(100, 0.1, 0)
    G = deco.graph_from(g)
    x0 = gg.uniform_x0(g.n, 1, 4)
    sched = [(1, 0, 0.01, 0.0), (1, 50, 0.01, 0.0), (2, 0, 0.001, 0.0)]
    res, z, pc = deco.deco_solve(G, 1, sched, deco.params(init=deco.DECO_INIT_EXPLICIT), 2, x0=x0)
    ref = O.solve(g, 1, [O.Phase(*s) for s in sched], O.Params(init="explicit"), 2, x0=x0)
    np.testing.assert_array_equal(pc, np.array(ref.phase_cuts))
    assert res.best_cut == ref.best_cut == O.cut_value(g, z)
    assert res.edge_updates == g.nnz * 50


@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
def test_lift_three_rounding_order(precision):
    # l = 3: the row sum is accumulated in the order i = 0, 1, 2 on both sides
    g = gg.er_graph(200, 0.05, 7)
    B, l = 40, 3
    rng = np.random.default_rng(3)
    Y = rng.uniform(-1, 1, size=(g.n, B * l)).astype(np.float32)
    dt = torch.bfloat16 if precision == deco.DECO_PREC_BF16 else torch.float32
    y = torch.from_numpy(Y).to(DEV).to(dt)
    zbits = torch.zeros(g.n * 2, dtype=torch.int32, device=DEV)
    cuts = torch.zeros(B, dtype=torch.int64, device=DEV)
    deco.deco_round_cut(deco.graph_from(g), B, l, B * l, precision, y, zbits, cuts)
    torch.cuda.synchronize()
    Yq = y.float().cpu().numpy()
    # the device sums in FP32 in order; the FP64 oracle's sum decides every row
    # whose FP32 and FP64 sums have the same sign (all but exact-zero ties)
    s32 = (Yq[:, 0::3] + Yq[:, 1::3]) + Yq[:, 2::3]
    ref = O.cut_values(g, (s32 >= 0).astype(np.uint8))
    np.testing.assert_array_equal(cuts.cpu().numpy(), ref)
    assert _agree(ref, O.cut_values(g, O.binarize(Yq, l))) >= 0.99


@pytest.mark.parametrize("n", [6, 9, 14])
def test_complete_graph_reaches_the_closed_form(n):
    u, v = np.triu_indices(n, 1)
    g = gg.from_edges(n, u, v)
    res, z, _ = deco.deco_solve(deco.graph_from(g), 64, [(1, 300, 0.01, 0.9), (2, 100, 0.002, 0.9)],
                                deco.params(init=deco.DECO_INIT_IDI_HALF_UNIFORM), 1)
    assert res.best_cut == (n // 2) * ((n + 1) // 2) == O.cut_value(g, z)


@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
def test_graph_near_the_shared_memory_limit_on_chip_equals_global(precision):
    # n = 1200 with a cluster of 8: the 150 KB replica of the column slab plus
    # the staging, momentum and CSR image of 150 own rows fill ~215 KB of the
    # ~226 KB of shared memory a CTA may use
    g = gg.er_graph(1200, 0.006, 9)
    G = deco.graph_from(g)
    cols = 64 if precision == deco.DECO_PREC_BF16 else 32
    C, ld = 2 * cols - 3, 2 * cols
    rng = np.random.default_rng(1)
    Y = np.zeros((g.n, ld), np.float32)
    Y[:, :C] = rng.uniform(-1e-3, 1e-3, size=(g.n, C))
    dt = torch.bfloat16 if precision == deco.DECO_PREC_BF16 else torch.float32
    outs = []
    for kern in (deco.DECO_KERNEL_GLOBAL, deco.DECO_KERNEL_ONCHIP | (8 << 8)):
        y = torch.from_numpy(Y).to(DEV).to(dt)
        v = torch.zeros(g.n, ld, device=DEV)
        a = deco.step_args(deco.DECO_OBJ_MULTILINEAR01, precision, 0.01, 0.9)
        deco.deco_run_phase(G, C, ld, y, v, 12, a, kern)
        torch.cuda.synchronize()
        outs.append((y, v))
    assert torch.equal(outs[0][0][:, :C], outs[1][0][:, :C]) and torch.equal(outs[0][1][:, :C], outs[1][1][:, :C])


@pytest.mark.parametrize("which", [0, 1, 2])
def test_bounded_wait_gives_up_and_the_context_stays_usable(which):
    """Failure detection without a GPU fault: one of the kernels' own bounded
    waits (dense mbarrier wait, dense grid barrier, on-chip exchange wait)
    runs on something nothing ever completes.  It must give up after its 2 s
    limit, report DECO_ERR_TIMEOUT through the error flag, and leave the
    context usable: a solve right after it matches the oracle."""
    status, ms = deco.deco_probe_wait_timeout(which)
    assert status == deco.DECO_ERR_TIMEOUT, deco.last_error()
    # the dense waits give up on the 2 s clock; the on-chip exchange wait on
    # the clock or on its iteration cap, whichever comes first
    assert (1900.0 if which < 2 else 1.0) <= ms <= 6000.0, ms
    assert "gave up" in deco.last_error()
    g = gg.er_graph(100, 0.1, 0)
    x0 = gg.uniform_x0(g.n, 16, 0)
    res, z, pc = deco.deco_solve(deco.graph_from(g), 16, [(1, 50, 0.01, 0.0)],
                                 deco.params(init=deco.DECO_INIT_EXPLICIT), 0, x0=x0)
    ref = O.solve(g, 16, [O.Phase(1, 50, 0.01, 0.0)], O.Params(init="explicit"), 0, x0=x0)
    assert res.best_cut == O.cut_value(g, z)
    assert _agree(pc[0], ref.phase_cuts[0]) >= 0.99


def test_injected_scratch_allocation_failures_leave_the_library_usable():
    """Host-side fault injection: the k-th scratch allocation of a solve fails
    with DECO_ERR_OOM (k = 1, 2, ... until the solve needs fewer); each failed
    call releases what it took, and the next call, on the same graph handle,
    gives the same result as before the failures."""
    g = gg.er_graph(100, 0.1, 0)
    G = deco.graph_from(g)
    x0 = gg.uniform_x0(g.n, 16, 1)
    sched = [(1, 30, 0.01, 0.9), (2, 10, 0.001, 0.9)]
    p = deco.params(init=deco.DECO_INIT_EXPLICIT)
    base, zb, pcb = deco.deco_solve(G, 16, sched, p, 0, x0=x0)
    failed = 0
    try:
        for k in range(1, 64):
            deco.deco_debug_fail_scratch_alloc(k)
            try:
                res, z, pc = deco.deco_solve(G, 16, sched, p, 0, x0=x0)
            except deco.DecoError as e:
                assert e.status == deco.DECO_ERR_OOM and "injected" in str(e), str(e)
                failed += 1
                deco.deco_debug_fail_scratch_alloc(0)
                res, z, pc = deco.deco_solve(G, 16, sched, p, 0, x0=x0)
                assert res.best_cut == base.best_cut and (pc == pcb).all() and (z == zb).all()
            else:
                assert res.best_cut == base.best_cut and (pc == pcb).all()
                break
    finally:
        deco.deco_debug_fail_scratch_alloc(0)
    assert failed >= 10, failed


@pytest.mark.parametrize("where", ["first", "middle", "last", "none"])
@pytest.mark.parametrize("family", ["er", "ba"])
def test_large_graph_symmetry_check_on_the_device(where, family):
    # graphs of unit weights with nnz >= 2^20 are checked for symmetry on the
    # device: a removed mirror entry is reported at the lowest offending row,
    # as the host check reports it on small graphs; a symmetric graph passes.
    # The BA graph's first rows are hubs of hundreds of entries (several
    # passes of a warp's lanes).
    g = gg.er_graph_avg_degree(120_000, 10, 6) if family == "er" else gg.ba_graph(140_000, 4, 6)
    rp, ci = g.row_ptr.astype(np.int32), g.col_idx.astype(np.int32)
    assert ci.size >= 1 << 20
    if where != "none":
        v = {"first": 0, "middle": g.n // 2, "last": g.n - 1}[where]
        while rp[v + 1] == rp[v]:
            v += 1
        e = rp[v + 1] - 1                              # drop the last entry (v, u) of row v
        u = int(ci[e])
        ci = np.delete(ci, e)
        rp = rp.copy()
        rp[v + 1:] -= 1
        # (u, v) is now the one entry without a mirror: row u is the offending row
        with pytest.raises(deco.DecoError) as ei:
            deco.deco_create_graph(g.n, rp, ci, None)
        assert ei.value.status == deco.DECO_ERR_GRAPH
        assert f"({u},{v}) stored but ({v},{u}) missing" in deco.last_error(), deco.last_error()
    else:
        G = deco.deco_create_graph(g.n, rp, ci, None)
        G.close()


def test_smem_probe_rate_is_plausible():
    # the shared-memory load path of all SMs: below the 152 SMs x 128 B/clk
    # x 2.07 GHz the hardware can deliver at most (plus a margin for the
    # clock), and well above a tenth of it
    derived = 152 * 128 * 2.07e9 / 1e9
    for width in (8, 16):
        gbs = deco.deco_probe_smem_rate(width, 1 << 14)
        assert 0.1 * derived < gbs < 1.1 * derived, (width, gbs)


CUT_GRAPHS = {
    "star": lambda rng: gg.from_edges(700, np.zeros(699, int), np.arange(1, 700)),      # one hub row, 699 short rows
    "gaps": lambda rng: gg.from_edges(500, [3, 400, 401], [499, 401, 499]),             # windows of empty rows
    "er": lambda rng: gg.er_graph(333, 0.03, 5),
    "signed": lambda rng: _weighted(gg.er_graph(257, 0.05, 6), rng.choice([-1.0, 1.0], 100000)),
    "large weights": lambda rng: _weighted(gg.ba_graph(150, 4, 7), rng.choice([-2.0 ** 20, 2.0 ** 20, 3.0, -77.0], 100000)),
}


def _weighted(g, w):
    u, v, _ = g.edges()
    if np.abs(w).max() > 1000:     # a row's |w| may sum to 2^24 at most
        deg = np.diff(g.row_ptr)
        w = np.where(np.maximum(deg[u], deg[v]) < 16, w[:u.size], 5.0)
    return gg.from_edges(g.n, u, v, w[:u.size])


@pytest.mark.parametrize("B", [1, 31, 32, 33, 64, 96, 128, 130])
@pytest.mark.parametrize("name", list(CUT_GRAPHS))
def test_cut_sums_over_entry_ranges_are_exact(name, B):
    # word vectors of 1, 2 and 4, ragged last words, hub rows, empty windows, every bit of the weights; the same
    # vectors as bytes, and from a word buffer that is only 4-byte aligned
    rng = np.random.default_rng(B)
    g = CUT_GRAPHS[name](rng)
    G = deco.graph_from(g)
    W = (B + 31) // 32
    Y = rng.uniform(-1, 1, size=(g.n, (B + 7) // 8 * 8)).astype(np.float32)
    Z = (Y[:, :B] > 0).astype(np.uint8)
    ref = O.cut_values(g, Z)
    cuts = torch.zeros(B, dtype=torch.int64, device=DEV)
    buf = torch.full((g.n * W + 1,), -1, dtype=torch.int32, device=DEV)
    for off in (0, 1):
        zbits = buf[off:off + g.n * W]
        deco.deco_round_cut(G, B, 1, Y.shape[1], deco.DECO_PREC_FP32, torch.from_numpy(Y).to(DEV), zbits, cuts)
        np.testing.assert_array_equal(cuts.cpu().numpy(), ref)
    words = zbits.cpu().numpy().view(np.uint32).reshape(g.n, W)
    bits = ((words[:, :, None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(g.n, 32 * W)
    np.testing.assert_array_equal(bits[:, :B], Z)
    assert not bits[:, B:].any()
    deco.deco_eval_cuts(G, B, torch.from_numpy(Z * np.uint8(3)).to(DEV), cuts)   # any nonzero byte is 1
    np.testing.assert_array_equal(cuts.cpu().numpy(), ref)


@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
@pytest.mark.parametrize("lift", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("pad", [0, 3, 8])
def test_rounding_by_vectors_equals_rounding_by_columns(lift, pad, precision):
    # rows whose length is a multiple of 8 are read as vectors, others column by column; what lies past the last
    # column (here: 7) must not count
    n, B = 70, 37
    C = B * lift
    ld = (C + 7) // 8 * 8 + pad
    y = torch.full((n, ld), 7.0, device=DEV, dtype=torch.bfloat16 if precision else torch.float32)
    y[:, :C] = (torch.randint(-2, 3, (n, C), device=DEV, generator=torch.Generator(device=DEV).manual_seed(lift)) / 2).to(y.dtype)
    zbits = torch.zeros(n * 2, dtype=torch.int32, device=DEV)
    cuts = torch.zeros(B, dtype=torch.int64, device=DEV)
    deco.deco_round_cut(deco.graph_from(gg.er_graph(n, 0.1, 3)), B, lift, ld, precision, y, zbits, cuts)
    s = y[:, :C].float().cpu().numpy().reshape(n, B, lift).sum(2)     # halves: exact in any order
    Z = s > 0 if lift == 1 else s >= 0
    words = zbits.cpu().numpy().view(np.uint32).reshape(n, 2)
    bits = ((words[:, :, None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(n, 64)
    np.testing.assert_array_equal(bits[:, :B], Z.astype(np.uint32))
    assert not bits[:, B:].any()


def test_scratch_pool_takes_back_what_calls_used_on_two_streams():
    G = deco.graph_from(gg.er_graph_avg_degree(3000, 6.0, 1))
    C = 64
    y0 = torch.rand(3000, C, device="cuda")
    blocks = [y0.clone(), y0.clone(), y0.clone()]
    args = deco.step_args(0, 0, 0.01, 0.0)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    before, _ = deco.deco_debug_pool_usage(reset=True)
    for _ in range(3):
        for y, st in zip(blocks, streams):   # both calls' scratch in flight at once
            deco.deco_run_phase(G, C, C, y, None, 9, args, deco.DECO_KERNEL_GLOBAL, stream=st.cuda_stream)
    torch.cuda.synchronize()
    now, high = deco.deco_debug_pool_usage()
    assert now == before and high >= before + 3000 * C * 4
    for _ in range(3):
        deco.deco_run_phase(G, C, C, blocks[2], None, 9, args, deco.DECO_KERNEL_GLOBAL)
    assert torch.equal(blocks[0], blocks[2]) and torch.equal(blocks[1], blocks[2])


# Steps small enough to start while the step before still runs, against single steps with the stream drained between
# them; a second program on another stream at the same time.
@pytest.mark.parametrize("n,degree,C,weights", [(1, 0.0, 8, None), (5000, 3.0, 8, None), (9001, 11.0, 37, "sign"),
                                                (20011, 6.0, 130, "weights")])
@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
@pytest.mark.parametrize("mu", [0.0, 0.9])
def test_overlapping_steps_equal_single_steps(n, degree, C, weights, precision, mu):
    g = gg.er_graph_avg_degree(n, degree, 3) if n > 1 else gg.from_edges(1, [], [])
    if weights:
        u, v, _ = g.edges()
        choices = [-1.0, 1.0] if weights == "sign" else [-3.0, 2.0, 7.0]
        g = gg.from_edges(g.n, u, v, np.random.default_rng(1).choice(np.array(choices), size=u.size))
    G = deco.graph_from(g)
    ld = (C + 63) // 64 * 64
    dtype = torch.bfloat16 if precision else torch.float32
    y0 = ((torch.rand(n, ld, device=DEV) * 2 - 1) * 0.3).to(dtype)
    args = deco.step_args(0, precision, 0.004, mu)
    T = 41
    a, b = y0.clone(), y0.clone()
    v = torch.zeros(n, ld, device=DEV)
    for _ in range(T):
        deco.deco_step(G, C, ld, a, b, v if mu else None, args)
        torch.cuda.synchronize()
        a, b = b, a
    other = torch.cuda.Stream()
    y, w = y0.clone(), torch.zeros(n, ld, device=DEV)
    y2, w2 = y0.clone(), torch.zeros(n, ld, device=DEV)
    torch.cuda.synchronize()
    deco.deco_run_phase(G, C, ld, y, w if mu else None, T, args, deco.DECO_KERNEL_GLOBAL)
    deco.deco_run_phase(G, C, ld, y2, w2 if mu else None, T, args, deco.DECO_KERNEL_GLOBAL, stream=other.cuda_stream)
    torch.cuda.synchronize()
    assert torch.equal(y[:, :C], a[:, :C]) and torch.equal(y2[:, :C], a[:, :C])
    if mu:
        assert torch.equal(w[:, :C], v[:, :C]) and torch.equal(w2[:, :C], v[:, :C])


# Cuts by bit planes: entry ranges that empty a lane's planes often, once or never; hub rows and ragged words.
@pytest.mark.parametrize("name", ["dense", "hub", "sparse"])
@pytest.mark.parametrize("B", [1, 33, 64, 97, 128, 200])
def test_cuts_by_bit_planes_match_oracle(name, B):
    if name == "dense":
        g = gg.er_graph(900, 0.9, 2)
    elif name == "hub":
        u = np.arange(1, 4001)
        g = gg.from_edges(4001, np.zeros(4000, np.int64), u)
    else:
        g = gg.er_graph_avg_degree(70001, 9.0, 4)
    Z = (np.random.default_rng(B).random((g.n, B)) < 0.5).astype(np.uint8)
    Z[:, 0] = 0
    if B > 1:
        Z[:, 1] = (np.arange(g.n) > 0)   # every entry of the hub is cut
    cuts = torch.zeros(B, dtype=torch.int64, device=DEV)
    deco.deco_eval_cuts(deco.graph_from(g), B, torch.from_numpy(Z.reshape(-1)).to(DEV), cuts)
    np.testing.assert_array_equal(cuts.cpu().numpy(), O.cut_values(g, Z))


# Cuts of byte vectors read where they are (few vectors, small graphs) and packed first; without scratch memory, and
# captured, they are read where they are whatever their number.
@pytest.mark.parametrize("name", list(CUT_GRAPHS) + ["edgeless", "many entries"])
@pytest.mark.parametrize("B", [1, 2, 3, 16, 17, 31, 32, 33, 75])
@pytest.mark.parametrize("how", ["plain", "no scratch", "captured"])
def test_cuts_of_byte_vectors_match_oracle(name, B, how):
    rng = np.random.default_rng(B)
    g = (gg.from_edges(40, [], []) if name == "edgeless" else gg.er_graph(2500, 0.08, 3) if name == "many entries"
         else CUT_GRAPHS[name](rng))
    G = deco.graph_from(g)
    Z = (rng.random((g.n, B)) < 0.5).astype(np.uint8)
    z = torch.from_numpy((Z * rng.integers(1, 256, Z.shape)).astype(np.uint8).reshape(-1)).to(DEV)   # nonzero is 1
    cuts = torch.full((B,), -1, dtype=torch.int64, device=DEV)
    if how == "captured":
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            deco.deco_eval_cuts(G, B, z, cuts, stream=torch.cuda.current_stream().cuda_stream)
        graph.replay()
    else:
        deco.deco_debug_fail_scratch_alloc(1 if how == "no scratch" else 0)
        try:
            deco.deco_eval_cuts(G, B, z, cuts)
        finally:
            deco.deco_debug_fail_scratch_alloc(0)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(cuts.cpu().numpy(), O.cut_values(g, Z))


# Steps of narrow blocks and long rows, whose launches overlap or not and come in blocks of 64, 128 and 256 threads,
# against single steps.
@pytest.mark.parametrize("n,degree,C", [(700, 90.0, 3), (700, 90.0, 9), (700, 90.0, 40), (1900, 200.0, 256), (3001, 40.0, 4),
                                        (12001, 20.0, 5), (40009, 18.0, 11)])
@pytest.mark.parametrize("weights", [None, "sign", "weights"])
@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
@pytest.mark.parametrize("mu", [0.0, 0.9])
def test_steps_of_long_rows_and_narrow_blocks_equal_single_steps(n, degree, C, weights, precision, mu):
    g = gg.er_graph(n, degree / n, 3) if degree >= 90 else gg.er_graph_avg_degree(n, degree, 3)
    if weights:
        u, v, _ = g.edges()
        choices = [-1.0, 1.0] if weights == "sign" else [-3.0, 2.0, 7.0]
        g = gg.from_edges(g.n, u, v, np.random.default_rng(1).choice(np.array(choices), size=u.size))
    G = deco.graph_from(g)
    ld = (C + 7) // 8 * 8
    y0 = ((torch.rand(n, ld, device=DEV) * 2 - 1) * 0.3).to(torch.bfloat16 if precision else torch.float32)
    args = deco.step_args(1, precision, 0.0004, mu)
    a, b, v = y0.clone(), y0.clone(), torch.zeros(n, ld, device=DEV)
    for _ in range(9):
        deco.deco_step(G, C, ld, a, b, v if mu else None, args)
        torch.cuda.synchronize()
        a, b = b, a
    y, w = y0.clone(), torch.zeros(n, ld, device=DEV)
    deco.deco_run_phase(G, C, ld, y, w if mu else None, 9, args, deco.DECO_KERNEL_GLOBAL)
    assert torch.equal(y[:, :C], a[:, :C]) and torch.equal(y[:, C:], y0[:, C:])
    assert mu == 0.0 or torch.equal(w, v)
