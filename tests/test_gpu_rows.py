"""The row-vector form of the on-chip kernel (the planner's choice for graphs
with short rows or few starts) against the per-step kernel: the same FP32
operations in the same order, so the blocks are bit-identical.

The planner takes slab widths of 1, 2, 4 or 8 vectors by the number of
columns, and more columns than the GPU holds at once run in several waves; the
tests ask the library which form and width a call takes."""
import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2509_18612_gb300 as deco  # noqa: E402

DEV = torch.device("cuda:0")


def _weighted(g, choices, seed):
    u, v, _ = g.edges()
    return gg.from_edges(g.n, u, v, np.random.default_rng(seed).choice(np.array(choices), size=u.size))


GRAPHS = {
    "one": lambda: gg.from_edges(1, [], []),
    "31": lambda: gg.er_graph(31, 0.3, 1),
    "33": lambda: gg.er_graph(33, 0.9, 2),                       # rows of 24 ... 32 entries: whole chunks of 8
    "er100": lambda: gg.er_graph(100, 0.1, 0),
    "isolated": lambda: gg.from_edges(90, [0, 1, 2, 5], [1, 2, 3, 9]),
    "hubs": lambda: gg.ba_graph(1025, 4, 7),                     # one slice more than 32 warps hold, long rows
    "torus": lambda: gg.torus_graph(40, 20, 3),                  # +-1: both lists, 0 ... 4 entries
    "sign": lambda: _weighted(gg.er_graph(257, 0.05, 3), [-1.0, 1.0], 1),
    "weights": lambda: _weighted(gg.ba_graph(300, 4, 5), [-3.0, 2.0, 7.0], 2),
    "long": lambda: gg.er_graph_avg_degree(2300, 5.0, 4),        # beyond the 128-byte slabs: AUTO only
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
@pytest.mark.parametrize("objective,mu", [(0, 0.0), (0, 0.9), (1, 0.9), (1, 0.0)])
@pytest.mark.parametrize("C", [1, 37, 64, 200, 1024, 3000, 9000])
def test_row_vector_form_bitwise_equals_per_step_kernel(name, precision, objective, mu, C):
    g = GRAPHS[name]()
    if C > 1024 and g.n > 300:
        pytest.skip("the widths are covered by the small graphs")
    G = deco.graph_from(g)
    ld = (C + 63) // 64 * 64
    gen = torch.Generator(device=DEV).manual_seed(C)
    y0 = (torch.rand(g.n, ld, device=DEV, generator=gen) * 2 - 1) * 0.3
    y0 = y0.bfloat16() if precision else y0
    v0 = torch.randn(g.n, ld, device=DEV, generator=gen) * 0.1 if mu else None
    alpha = torch.rand(C, device=DEV, generator=gen) * 0.02
    budget = torch.randint(0, 8, (C,), device=DEV, generator=gen, dtype=torch.int32)
    for cols in (False, True):
        args = deco.step_args(objective, precision, 0.01, mu, alpha_cols=alpha if cols else None,
                              steps_cols=budget if cols else None)
        out = []
        for kernel in (deco.DECO_KERNEL_GLOBAL, deco.DECO_KERNEL_AUTO, deco.DECO_KERNEL_ONCHIP):
            if kernel == deco.DECO_KERNEL_ONCHIP and g.n > 1700:
                continue
            y, v = y0.clone(), None if v0 is None else v0.clone()
            for steps in (0, 3, 4):      # both replicas; state carried from call to call
                deco.deco_run_phase(G, C, ld, y, v, steps, args, kernel=kernel)
            out.append((y, v))
        for y, v in out[1:]:
            assert torch.equal(y, out[0][0])
            assert mu == 0.0 or torch.equal(v, out[0][1])


def test_row_vector_form_flags_nonfinite_and_keeps_limits():
    g = GRAPHS["er100"]()
    G = deco.graph_from(g)
    y = torch.zeros(100, 64, device=DEV)
    y[5, 3] = float("inf")
    flag = torch.zeros(1, dtype=torch.int32, device=DEV)
    deco.deco_run_phase(G, 64, 64, y, None, 1, deco.step_args(), flag=flag)
    assert flag.item() & 1
    # a graph beyond the 128-byte slabs is refused where the on-chip kernel is demanded, as ever
    big = deco.graph_from(GRAPHS["long"]())
    with pytest.raises(deco.DecoError):
        deco.deco_run_phase(big, 64, 64, torch.zeros(2300, 64, device=DEV), None, 1, deco.step_args(),
                            kernel=deco.DECO_KERNEL_ONCHIP)


# Batches: members of unequal sizes in the on-chip form that the planner takes (rows or, for the dense members,
# 128-byte slabs) and the per-step kernels over the union give the same cuts, scores and population.  Candidates
# own between one and several slabs' columns, so CTAs stop at budgets of their own.
@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
@pytest.mark.parametrize("kind", ["ba", "sign", "weights", "dense"])
@pytest.mark.parametrize("objective,mu,B,P", [(0, 0.9, 64, 4), (1, 0.9, 30, 15), (1, 0.0, 200, 2)])
def test_batched_row_vector_form_equals_the_other_forms(precision, kind, objective, mu, B, P):
    rng = np.random.default_rng(5)
    graphs = [gg.ba_graph(int(n), 4, 10 + i) for i, n in enumerate(list(rng.integers(20, 900, 20)) + [33])] + [gg.from_edges(1, [], []), gg.er_graph(40, 0.2, 3)]
    if kind == "sign":
        graphs = [_weighted(g, [-1.0, 1.0], i) if g.n > 1 else g for i, g in enumerate(graphs)]
    elif kind == "weights":
        graphs = [_weighted(g, [-3.0, 2.0, 7.0], i) if g.n > 1 else g for i, g in enumerate(graphs)]
    elif kind == "dense":
        graphs = [gg.er_graph(int(n), 0.3, int(n)) for n in rng.integers(20, 300, 12)]
    batch = deco.deco_create_batch([deco.graph_from(g) for g in graphs])
    pop = deco.population(candidates=P, rounds=3, t_lo=0, t_hi=25, e_lo=-2.5, e_hi=-1.5, momentum=mu, lifts=(1, 2))
    outs = []
    for kernel in (deco.DECO_KERNEL_GLOBAL, deco.DECO_KERNEL_AUTO):
        p = deco.params(objective=objective, init=deco.DECO_INIT_IDI, precision=precision, kernel=kernel)
        for _ in range(2):   # the images are kept with the batch
            _, best, ex = deco.deco_solve_batch(batch, B, p, pop, 9, want_assignment=True, want_round_cuts=True)
            outs.append((best.tolist(), ex["assignment"].tobytes(), ex["round_cuts"].tobytes(),
                         ex["round_scores"].tobytes(), ex["final_T"].tobytes()))
    assert all(o == outs[0] for o in outs)


FORM_COLUMNS = (64, 500, 800, 1024, 1300, 1600, 2000, 2400, 3000, 4000, 5000, 6000, 7000, 9000)


# Every width of the form, for every storage of the weights, with a row's data in registers where the planner takes that
# (not with per-column step sizes), against the per-step kernel.
@pytest.mark.parametrize("name,registers", [("er100", True), ("isolated", True), ("sign", False), ("weights", False)])
@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
@pytest.mark.parametrize("width", [1, 2, 4, 8])
def test_every_width_of_the_row_vector_form_equals_the_per_step_kernel(name, registers, precision, width):
    g = GRAPHS[name]()
    G = deco.graph_from(g)

    def form(C, cols):
        return deco.deco_debug_phase_form(G, C, (C + 63) // 64 * 64, precision, cols)

    taken = [C for C in FORM_COLUMNS if form(C, True) == (deco.DECO_FORM_ROWS, width)]
    if name == "isolated" and width == 8:
        assert not taken   # 90 rows of up to 2 entries: never worth more than 4 vectors at these columns
        return
    C = taken[0]
    if registers:
        assert form(C, False) == (deco.DECO_FORM_ROWS_REG, width)
    else:
        assert form(C, False)[0] in (deco.DECO_FORM_ROWS, deco.DECO_FORM_ROWS_REG)
    ld = (C + 63) // 64 * 64
    y0 = ((torch.rand(g.n, ld, device=DEV) * 2 - 1) * 0.3).to(torch.bfloat16 if precision else torch.float32)
    alpha = torch.rand(C, device=DEV) * 0.02
    budget = torch.randint(0, 8, (C,), device=DEV, dtype=torch.int32)
    for cols in (False, True):
        args = deco.step_args(1, precision, 0.01, 0.9, alpha_cols=alpha if cols else None,
                              steps_cols=budget if cols else None)
        out = []
        for kernel in (deco.DECO_KERNEL_GLOBAL, deco.DECO_KERNEL_AUTO):
            y, v = y0.clone(), torch.zeros(g.n, ld, device=DEV)
            deco.deco_run_phase(G, C, ld, y, v, 7, args, kernel=kernel)
            out.append((y, v))
        assert torch.equal(out[1][0], out[0][0]) and torch.equal(out[1][1], out[0][1])


# The batched forms by name: the planner's row-vector form, and k_slab (demanded by a modifier, which takes a union that
# fits on chip as well) with its staging area or, for members of 620 rows, lean.  Four candidates of 32 columns: slabs
# stop at budgets of their own.
@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
@pytest.mark.parametrize("sizes,slab", [((200, 150, 33, 120), deco.DECO_FORM_SLAB), ((620, 200), deco.DECO_FORM_SLAB_LEAN)])
@pytest.mark.parametrize("mu", [0.0, 0.9])
@pytest.mark.parametrize("weights", [None, [-1.0, 1.0], [-3.0, 2.0, 7.0]])
def test_batched_forms_equal_the_per_step_kernels(precision, sizes, slab, mu, weights):
    graphs = [gg.ba_graph(n, 2, 800 + n) for n in sizes]
    if weights:
        graphs = [_weighted(g, weights, g.n) for g in graphs]
    batch = deco.deco_create_batch([deco.graph_from(g) for g in graphs])
    pairs = deco.DECO_KERNEL_ONCHIP | deco.DECO_KERNEL_ROW_PAIRS
    assert deco.deco_debug_batch_form(batch, 128, 128, precision, kernel=pairs)[0] == slab
    assert deco.deco_debug_batch_form(batch, 128, 128, precision)[0] == deco.DECO_FORM_ROWS
    pop = deco.population(candidates=4, rounds=3, t_lo=1, t_hi=50, e_lo=-2.5, e_hi=-1.5, momentum=mu, lifts=(1, 2))
    outs = []
    for kernel in (deco.DECO_KERNEL_GLOBAL, pairs, deco.DECO_KERNEL_AUTO):
        p = deco.params(objective=deco.DECO_OBJ_LAPLACIAN, init=deco.DECO_INIT_IDI, precision=precision, kernel=kernel)
        _, best, ex = deco.deco_solve_batch(batch, 128, p, pop, 9, want_assignment=True, want_round_cuts=True)
        outs.append((best.tolist(), ex["assignment"].tobytes(), ex["round_cuts"].tobytes(), ex["round_scores"].tobytes()))
    assert outs[1] == outs[0] and outs[2] == outs[0]
