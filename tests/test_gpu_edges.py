"""Sizes where a kernel variant or a dispatch rule changes, against the oracle."""
import numpy as np
import pytest

import workloads as WL
import paper_2510_09103_b200 as A

from harness import ParityRun

pytestmark = pytest.mark.gpu


def _blocks(specs):
    out, cur = [], 0
    for rows, cols, mode, rank, vmode, gr in specs:
        cur = -(-cur // 8) * 8
        out.append(A.adapm_block(cur, rows, cols, mode, rank, vmode, gr, 0.75 if mode == A.MOM_NONE else 1.0, 0.1))
        cur += rows * cols
    return out


def _follow(specs, dtype="bf16", steps=4, path=A.PATH_AUTO, **hp):
    run = ParityRun(WL.Workload("edges", [], dtype, "normal", steps=steps), True, lowrank_path=path,
                    hp_overrides=hp, custom_blocks=_blocks(specs))
    try:
        for _ in range(steps):
            run.step()
            run.compare()
        assert run.ctx.adapm_get_status() == 0
    finally:
        run.close()


@pytest.mark.parametrize("rank", [128, 129, 176, 192, 208, 209, 256])
def test_ranks_at_the_edges_of_the_apply_kernels_forms(rank):
    _follow([(264, 328, A.MOM_LOWRANK, rank, A.V_BLOCKMEAN, 1), (300, 264, A.MOM_LOWRANK, rank, A.V_ELEMENT, 0)],
            path=A.PATH_TENSOR)


@pytest.mark.parametrize("rank", [1, 7, 16, 97, 112, 128, 130])
@pytest.mark.parametrize("iters", [2, 3, 5])
def test_refit_on_the_tensor_path_by_rank_and_number_of_passes(iters, rank):
    """The fp32 factors between two passes are kept in the order of the epilogue's threads, the first pass reads and the
    last one writes the state: by rows, by columns and turned, panels and ranks with remainders, one pass to four."""
    _follow([(130, 1032, A.MOM_LOWRANK, rank, A.V_BLOCKMEAN, 1), (648, 264, A.MOM_LOWRANK, rank, A.V_BLOCKMEAN, 8),
             (256, 384, A.MOM_LOWRANK, max(1, rank // 8 * 8), A.V_ELEMENT, 0)], path=A.PATH_TENSOR, inner_iters=iters)


@pytest.mark.parametrize("panels,stage_k", [(0, 0), (1, 64), (2, 128), (3, 64)])
@pytest.mark.parametrize("rank", [5, 33, 80, 128, 144, 256])
def test_panels_at_the_edges_of_a_pair_of_ctas(rank, panels, stage_k):
    """A pair has up to six panels of 128 rows or columns, three for each CTA: sides where the second CTA has none, one row of
    one, or fewer panels than the first; ranks that a CTA's half of the factor's columns fills partly, whole and with a second MMA."""
    _follow([(n, m, A.MOM_LOWRANK, min(rank, n, m), A.V_BLOCKMEAN, 1)
             for n, m in [(100, 264), (128, 129 * 8), (257, 384), (385, 520), (640, 776)]], path=A.PATH_TENSOR, steps=3,
            tune_panels=panels, tune_stage_k=stage_k)


@pytest.mark.parametrize("rank", [12, 80, 144])
def test_a_step_repeats_bit_for_bit_beside_other_work(rank):
    """The order between the two CTAs of a pair (stages filled by one and multiplied by the other, tensor memory read by one
    and overwritten by the other, row sums of the second CTA) does not depend on timing: the same step again and again, while
    copies on another stream come and go."""
    import torch
    blocks = _blocks([(n, m, A.MOM_LOWRANK, rank, A.V_BLOCKMEAN, 1) for n, m in [(640, 776), (1000, 520), (384, 2048), (2050, 264)]])
    total = blocks[-1].offset + blocks[-1].rows * blocks[-1].cols
    ctx = A.adapm_create(blocks, A.hparams(grad_dtype=A.GRAD_BF16, lowrank_path=A.PATH_TENSOR))
    gen = torch.Generator(device="cuda").manual_seed(rank)
    params0 = torch.randn(total, generator=gen, device="cuda")
    grads = torch.randn(total, generator=gen, device="cuda").mul_(1e-3).bfloat16()
    state = torch.zeros(ctx.adapm_state_bytes() // 4, device="cuda")
    work = torch.zeros(ctx.adapm_workspace_bytes() // 4, device="cuda")
    ctx.adapm_set_workspace(work)
    ctx.adapm_state_init(state)
    ctx.adapm_step(params0, grads, state, 1)
    state0, params = state.clone(), params0.clone()
    noise, side = torch.zeros(1 << 24, device="cuda"), torch.cuda.Stream()
    first = None
    for i in range(24):
        params.copy_(params0)
        state.copy_(state0)
        ctx.adapm_state_changed()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            for _ in range(i % 4):
                noise.add_(1.0)
        ctx.adapm_step(params, grads, state, 2)
        torch.cuda.synchronize()
        if first is None:
            first = params.clone(), state.clone()
        assert torch.equal(first[0], params) and torch.equal(first[1], state), f"repeat {i}"
    assert ctx.adapm_get_status() == 0
    ctx.adapm_destroy()


def test_a_cta_that_gives_up_takes_the_other_one_of_its_pair_along():
    """One CTA's wait runs out after a millisecond; the other one, in a wait of its own of more than a second (2^22 polls of at
    least 256 ns), leaves with it."""
    import time
    ctx = A.adapm_create(_blocks([(256, 256, A.MOM_LOWRANK, 12, A.V_BLOCKMEAN, 1)]), A.hparams(grad_dtype=A.GRAD_BF16))
    took = []
    for _ in range(3):                  # (the first one also loads the kernel)
        t0 = time.perf_counter()
        ctx.adapm_selftest_expired_wait()
        assert ctx.adapm_get_status() == A.ST_WAIT_TEAM
        took.append(time.perf_counter() - t0)
    assert min(took) < 0.5, took
    ctx.adapm_destroy()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("rank", [1, 8, 9, 24, 40, 41, 81, 300])
def test_exact_fp32_refit_at_the_edges_of_its_tiles(rank, dtype):
    """Column tiles of every width, one to eight of them, K loops that are cut and that are not, aligned and
    unaligned rows."""
    big = rank > 64
    _follow([(130, 1030 if not big else 330, A.MOM_LOWRANK, min(rank, 130), A.V_BLOCKMEAN, 1),
             (400, 517 if not big else 380, A.MOM_LOWRANK, rank, A.V_ELEMENT, 0),
             (304, 304, A.MOM_LOWRANK, rank, A.V_BLOCKMEAN, 0)], dtype=dtype, path=A.PATH_SIMT)


@pytest.mark.parametrize("rank", [3, 12, 38])
def test_exact_fp32_refit_at_the_ends_of_its_stages(rank):
    """K of less than the stages in flight, of whole stages and one more; rows and columns that are not a multiple of four, or
    of eight."""
    _follow([(m, n, A.MOM_LOWRANK, min(rank, m, n), A.V_BLOCKMEAN, 1)
             for m, n in [(5, 4), (16, 17), (33, 31), (47, 48), (49, 132), (129, 130), (136, 64)]], dtype="f32",
            path=A.PATH_SIMT)


@pytest.mark.parametrize("iters,period", [(1, 0), (2, 0), (3, 0), (2, 3), (3, 3), (5, 3)])
def test_exact_fp32_refit_by_number_of_passes(iters, period):
    """K = 1 has no effective pass, K = 2 a single one that ends in the workspace, K = 3 two."""
    _follow([(150, 77, A.MOM_LOWRANK, 12, A.V_BLOCKMEAN, 1), (64, 264, A.MOM_LOWRANK, 5, A.V_BLOCKMEAN, 0)], dtype="f32",
            steps=5, inner_iters=iters, refresh_period=period)


@pytest.mark.parametrize("vmode", [A.V_BLOCKMEAN, A.V_ELEMENT])
@pytest.mark.parametrize("cols,rank", [(257, 12), (2049, 20), (1366, 128), (333, 160), (513, 209)])
def test_bf16_gradients_whose_rows_do_not_start_on_16_bytes(cols, rank, vmode):
    """The refit reads a padded copy, the apply kernel the gradient itself; beside an aligned block, with clipping and the
    bf16 copy of the parameters."""
    import torch
    blocks = _blocks([(300, cols, A.MOM_LOWRANK, rank, vmode, 0 if vmode == A.V_ELEMENT else 1),
                      (264, 264, A.MOM_LOWRANK, 16, vmode, 0 if vmode == A.V_ELEMENT else 8)])
    run = ParityRun(WL.Workload("odd_rows", [], "bf16", "normal", steps=4), True, custom_blocks=blocks, shadow=True,
                    hp_overrides=dict(max_grad_norm=0.5))
    try:
        for _ in range(4):
            run.step()
            run.compare()
            for blk in run.blocks:
                sl = slice(blk.offset, blk.offset + blk.rows * blk.cols)
                assert torch.equal(run.shadow[sl], run.params[sl].to(torch.bfloat16))
        assert run.ctx.adapm_get_status() == 0
    finally:
        run.close()


@pytest.mark.parametrize("dtype,period", [("bf16", 0), ("bf16", 3), ("f32", 0)])
def test_group_sums_left_by_the_norm_pass(dtype, period):
    """Clipped steps: rows of less than a warp unit of 2048, of exactly one, of one and a piece, groups of several rows, the
    whole block as one group, more and fewer units than a CTA takes, and a row length that the pass leaves to others."""
    _follow([(33, 2040, A.MOM_LOWRANK, 5, A.V_BLOCKMEAN, 1), (16, 2048, A.MOM_LOWRANK, 6, A.V_BLOCKMEAN, 1),
             (18, 2056, A.MOM_LOWRANK, 7, A.V_BLOCKMEAN, 3), (200, 136, A.MOM_LOWRANK, 8, A.V_BLOCKMEAN, 0),
             (30, 77, A.MOM_LOWRANK, 4, A.V_BLOCKMEAN, 1), (64, 80, A.MOM_LOWRANK, 4, A.V_ELEMENT, 0),
             (5, 264, A.MOM_FULL, 0, A.V_BLOCKMEAN, 1)], dtype=dtype, steps=5, max_grad_norm=0.2, refresh_period=period)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_streaming_update_at_the_edges_of_its_teams(dtype):
    """Groups that one, two, four and eight warps hold, and one element more and less."""
    sizes = [2047, 2048, 2049, 4096, 4097, 4104, 8192, 8200, 16384, 16385]
    _follow([(5 if n % 2 else 6, n, A.MOM_FULL if i % 3 else A.MOM_NONE, 0, A.V_BLOCKMEAN, 1)
             for i, n in enumerate(sizes)], dtype=dtype)


# rows x cols of a block whose parameters move by TMA, of one whose rows start at any element, and the CUDA-core path
UPDATE_FORMS = [(200, 264, A.PATH_TENSOR), (200, 267, A.PATH_AUTO), (200, 267, A.PATH_SIMT)]


def _one_block(rows, cols, path, vmode=A.V_ELEMENT, **hp):
    """A low-rank block with frozen factors and a step that writes -lr * ratio over W = 0."""
    import torch
    blocks = [A.adapm_block(0, rows, cols, A.MOM_LOWRANK, 3, vmode, 0 if vmode == A.V_ELEMENT else 1, 1.0, 0.0)]
    ctx = A.adapm_create(blocks, A.hparams(lr=1.0, grad_dtype=A.GRAD_BF16, inner_iters=0, lowrank_path=path, **hp))
    state = torch.zeros(ctx.adapm_state_bytes() // 4, device="cuda")
    work = torch.zeros(max(ctx.adapm_workspace_bytes() // 4, 1), device="cuda")
    ctx.adapm_set_workspace(work)

    def view(which):
        at, n = ctx.adapm_state_layout(0, which)
        return state[at:at + n]
    return ctx, torch.zeros(-(-rows * cols // 8) * 8, device="cuda"), state, view


@pytest.mark.parametrize("rows,cols,path", UPDATE_FORMS)
def test_huge_quotients_are_clamped_and_not_turned_into_nan(rows, cols, path):
    """m^c = beta1 L R of 1e15 to 1e29 over sqrt(v) + eps of 4e-15: the quotient overflows, the ratio is the clamp's."""
    import torch
    ctx, params, state, view = _one_block(rows, cols, path, beta1=0.9, beta2=0.0, eps=1e-20, clip=1.0, correction=0)
    view(A.STATE_L).view(rows, 3)[:, 0] = 1.0
    p = 10.0 ** torch.linspace(15, 29, cols, device="cuda")
    p[1::2] *= -1
    view(A.STATE_R).view(3, cols)[0] = p
    grads = torch.full((params.numel(),), 4e-15, dtype=torch.bfloat16, device="cuda")
    ctx.adapm_step(params, grads, state, 1)
    got = params[:rows * cols].view(rows, cols).cpu()
    assert torch.equal(got, -torch.sign(p).cpu().expand(rows, cols))
    ctx.adapm_destroy()


@pytest.mark.parametrize("rows,cols,path", UPDATE_FORMS)
def test_rows_without_a_gradient_move_by_their_momentum_when_eps_is_zero(rows, cols, path):
    """v = 0 and eps = 0: m^c = beta1 L R over zero is infinite and clamped, as long as m^c is not zero itself."""
    import torch
    ctx, params, state, view = _one_block(rows, cols, path, A.V_BLOCKMEAN, beta1=0.9, beta2=0.95, eps=0.0, clip=1.0,
                                          correction=0)
    view(A.STATE_L).view(rows, 3)[:, 0] = 1.0
    p = torch.linspace(-1e-3, 1e-3, cols, device="cuda") + 1e-6
    view(A.STATE_R).view(3, cols)[0] = p
    grads = torch.zeros(params.numel(), dtype=torch.bfloat16, device="cuda")
    grads[:rows // 2 * cols] = 1e-3
    ctx.adapm_step(params, grads, state, 1)
    got = params[:rows * cols].view(rows, cols).cpu()
    assert torch.equal(got[rows // 2:], -torch.sign(p).cpu().expand(rows - rows // 2, cols))
    assert bool(torch.isfinite(got).all())
    ctx.adapm_destroy()


@pytest.mark.parametrize("rows,cols,path", UPDATE_FORMS)
@pytest.mark.parametrize("t", [1, 2, 7])
@pytest.mark.parametrize("eps", [0.0, 1e-8])
@pytest.mark.parametrize("v_lo,v_hi,g_lo,g_hi", [(-14, -3, -8, 0), (-29.9, 29.9, -6, 6), (-31, -29, -20, -14),
                                                 (29, 31, -3, 19), (-45, -36, -20, -18)])
def test_root_and_quotient_of_the_update_against_the_functions(rows, cols, path, t, eps, v_lo, v_hi, g_lo, g_hi):
    """W = 0, lr = 1, no decay, no clamp, frozen zero factors: the step writes -(g b1) / (sqrt(v b2) + eps) with b1, b2
    the bias corrections of step t, and leaves v.  The same in numpy's fp32, whose root and quotient are rounded to
    nearest as CUDA's sqrtf and / are, has to agree to the last bit but one; in 64 bits, to the roundings of g b1, v b2,
    the root, the sum and the quotient, half an ulp each of them or of what they carry into the quotient (an ulp is up to
    2^-23 of the value, the root halves what v b2 carries): 4.5 half ulps."""
    import torch
    ctx, params, state, view = _one_block(rows, cols, path, beta1=0.9, beta2=0.95, eps=eps, clip=float("inf"), adam_debias=1)
    gen = torch.Generator(device="cuda").manual_seed(17 + t)
    n = rows * cols

    def log_uniform(lo, hi):
        return 10.0 ** (torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * (hi - lo) + lo)
    grads = torch.zeros(params.numel(), dtype=torch.bfloat16, device="cuda")
    grads[:n] = (log_uniform(g_lo, g_hi) * (2.0 * torch.randint(0, 2, (n,), generator=gen, device="cuda") - 1)).to(torch.bfloat16)
    view(A.STATE_V).copy_(log_uniform(v_lo, v_hi).float())
    ctx.adapm_step(params, grads, state, t)
    got = -params[:n].cpu().numpy()
    v, g = view(A.STATE_V).cpu().numpy(), grads[:n].float().cpu().numpy()
    ctx.adapm_destroy()
    f = np.float32
    bc1 = f(1.0 / (1.0 - float(f(0.9)) ** t))
    bc2 = f(1.0 / (1.0 - float(f(0.95)) ** t))
    with np.errstate(all="ignore"):
        want = (g * bc1) / (np.sqrt(v * bc2) + f(eps))
        exact = g.astype(np.float64) * float(bc1) / (np.sqrt(v.astype(np.float64) * float(bc2)) + float(f(eps)))
        inside = np.isfinite(want) & (np.abs(want) >= np.finfo(f).tiny) & (v >= np.finfo(f).tiny)
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    ulps = np.abs(got[inside].astype(np.float64) - want[inside]) / np.spacing(np.abs(want[inside]))
    assert ulps.max() <= 1.0
    rel = np.abs(got[inside] - exact[inside]) / np.abs(exact[inside])
    assert rel.max() <= 4.5 * 2.0 ** -24


# a block whose update outlasts the low-rank launches many times over, beside low-rank blocks of both kinds of rows
FORKED = [(32768, 4096, A.MOM_NONE, 0, A.V_BLOCKMEAN, 1), (264, 264, A.MOM_LOWRANK, 16, A.V_BLOCKMEAN, 8),
          (300, 267, A.MOM_LOWRANK, 12, A.V_BLOCKMEAN, 1)]


class _Copies:
    """The same steps on one stream, launch after launch (the per-launch events switch the second stream off), and as a user
    takes them."""

    def __init__(self, dtype, stream, **hp):
        import torch
        gd, td = (A.GRAD_F32, torch.float32) if dtype == "f32" else (A.GRAD_BF16, torch.bfloat16)
        blocks = _blocks(FORKED)
        n = -(-(blocks[-1].offset + blocks[-1].rows * blocks[-1].cols) // 8) * 8
        gen = torch.Generator(device="cuda").manual_seed(5)
        self.given = torch.randn(n, generator=gen, device="cuda").mul_(1e-3).to(td)
        self.one, self.user = [], []
        for kept in (self.one, self.user):
            ctx = A.adapm_create(blocks, A.hparams(grad_dtype=gd, max_grad_norm=1.0, **hp))
            state = torch.empty(ctx.adapm_state_bytes() // 4, device="cuda")
            work = torch.zeros(ctx.adapm_workspace_bytes() // 4, device="cuda")
            ctx.adapm_set_workspace(work)
            ctx.adapm_state_init(state)
            kept += [ctx, torch.full((n,), 0.02, device="cuda"), self.given.clone(), state]
        self.one[0].adapm_set_profiling(True)
        torch.cuda.synchronize()
        self.stream, self.t = stream, 0

    def expected(self):
        import torch
        ctx, params, grads, state = self.one
        self.t += 1
        ctx.adapm_step(params, grads, state, self.t)
        torch.cuda.synchronize()
        return params, state

    def close(self):
        for kept in (self.one, self.user):
            assert kept[0].adapm_get_status() == 0
            kept[0].adapm_destroy()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_work_behind_a_step_on_the_callers_stream_waits_for_all_of_it(dtype):
    """The copies that follow a step see what it wrote, and what overwrites the gradients does not reach it."""
    import torch
    stream = torch.cuda.Stream()
    c = _Copies(dtype, stream)
    ctx, params, grads, state = c.user
    for _ in range(3):
        want_p, want_s = c.expected()
        with torch.cuda.stream(stream):
            ctx.adapm_step(params, grads, state, c.t)
            got_p, got_s = params.clone(), state.clone()
            grads.zero_()
            grads.copy_(c.given)
        stream.synchronize()
        assert torch.equal(got_p, want_p) and torch.equal(got_s, want_s)
        torch.cuda.synchronize()
        assert torch.equal(params, got_p) and torch.equal(state, got_s)
    c.close()


@pytest.mark.parametrize("dtype,flags", [("f32", 0), ("bf16", 0), ("bf16", A.FLAG_FORCE_PANEL_TEAMS)])
def test_a_step_captured_in_a_graph(dtype, flags):
    """Two steps, a captured one that is replayed, and one more, against the same steps launch by launch."""
    import torch
    stream = torch.cuda.Stream()
    c = _Copies(dtype, stream, flags=flags)
    ctx, params, grads, state = c.user
    for t in (1, 2, 3, 4):
        want_p, want_s = c.expected()
        if t == 3:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                ctx.adapm_step(params, grads, state, t)
            with torch.cuda.stream(stream):
                graph.replay()
        else:
            with torch.cuda.stream(stream):
                ctx.adapm_step(params, grads, state, t)
        torch.cuda.synchronize()
        assert torch.equal(params, want_p) and torch.equal(state, want_s)
    del graph
    c.close()


def test_contexts_of_different_shapes_side_by_side():
    """Shared-memory needs differ by rank, by kind of v and by form of the apply kernel: contexts made later, larger or
    smaller, leave the earlier ones working."""
    runs = [ParityRun(WL.Workload(f"c{i}", [], "bf16", "normal", steps=2), True, custom_blocks=_blocks([spec]))
            for i, spec in enumerate([(264, 328, A.MOM_LOWRANK, 128, A.V_ELEMENT, 0), (264, 264, A.MOM_LOWRANK, 200, A.V_BLOCKMEAN, 1),
                                      (300, 333, A.MOM_LOWRANK, 40, A.V_BLOCKMEAN, 1), (264, 264, A.MOM_LOWRANK, 8, A.V_BLOCKMEAN, 1)])]
    try:
        for _ in range(2):
            for run in runs:
                run.step()
                run.compare()
    finally:
        for run in runs:
            run.close()
