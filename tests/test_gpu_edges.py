"""Sizes where a kernel variant or a dispatch rule changes, against the oracle."""
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


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("rank", [1, 8, 9, 24, 40, 41, 81, 300])
def test_exact_fp32_refit_at_the_edges_of_its_tiles(rank, dtype):
    """Column tiles of every width, one to eight of them, K loops that are cut and that are not, aligned and
    unaligned rows."""
    big = rank > 64
    _follow([(130, 1030 if not big else 330, A.MOM_LOWRANK, min(rank, 130), A.V_BLOCKMEAN, 1),
             (400, 517 if not big else 380, A.MOM_LOWRANK, rank, A.V_ELEMENT, 0),
             (304, 304, A.MOM_LOWRANK, rank, A.V_BLOCKMEAN, 0)], dtype=dtype, path=A.PATH_SIMT)


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


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_streaming_update_at_the_edges_of_its_teams(dtype):
    """Groups that one, two, four and eight warps hold, and one element more and less."""
    sizes = [2047, 2048, 2049, 4096, 4097, 4104, 8192, 8200, 16384, 16385]
    _follow([(5 if n % 2 else 6, n, A.MOM_FULL if i % 3 else A.MOM_NONE, 0, A.V_BLOCKMEAN, 1)
             for i, n in enumerate(sizes)], dtype=dtype)
