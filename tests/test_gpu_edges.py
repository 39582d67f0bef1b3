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
