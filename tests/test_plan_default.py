"""The plans that plan_rows 0 gives, on the host: pieces of 1 and 2 rows where 8-row ones would leave
blocks idle, every node exactly once."""
import numpy as np
import pytest

from paper_1903_01168_gb300 import lbm as L

rng = np.random.default_rng(11)
SETS = {
    "one_64": [(64, 64)],
    "one_channel": [(2048, 128)],
    "ragged": [(1000, 301)],
    "short": [(8, 4), (33, 7), (130, 5)],
    "sweep": [(256, 256)] * 40,
    "uneven": [(int(rng.integers(2, 17)) * 32, int(rng.integers(2, 33)) * 32) for _ in range(32)],
}


@pytest.mark.parametrize("name", SETS)
@pytest.mark.parametrize("plan", [L.LBM_PLAN_AUTO, L.LBM_PLAN_BALANCED, L.LBM_PLAN_SPLIT])
@pytest.mark.parametrize("max_blocks", [1, 97, 912])
def test_default_pieces_cover_every_node_once(name, plan, max_blocks):
    sizes = SETS[name]
    blocks, items = L.lbm_plan_preview(sizes, max_blocks, plan=plan, plan_rows=[0] * len(sizes))
    cover = [np.zeros((ny, nx), np.int32) for nx, ny in sizes]
    for m, x0, w, ya, yb, _ in items:
        assert 0 < w <= 128 and x0 % 128 == 0 and 0 <= ya < yb
        cover[m][ya:yb, x0:x0 + w] += 1
    assert all((c == 1).all() for c in cover)
    assert blocks <= max_blocks and set(items[:, 5]) <= set(range(blocks))


def heights(sizes, max_blocks=912):
    _, items = L.lbm_plan_preview(sizes, max_blocks, plan_rows=[0] * len(sizes))
    return sorted(set(items[:, 4] - items[:, 3]))


def test_short_pieces_where_blocks_would_be_idle():
    assert heights([(64, 64)]) == [1]
    assert heights([(256, 256)]) == [2]                  # single rows only up to a third of the blocks
    assert heights([(2048, 128)]) == [2, 3]              # as short as the blocks allow
    assert min(heights([(256, 256)] * 40)) >= 8          # the blocks are full with 8 rows


def test_members_rows_keep_their_own_minimum():
    _, items = L.lbm_plan_preview([(256, 256), (256, 256)], 912, plan_rows=[16, 0])
    rows = items[:, 4] - items[:, 3]
    assert (rows[items[:, 0] == 0] >= 16).all() and (rows[items[:, 0] == 1] == 2).all()


@pytest.mark.gpu
@pytest.mark.parametrize("storage", [L.LBM_F32, L.LBM_F16DEV])
@pytest.mark.parametrize("name", ["one_64", "one_channel", "ragged", "uneven"])
def test_preview_has_the_items_of_the_batch(name, storage):
    torch = pytest.importorskip("torch")
    resident = 6 * torch.cuda.get_device_properties(0).multi_processor_count   # six blocks per SM
    if storage == L.LBM_F32 and sum(a * b for a, b in SETS[name]) >= 1500000:
        resident = resident * 5 // 6
    sims = [L.Simulation(nx, ny, gamma=2.0, storage=storage) for nx, ny in SETS[name]]
    b = L.Batch(sims)
    try:
        blocks, items = L.lbm_plan_preview(SETS[name], resident, plan_rows=[0] * len(sims))
        assert b.items == len(items)
    finally:
        b.close()
        for s in sims:
            s.close()
