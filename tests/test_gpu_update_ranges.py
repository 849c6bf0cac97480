"""The update's walk over the layer table: many short layers with gaps in a block's range, layers that end inside a group
of four, and arenas at the edges of one and two rounds a block.  One call over all layers against one call for each: the
same arithmetic per element, so the same bits, and nothing outside the layers changes."""
import pytest
import torch

import paper_2607_01125_gb300 as zo
from synth import normal

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = zo.Context(0)
    yield c
    assert c.device_status() == 0
    c.close()


def _short(n):
    blocks, at = [], 4
    for i in range(n):
        d_out, r = 1 + i % 7, 1 + i % 3
        blocks.append((at, d_out, r, 5 * i + 1))
        at += (d_out * r + 3) // 4 * 4 + 4 * (i % 4)      # gaps of up to three groups
    return blocks


@pytest.mark.parametrize("queries", [1, 5])
@pytest.mark.parametrize("blocks", [
    _short(300),                                                    # two tables; layers of 1 to 21 elements
    _short(40) + [(4096, 1001, 3, 7)] + [(8192 + 4 * i, 1, 1, i) for i in range(100)],
    [(0, 152 * 8 * 1024, 1, 3)],                                    # one round of the blocks
    [(0, 152 * 8 * 1024 + 5, 1, 3), (1300000, 7, 9, 4)],            # a group more
])
def test_layer_walk(ctx, blocks, queries):
    n = (max(b[0] + b[1] * b[2] for b in blocks) + 67) // 4 * 4
    arena = [normal((n,), 1, DEV), normal((n,), 2, DEV, std=0.01), normal((n,), 3, DEV).abs()]
    a = normal((queries,), 4, DEV).double()
    qs = list(range(2, 2 + queries))
    for sgd in (False, True):
        one, each = [t.clone() for t in arena], [t.clone() for t in arena]

        def update(t, bl):
            if sgd:
                zo.zoact_sgd_step_multi(ctx, t[0], bl, a, qs, 1e-2, 9)
            else:
                zo.zoact_adam_step_multi(ctx, *t, bl, a, qs, 1e-2, 0.9, 0.999, 1e-8, 3, 9)

        update(one, blocks)
        for b in blocks:
            update(each, [b])
        torch.cuda.synchronize()
        inside = torch.zeros(n, dtype=torch.bool, device=DEV)
        for off, d_out, r, _ in blocks:
            inside[off:off + d_out * r] = True
        for x, y, z in zip(one, each, arena):
            assert torch.equal(x, y)
            assert torch.equal(x[~inside], z[~inside])
        # (a change below half an ulp leaves an element as it was)
        assert float((one[0][inside] != arena[0][inside]).double().mean()) > 0.99
