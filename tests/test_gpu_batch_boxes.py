"""hpsi_apply_batch over boxes of different edges: one launch of the plane kernel serves all items, with the block size of
the item with the largest planes and the code instance of the item with the largest radix, whose launch bound is
smaller.  Each pair below asks for a larger block than that bound (plane_shape gives 672 to 1024 threads)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _cell(n, mmax):
    """A cubic cell of box edge n whose sphere has Miller indices up to mmax."""
    ecut = 8.0
    a = 2.0 * np.pi * (mmax + 0.3) / np.sqrt(2.0 * ecut)
    return np.diag([a, a, a]), ecut, (n, n, n)


# float64: radices above 10 hold 512 threads; float32: radices above 12 hold 768
@pytest.mark.parametrize("precision,boxes", [
    (0, [(72, 31), (48, 5)]), (0, [(81, 30), (60, 5)]), (0, [(100, 26), (96, 5), (25, 5)]),
    (1, [(144, 33), (75, 5)]), (1, [(120, 45), (80, 5)])])
@pytest.mark.parametrize("nb", [1, 2])
def test_unequal_boxes_match_single_calls(lib, precision, boxes, nb):
    import torch
    from paper_0906_2569_gb300 import binding as B
    cells = [_cell(n, mmax) for n, mmax in boxes]
    rng = np.random.default_rng(len(boxes) + nb)
    vrs = [rng.standard_normal(c[2]) for c in cells]
    ms = [B.hpsi_gsphere(c[0], c[1], np.zeros(3)) for c in cells]
    ctx = B.hpsi_setup_cells([c[0] for c in cells], [c[1] for c in cells], [c[2] for c in cells], vrs,
                             [None] * len(cells), [None] * len(cells), precision, torch.cuda.current_stream().cuda_stream)
    xs = [torch.from_numpy(workloads.random_block(len(m), nb, i)).cuda() for i, m in enumerate(ms)]
    each = [torch.full_like(x, float("nan")) for x in xs]
    for i, x in enumerate(xs):
        B.hpsi_apply(ctx, i, x, each[i])
    ys = [torch.empty_like(x) for x in xs]
    for _ in range(2):   # eager with capture, then the replay
        for y in ys:
            y.fill_(float("nan"))
        B.hpsi_apply_batch(ctx, list(range(len(xs))), xs, ys)
        B.hpsi_sync(ctx)
        for y, e in zip(ys, each):
            assert torch.equal(y, e)
    ctx.close()
