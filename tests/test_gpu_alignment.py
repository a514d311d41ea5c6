"""GPU parity of the wide paths for buffers off a 16-byte boundary, at the
sizes where they can go wrong: lengths around a vector, a unit and a tile, and
every kind of offset of either side."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_21686_gb300 import pcs
from helpers import u64

pytestmark = pytest.mark.gpu

OFFSETS = [0, 1, 2, 3, 4, 7, 8, 11, 12, 15]


def _arena(n, seed, dev):
    h = torch.randint(0, 256, (n,), generator=torch.Generator().manual_seed(seed), dtype=torch.uint8)
    return h, h.to(dev)


@pytest.mark.parametrize("oa", OFFSETS)
def test_mismatch_of_offset_pairs(ctx, dev, oa):
    # Differences at the first and the last byte of a pair and in between.
    sizes = [0, 1, 5, 15, 16, 17, 31, 32, 33, 47, 48, 63, 2047, 2048, 2049, 2064, 2079, 4096 + 15,
             6 * 2048 + 16, 70001]
    ha, da = _arena(70100, 1, dev)
    a, b, want = [], [], []
    for ob in OFFSETS:
        for n in sizes:
            hb = ha[oa:oa + n].clone()
            for at in {0, n - 1, n // 2, n // 3, n - 16, n - 17, 16}:
                if 0 <= at < n:
                    hb[at] ^= 1 + (at + ob) % 255
            full = torch.zeros(ob + n + 3, dtype=torch.uint8)
            full[ob:ob + n] = hb
            a.append(da[oa:oa + n])
            b.append(full.to(dev)[ob:ob + n])
            want.append(int((hb != ha[oa:oa + n]).sum()))
            assert want[-1] == oracle.mismatch(ha[oa:oa + n].numpy(), hb.numpy())
    assert ctx.mismatch(a, b).cpu().tolist() == want
    assert ctx.mismatch(a, b).cpu().tolist() == want  # the scratch sums start over
