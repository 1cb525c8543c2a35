"""The kernel that a batched plan takes by default, at the sizes where the rule changes (40,704 queries fit the
join whatever k is, 51,968 for k up to 10; the few-pairs rule holds within that), and its matches against another
kernel's on the same set."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import ch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top_k", [10, 32])
def test_default_kernel_by_sizes(ch, top_k):  # noqa: F811
    sizes = [40000, 52000, 65535, 65536, 300]
    s = synth.random_set(1616, sizes, copy_frac=0.0)
    p = ch.cashash_default_params(schedule=1, top_k=top_k)
    ctx = ch.cashash_create(p, s.R)
    ds = ch.DeviceSet(p, s.img_off, s.desc)
    ch.cashash_build_codes(ctx, ds)
    W, J, Q = ch.CASHASH_KERNEL_WARP, ch.CASHASH_KERNEL_JOIN, ch.CASHASH_KERNEL_QUERY
    for pairs, want in (([[0, 4]], W), ([[4, 2]], W), ([[4, 3]], J), ([[1, 4]], Q), ([[2, 4], [4, 0]], Q),
                        ([[4, 1], [0, 4], [4, 4]], W), ([[4, 1], [4, 2], [4, 4], [4, 0]], J), ([[3, 4]], Q)):
        pairs = np.array(pairs, np.uint32)
        cap = int(s.sizes()[pairs[:, 0]].sum())
        plan = ch.cashash_plan_create(ctx, ds, pairs)
        assert ch.cashash_plan_get_tuning(plan)["kernel"] == want, pairs
        lists = []
        for kernel in (0, Q if want == W else W):
            if kernel:
                ch.cashash_plan_set_tuning(plan, kernel)
            moff = torch.zeros(len(pairs) + 1, dtype=torch.int64, device="cuda")
            mt = torch.zeros((cap, 2), dtype=torch.int32, device="cuda")
            ch.cashash_match_plan(ctx, plan, moff, mt, cap)
            assert ch.cashash_sync_status(ctx) == ch.CASHASH_OK
            lists.append((moff.cpu().numpy(), mt[:int(moff[-1])].cpu().numpy()))
        assert np.array_equal(lists[0][0], lists[1][0]) and np.array_equal(lists[0][1], lists[1][1])
        plan.close()
    ctx.close()
