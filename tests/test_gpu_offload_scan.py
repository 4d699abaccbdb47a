"""A whole offload step whose first fetch finds the distinct ids itself (batches of up to 256 tokens; one more takes the dedup
kernel), and its groups of layers, at the edges of warps, of the vector comparisons and of the grouping."""
import numpy as np
import pytest
import torch

import oracle
from paper_2503_15798_b200 import binding as mole

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,L,cap,few", [(1, 9, 256, 1), (3, 16, 256, 2), (31, 5, 256, 9), (33, 24, 256, 40), (64, 9, 200, 1000), (100, 4, 256, 1),
                                         (255, 3, 256, 130), (256, 2, 256, 1000), (257, 2, 257, 130)])
def test_scanned_ids_and_groups_of_layers(M, L, cap, few):
    N, d, V = 16, 512, 1000
    g = torch.Generator().manual_seed(M)
    host = mole.HostTable((L, V, N, d), torch.bfloat16)
    ctx = mole.OffloadContext(max_tokens=cap, N=N, d=d, V=V, n_buffers=2)
    side = torch.cuda.Stream()
    try:
        host.tensor.copy_(torch.empty(L, V, N, d).normal_(0, 0.05, generator=g).to(torch.bfloat16))
        wrs = torch.empty(L, d, N).normal_(0, 0.02, generator=g).to(torch.bfloat16).cuda()
        hidden = torch.empty(M, d).normal_(0, 1, generator=g).to(torch.bfloat16).cuda()
        ids_np = np.random.default_rng(M).integers(0, few, M).astype(np.int32) * (V // few)
        if M > 2:
            ids_np[M // 2], ids_np[M - 1] = -1, V  # no row of the table
        ids, luts = torch.from_numpy(ids_np).cuda(), host.tensor.cuda()
        out, tmp, status = torch.empty_like(hidden), torch.empty_like(hidden), torch.zeros(1, dtype=torch.int32, device="cuda")
        for _ in range(2):
            ctx.decode_step(hidden, ids, host.tensor, wrs, out, tmp, status=status, side_stream=side)
        h = hidden
        for l in range(L):
            h = mole.layer_forward(h, ids, luts[l], wrs[l], kernel=mole.KERNEL_RING)
        uniq, slot, n = ctx.read_buffer(0)
        assert torch.equal(out, h)  # the same kernel on the same rows: the same bytes
        ok = (ids_np >= 0) & (ids_np < V)
        want_uniq, want_slot = oracle.dedup(ids_np[ok])
        slot = np.asarray(slot)[:M]
        assert n == len(want_uniq) and (np.asarray(uniq)[:n] == want_uniq).all()
        assert (slot[ok] == want_slot).all() and (slot[~ok] == -1).all()
        assert int(status.item()) == (0 if ok.all() else mole.STATUS_BAD_ID)
    finally:
        ctx.destroy()
        host.free()
