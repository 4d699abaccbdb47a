"""MOLE_KERNEL_RING with a given number of chunks: a token's output is the same bits in every batch, on both sides of each line
where MOLE_KERNEL_AUTO changes the kernel family, and the families it picks agree with it within a rounding."""
import pytest
import torch

from paper_2503_15798_b200 import binding as mole

pytestmark = pytest.mark.gpu
DEV = "cuda"

# N, d, L, norm, d_split, token counts with a line between every two of them, the families of MOLE_KERNEL_AUTO there
CASES = [(16, 768, 1, False, 1, (40, 888, 889), ("slice_layer", "slice_layer", "tile")),
         (16, 1024, 1, True, 1, (40, 888, 889), ("slice_layer", "slice_layer", "tile")),
         (8, 256, 1, False, 1, (3, 1184, 1185), ("step", "step", "tile")), (32, 640, 1, True, 2, (20, 296, 297), ("step", "step", "tile")),
         (32, 2048, 1, False, 4, (128, 140, 296, 297), ("cdecode", "step", "step", "tile")), (32, 1920, 1, True, 4, (148, 296, 297), ("step", "step", "tile")),
         (32, 2048, 3, False, 4, (20, 64, 75), ("slice_step", "mma", "step")), (8, 1024, 2, True, 1, (148, 296, 297), ("mma", "mma", "step")),
         (32, 512, 2, False, 1, (100, 148, 149), ("mma", "mma", "step")), (16, 768, 3, False, 1, (64, 300), ("slice_step", "slice_step"))]


@pytest.mark.parametrize("N,d,L,norm,split,counts,families", CASES)
def test_ring_bits_do_not_depend_on_the_batch(N, d, L, norm, split, counts, families):
    V, M = 64, counts[-1]
    g = torch.Generator(device=DEV).manual_seed(N + d + L)
    luts = torch.empty(L, V, N, d, device=DEV).normal_(0, 0.05, generator=g).to(torch.bfloat16)
    wrs = torch.empty(L, d, N, device=DEV).normal_(0, 0.02, generator=g).to(torch.bfloat16)
    gam = (1.0 + 0.2 * torch.empty(L, d, device=DEV).normal_(0, 1, generator=g)).to(torch.bfloat16) if norm else None
    hidden = torch.empty(M, d, device=DEV).normal_(0, 1, generator=g).to(torch.bfloat16)
    ids = torch.randint(0, V, (M,), generator=g, dtype=torch.int32, device=DEV)

    def step(m, kernel, d_split):
        return mole.decode_step_args(hidden[:m].contiguous(), ids[:m].contiguous(), luts, wrs, torch.empty(m, d, dtype=torch.bfloat16, device=DEV),
                                     mode=mole.STEP_FUSED, norm_weights=gam, norm_eps=1e-5, kernel=kernel, d_split=d_split)

    want = step(M, mole.KERNEL_RING, split)
    for m, family in zip(counts, families):
        assert mole.variant(m, N, d, L=L, norm=norm)[0].split("<")[0] == family
        assert torch.equal(step(m, mole.KERNEL_RING, split), want[:m])
        auto = step(m, mole.KERNEL_AUTO, 0).double()
        # one rounding per layer may fall the other way, and (norm) a tie of the normalised state moves a gate
        bound = L * 2.0 ** -7 * torch.clamp(want[:m].double().abs(), min=1.0) + (L * 1e-3 * float(luts.abs().max()) * N if norm else 0.0)
        assert bool(((auto - want[:m].double()).abs() <= bound).all())
