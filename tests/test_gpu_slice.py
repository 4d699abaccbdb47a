"""The kernels of the two narrow widths (16 experts, d = 768 and 1024): a cluster of two blocks, a block and half a block per token, on
both sides of each line, against the oracle's chain; a token's bits in every batch and in single, chained and fused launches; ids
outside the table beside a valid one; bounded waits; and the fused step of the widest layer (32 x 2048): the bits of the step it
stands beside, and slots that fill slowly."""
import numpy as np
import pytest
import torch

from gpu_util import as_f64, check_gates, check_out, oracle_layer
from paper_2503_15798_b200 import binding as mole
from test_gpu_variants import _oracle_chain

pytestmark = pytest.mark.gpu
DEV = "cuda"
N, V, SMS = 16, 61, 148
COUNTS = [1, SMS // 2, SMS // 2 + 1, SMS, SMS + 1, 2 * SMS + 1, 4 * SMS, 4 * SMS + 3]


def _case(d, M, L, norm):
    g = torch.Generator().manual_seed(d + M + L)
    luts = torch.empty(L, V, N, d).normal_(0, 0.05, generator=g).to(torch.bfloat16)
    wrs = torch.empty(L, d, N).normal_(0, 0.02, generator=g).to(torch.bfloat16)
    hidden = (1.5 * torch.empty(M, d).normal_(0, 1, generator=g)).to(torch.bfloat16)
    ids = torch.randint(0, V, (M,), generator=g, dtype=torch.int32)
    gammas = (1.0 + 0.2 * torch.empty(L, d).normal_(0, 1, generator=g)).to(torch.bfloat16) if norm else None
    return luts, wrs, hidden, ids, gammas


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("d", [768, 1024])
def test_steps_against_the_oracles_chain_and_bits_in_every_batch(d, norm):
    L, M = 3, COUNTS[-1]
    luts, wrs, hidden, ids, gammas = _case(d, M, L, norm)
    ids[0] = -1      # the first of a pair, and
    ids[3] = V       # the second, beside valid ones
    ids[M - 1] = V   # and one that is alone in its block
    ref, _, _ = _oracle_chain(hidden, ids, luts, wrs, gammas, 1e-5)
    h, i, lu, w = hidden.to(DEV), ids.to(DEV), luts.to(DEV), wrs.to(DEV)
    gam = None if gammas is None else gammas.to(DEV)
    outs = {}
    for M in COUNTS:
        for mode in (mole.STEP_FUSED, mole.STEP_CHAINED):
            x, status = h[:M].contiguous(), torch.zeros(1, dtype=torch.int32, device=DEV)
            out = mole.decode_step_args(x, i[:M].contiguous(), lu, w, torch.empty_like(x), torch.empty_like(x), status=status, mode=mode, norm_weights=gam, norm_eps=1e-5)
            assert int(status.item()) == mole.STATUS_BAD_ID
            outs[M, mode] = out
    last = outs[COUNTS[-1], mole.STEP_FUSED]
    err = np.abs(as_f64(last) - ref)
    slack = L * 1e-3 * float(luts.abs().max()) * N if norm else 0.0  # a rounding tie in a normalised element moves a gate
    assert (err <= L * 2.0 ** -7 * np.maximum(1.0, np.abs(ref)) + slack).all(), float(err.max())
    for (M, mode), out in outs.items():
        assert torch.equal(out, last[:M]), (M, mode)
    for t in (0, 3, COUNTS[-1] - 1):
        assert torch.equal(last[t], h[t])


@pytest.mark.parametrize("M", [1, SMS, SMS + 2, 301, 4 * SMS + 1, 6 * SMS, 1501])
@pytest.mark.parametrize("d", [768, 1024])
def test_single_layer_with_gates_residual_and_wide_ids(d, M):
    """One token or two per block, and blocks that walk several pairs."""
    luts, wrs, hidden, ids, _ = _case(d, M, 1, False)
    res = torch.empty(M, d).normal_(0, 1, generator=torch.Generator().manual_seed(M)).to(torch.bfloat16)
    ref, gref, _ = oracle_layer(hidden, ids, luts[0], wrs[0], residual=res)
    gates = torch.zeros(M, N, dtype=torch.float32, device=DEV)
    out = mole.layer_forward(hidden.to(DEV), ids.long().to(DEV), luts[0].to(DEV), wrs[0].to(DEV), residual=res.to(DEV), gates_out=gates, kernel=mole.KERNEL_RING)
    check_out(out, ref)
    check_gates(gates, gref)


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("d", [768, 1024])
def test_layers_of_blocks_that_walk_several_pairs(d, norm):
    """1501 tokens, up to three pairs per block and one token left over: chained, in place, with residual, ids outside the table anywhere;
    every token has the bits it has among few."""
    M = 1501
    luts, wrs, hidden, ids, gammas = _case(d, M, 2, norm)
    bad = [0, 2 * 2 * SMS + 1, 700, 1199, M - 1]
    ids[bad] = torch.tensor([-1, V, V + 7, -5, V], dtype=torch.int32)
    h, i, lu, w = hidden.to(DEV), ids.to(DEV), luts.to(DEV), wrs.to(DEV)
    res = torch.empty(M, d, device=DEV).normal_(0, 1, generator=torch.Generator(device=DEV).manual_seed(2)).to(torch.bfloat16)
    gam = [None, None] if gammas is None else list(gammas.to(DEV))

    def layers(s, status):
        x = h[s].clone()
        mole.layer_forward(x, i[s], lu[0], w[0], out=x, norm_weight=gam[0], norm_eps=1e-5, kernel=mole.KERNEL_RING, status=status)
        return mole.layer_forward(x, i[s], lu[1], w[1], residual=res[s], norm_weight=gam[1], norm_eps=1e-5, kernel=mole.KERNEL_RING, status=status, chain=True)

    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    out = layers(slice(0, M), status)
    assert int(status.item()) == mole.STATUS_BAD_ID
    for a, n in ((0, 1), (5, 40), (593, 300), (1301, 200)):
        assert torch.equal(layers(slice(a, a + n), None), out[a:a + n]), (a, n)
    assert torch.equal(out[bad], res[bad])


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("d", [768, 1024])
def test_waits_of_the_cluster_that_run_out_are_reported(d, norm):
    """No polls allowed: the waits for the other block's logits give up.  The launch returns, reports it, writes nothing beyond its
    rows, and the next launch is right."""
    M, L, guard = 5, 6, 3
    luts, wrs, hidden, ids, gammas = _case(d, M, L, norm)
    x, i, lu, w = hidden.to(DEV), ids.to(DEV), luts.to(DEV), wrs.to(DEV)
    gam = None if gammas is None else gammas.to(DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    buf = torch.full((M + 2 * guard, d), 12345.0, dtype=torch.bfloat16, device=DEV)
    out = buf[guard:guard + M]

    def step(o):
        return mole.decode_step_args(x, i, lu, w, o, None, status=status, mode=mole.STEP_FUSED, norm_weights=gam, norm_eps=1e-5)

    want = step(torch.empty_like(x)).clone()
    with mole.debug_env(MOLE_DEBUG_WAIT_LIMIT=-1):
        step(out)
        torch.cuda.synchronize()
    assert int(status.item()) & mole.STATUS_TIMEOUT
    assert (buf[:guard] == 12345.0).all() and (buf[guard + M:] == 12345.0).all()
    status.zero_()
    step(out)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and torch.equal(out, want)


def _peaked(N, d, M, L, seed, norm):
    """Tables of standard deviation 1 and routers that favour other experts in every layer: a router matrix of another layer, or parts of
    one, shows far above a rounding."""
    g = torch.Generator().manual_seed(seed)
    luts = torch.empty(L, V, N, d).normal_(0, 1, generator=g).to(torch.bfloat16)
    wrs = torch.empty(L, d, N).normal_(0, 3.0 / d ** 0.5, generator=g).to(torch.bfloat16)
    hidden = torch.empty(M, d).normal_(0, 1, generator=g).to(torch.bfloat16)
    ids = torch.randint(0, V, (M,), generator=g, dtype=torch.int32)
    gammas = (1.0 + 0.2 * torch.empty(L, d).normal_(0, 1, generator=g)).to(torch.bfloat16) if norm else None
    return luts, wrs, hidden, ids, gammas


def _fused(h, i, lu, w, gam):
    return mole.decode_step_args(h, i, lu, w, torch.empty_like(h), None, mode=mole.STEP_FUSED, norm_weights=gam, norm_eps=1e-5)


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("L", [2, 3, 16])
def test_widest_step_has_the_same_bits_on_both_sides_of_its_line(L, norm):
    """32 x 2048: up to 37 tokens a kernel with the sizes compiled in, beyond it the general tensor-core step."""
    few, many = SMS // 4, SMS // 4 + 27
    luts, wrs, hidden, ids, gammas = _peaked(32, 2048, many, L, 7 * L + norm, norm)
    h, i, lu, gam = hidden.to(DEV), ids.to(DEV), luts.to(DEV), None if gammas is None else gammas.to(DEV)
    want = _fused(h, i, lu, wrs.to(DEV), gam)
    for M in (1, few - 1, few, few + 1):
        for _ in range(3):  # routers in memory that no launch has read yet
            assert torch.equal(_fused(h[:M].contiguous(), i[:M].contiguous(), lu, wrs.to(DEV), gam), want[:M]), M


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("L", [2, 7])
def test_widest_step_against_the_oracles_chain(L, norm):
    """Entries of standard deviation 1, so that the routed term is what is compared: a bf16 rounding per layer, carried into the
    layers after it by gates whose logits have a standard deviation of 3 and more."""
    M = 6
    luts, wrs, hidden, ids, gammas = _peaked(32, 2048, M, L, 31 + L, norm)
    ref, _, _ = _oracle_chain(hidden, ids, luts, wrs, gammas, 1e-5)
    out = _fused(hidden.to(DEV), ids.to(DEV), luts.to(DEV), wrs.to(DEV), None if gammas is None else gammas.to(DEV))
    rel = np.linalg.norm(as_f64(out) - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert rel.max() <= L * 2.0 ** -7, rel


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("N,d,M", [(32, 2048, 1), (32, 2048, SMS // 4), (16, 1024, 5), (16, 768, 100), (16, 1024, SMS + 3)])
def test_slots_that_fill_slowly(N, d, M, norm):
    """Routers, then tables too, in pinned host memory, which the kernel reads across the link: copies that take many layers' time, of
    which none may be used before it has landed or overwritten before it is read."""
    L = 9
    luts, wrs, hidden, ids, gammas = _peaked(N, d, M, L, M + d, norm)
    h, i, lu, gam = hidden.to(DEV), ids.to(DEV), luts.to(DEV), None if gammas is None else gammas.to(DEV)
    want = _fused(h, i, lu, wrs.to(DEV), gam)
    slow_w = wrs.pin_memory()
    for table in (lu, luts.pin_memory()):
        for _ in range(3):
            out = _fused(h, i, table, slow_w, gam)
            torch.cuda.synchronize()
            assert torch.equal(out, want)


# a cluster of two blocks per token, a block, half a block (the neighbour of an extreme token is an ordinary one), blocks that walk pairs
@pytest.mark.parametrize("M", [11, 100, 301, 4 * SMS + 2])
@pytest.mark.parametrize("d", [768, 1024])
def test_extreme_tokens_beside_ordinary_ones(d, M):
    """Every second token has infinite table entries, or logits far beyond +-60, or (with the norm) a sum of squares that overflows: what
    it gives is what such values mean, and the token beside it has the bits it has in a launch without them."""
    L = 2
    luts, wrs, hidden, _, gammas = _case(d, M, L, True)
    ids = torch.arange(M, dtype=torch.int32) % 20
    odd = torch.arange(M) % 2 == 1
    ids[odd] = 20 + ids[odd]
    i, w, gam = ids.to(DEV), wrs.to(DEV), gammas.to(DEV)
    modes = (mole.STEP_FUSED, mole.STEP_CHAINED)

    def step(lu, h, routers, g, mode):
        return mole.decode_step_args(h, i, lu, routers, torch.empty_like(h), torch.empty_like(h), mode=mode, norm_weights=g, norm_eps=1e-6, kernel=mole.KERNEL_RING).cpu()

    plain, h = luts.to(DEV), hidden.to(DEV)
    # infinite entries, under a router of zeros (numerators of exactly 1, two of whose three parts are zero) and under an ordinary one
    inf = luts.clone()
    want = torch.zeros(M, d)
    for row in range(20, 40):
        for col, sign in ((row, 1.0), (d - 1 - 7 * row, -1.0), (d // 2 + row, 1.0)):
            inf[L - 1, row, row % N, col] = sign * float("inf")
            want[ids == row, col] = sign * float("inf")
    for routers in (torch.zeros_like(w), w):
        for mode in modes:
            out, ordinary = step(inf.to(DEV), h, routers, None, mode), step(plain, h, routers, None, mode)
            assert torch.equal(torch.isinf(out), torch.isinf(want)) and not torch.isnan(out).any()
            assert torch.equal(out[torch.isinf(want)].float(), want[torch.isinf(want)])
            assert torch.equal(out[~odd], ordinary[~odd])
            assert torch.equal(out[~torch.isinf(want)], ordinary[~torch.isinf(want)])
    # logits of hundreds: the gates are those of the largest, and the neighbour's bits do not move
    big = hidden.clone()
    big[odd] *= 300.0
    ref, gref, _ = oracle_layer(big, ids, luts[0], wrs[0])
    assert gref[odd.numpy()].max() > 0.999
    gates = torch.zeros(M, N, dtype=torch.float32, device=DEV)
    one = mole.layer_forward(big.to(DEV), i, plain[0], w[0], gates_out=gates, kernel=mole.KERNEL_RING)
    # a logit of z carries |z| 2^-22 of fp32 rounding, and so does a gate relative to itself
    slack = 2.0 ** -20 * np.abs(as_f64(big) @ as_f64(wrs[0])).max(axis=1, keepdims=True)
    assert (np.abs(as_f64(gates) - gref) <= 1e-5 + slack).all()
    assert (np.abs(as_f64(one) - ref) <= 2.0 ** -8 * np.abs(ref) + 2e-5 + slack * N * float(luts.abs().max())).all()
    for mode in modes:
        assert torch.equal(step(plain, big.to(DEV), w, None, mode)[~odd], step(plain, h, w, None, mode)[~odd])
    # an overflowing sum of squares: the normalised state is zero and the gates are 1 / N
    over = hidden.clone()
    over[odd, 7], over[odd, d - 1] = 2e19, -3e38
    gates.zero_()
    mole.layer_forward(over.to(DEV), i, plain[0], w[0], gates_out=gates, norm_weight=gam[0], norm_eps=1e-6, kernel=mole.KERNEL_RING)
    assert (gates[odd.to(DEV)] == 1.0 / N).all()
    for mode in modes:
        out, ordinary = step(plain, over.to(DEV), w, gam, mode), step(plain, h, w, gam, mode)
        assert torch.equal(out[~odd], ordinary[~odd])
        for t in torch.nonzero(odd).flatten().tolist()[:6]:
            r = as_f64(over[t])
            for l in range(L):  # each layer's output is rounded once
                r = as_f64(torch.from_numpy(r + as_f64(luts[l, int(ids[t])]).mean(axis=0)).to(torch.bfloat16))
            # a rounding tie of a layer may fall the other way: an ulp of bf16 per layer
            assert (np.abs(as_f64(out[t]) - r) <= L * 2.0 ** -7 * np.maximum(1.0, np.abs(r))).all(), (mode, t)


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("n,d,M", [(16, 768, 9), (16, 1024, 100), (16, 768, 4 * SMS + 3), (32, 2048, 20)])
def test_layers_that_share_a_table_or_lie_apart(n, d, M, norm):
    """Strides of zero (one table, router and scale for all layers) and layers with other memory between them."""
    L = 4
    luts, wrs, hidden, ids, gammas = _peaked(n, d, M, 2 * L, d + M, norm)
    h, i, lu, w, gam = hidden.to(DEV), ids.to(DEV), luts.to(DEV), wrs.to(DEV), None if gammas is None else gammas.to(DEV)
    strided = (lu[::2], w[::2], None)
    shared = (lu[1:2].expand(L, -1, -1, -1), w[1:2].expand(L, -1, -1), None if gam is None else gam[1:2].repeat(L, 1))
    for a, b, g in (strided, shared):
        if gam is not None and g is None:
            g = gam[::2].contiguous()
        for mode in (mole.STEP_FUSED, mole.STEP_CHAINED):
            def step(x, y):
                return mole.decode_step_args(h, i, x, y, torch.empty_like(h), torch.empty_like(h), mode=mode, norm_weights=g, norm_eps=1e-5)

            assert torch.equal(step(a, b), step(a.contiguous(), b.contiguous()))
