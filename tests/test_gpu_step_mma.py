"""The tensor-core step kernel (the library's choice for fused steps of one or two blocks per SM) against the oracle's
chain: one, two and four blocks per token, one to eight warps, every expert count, one block to an SM and two, RMSNorm,
ids outside the table, output in place; and its bounded waits."""
import numpy as np
import pytest
import torch

from gpu_util import as_f64, rand_case
from paper_2503_15798_b200 import binding as mole
from test_gpu_variants import _oracle_chain

pytestmark = pytest.mark.gpu
DEV = "cuda"

# N, d, M, L
CASES = [(8, 128, 1, 3), (8, 256, 290, 2), (8, 1024, 37, 3), (8, 2048, 74, 2), (8, 2048, 5, 4), (16, 128, 148, 3), (16, 640, 9, 5), (16, 1280, 74, 2),
         (16, 2048, 3, 3), (32, 128, 64, 2), (32, 512, 148, 2), (32, 768, 20, 3), (32, 1024, 74, 2), (32, 1536, 11, 3), (32, 2048, 1, 4), (32, 2048, 30, 2),
         (32, 2048, 60, 2)]


@pytest.mark.parametrize("N,d,M,L", CASES)
@pytest.mark.parametrize("norm", [False, True])
def test_fused_step_against_the_oracles_chain(N, d, M, L, norm):
    V = 83
    name = mole.variant(M, N, d, L=L, norm=norm)[0]
    assert name == (f"slice_step<32,2048,1,{int(norm)},4>" if d == 2048 and N == 32 and 4 * M <= 148 else f"mma<{N},{int(norm)},{1 if N * d <= 16384 and d <= 1024 else 2 if N * d <= 32768 else 4}>")
    g = torch.Generator().manual_seed(N * d + M + L)
    luts = torch.empty(L, V, N, d).normal_(0, 0.05, generator=g).to(torch.bfloat16)
    wrs = torch.empty(L, d, N).normal_(0, 0.02, generator=g).to(torch.bfloat16)
    hidden = (1.5 * torch.empty(M, d).normal_(0, 1, generator=g)).to(torch.bfloat16)
    ids = torch.randint(0, V, (M,), generator=g, dtype=torch.int32)
    if M > 1:
        ids[M - 1] = V  # outside the table: its routed term is dropped in every layer
    gammas = (1.0 + 0.2 * torch.empty(L, d).normal_(0, 1, generator=g)).to(torch.bfloat16) if norm else None
    ref, _, _ = _oracle_chain(hidden, ids, luts, wrs, gammas, 1e-5)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    h = hidden.to(DEV)
    gd = None if gammas is None else gammas.to(DEV)
    out = mole.decode_step_args(h, ids.to(DEV), luts.to(DEV), wrs.to(DEV), torch.empty_like(h), None, status=status, mode=mole.STEP_FUSED,
                                norm_weights=gd, norm_eps=1e-5)
    again = mole.decode_step_args(h, ids.to(DEV), luts.to(DEV), wrs.to(DEV), h, None, status=status, mode=mole.STEP_FUSED, norm_weights=gd,
                                  norm_eps=1e-5)  # in place
    torch.cuda.synchronize()
    assert int(status.item()) == (mole.STATUS_BAD_ID if M > 1 else 0)
    assert torch.equal(out, again)
    err = np.abs(as_f64(out) - ref)
    slack = L * 1e-3 * float(luts.abs().max()) * N if norm else 0.0  # a rounding tie in a normalised element moves a gate
    assert (err <= L * 2.0 ** -7 * np.maximum(1.0, np.abs(ref)) + slack).all(), float(err.max())
    if M > 1:
        assert torch.equal(out[M - 1].cpu(), hidden[M - 1])


def test_a_tokens_bits_do_not_depend_on_its_batch_and_large_logits():
    """Logits far beyond the range where the maximum has to be subtracted; tokens alone and in a batch."""
    N, d, M, L, V = 16, 512, 40, 3, 50
    _, ids, _, _ = rand_case(M, N, d, V, seed=3)
    g = torch.Generator().manual_seed(8)
    luts = torch.empty(L, V, N, d).normal_(0, 0.05, generator=g).to(torch.bfloat16)
    wrs = torch.empty(L, d, N).normal_(0, 4.0, generator=g).to(torch.bfloat16)
    hidden = torch.empty(M, d).normal_(0, 1, generator=g).to(torch.bfloat16)
    ref, gref, _ = _oracle_chain(hidden, ids, luts, wrs, None, 0.0)
    assert gref.max() > 0.999
    h, i, lu, w = hidden.to(DEV), ids.to(DEV), luts.to(DEV), wrs.to(DEV)
    out = mole.decode_step(h, i, lu, w, torch.empty_like(h))
    # a gate near 1/2 can turn over when a state's rounding moves a logit of ~90 by an ulp of the state: such tokens are few
    bad = (np.abs(as_f64(out) - ref) > L * 2.0 ** -7 * np.maximum(1.0, np.abs(ref)) + 0.02).any(axis=1)
    assert bad.mean() <= 0.1
    for t in (0, 7, M - 1):
        one = mole.decode_step(h[t:t + 1].contiguous(), i[t:t + 1].contiguous(), lu, w, torch.empty(1, d, dtype=torch.bfloat16, device=DEV))
        assert torch.equal(one[0], out[t])


@pytest.mark.parametrize("N,d,M", [(8, 256, 6), (32, 2048, 5), (16, 2048, 4)])
def test_waits_that_run_out_are_reported(N, d, M):
    """No polls allowed: every wait that is not satisfied at once gives up -- for slots, for copies, for the other blocks of the
    cluster.  The launch returns, reports it, writes nothing beyond its rows, and the next launch is right."""
    L, V, guard = 6, 20, 3
    g = torch.Generator().manual_seed(3)
    luts = torch.empty(L, V, N, d).normal_(0, 0.05, generator=g).to(torch.bfloat16).to(DEV)
    wrs = torch.empty(L, d, N).normal_(0, 0.02, generator=g).to(torch.bfloat16).to(DEV)
    hidden = torch.empty(M, d).normal_(0, 1, generator=g).to(torch.bfloat16).to(DEV)
    ids = torch.randint(0, V, (M,), generator=g, dtype=torch.int32).to(DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    buf = torch.full((M + 2 * guard, d), 12345.0, dtype=torch.bfloat16, device=DEV)
    out = buf[guard:guard + M]
    want = mole.decode_step(hidden, ids, luts, wrs, torch.empty_like(hidden)).clone()
    with mole.debug_env(MOLE_DEBUG_WAIT_LIMIT=-1):
        mole.decode_step(hidden, ids, luts, wrs, out, status=status)
        torch.cuda.synchronize()
    assert int(status.item()) & mole.STATUS_TIMEOUT
    assert (buf[:guard] == 12345.0).all() and (buf[guard + M:] == 12345.0).all()
    status.zero_()
    mole.decode_step(hidden, ids, luts, wrs, out, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and torch.equal(out, want)


@pytest.mark.parametrize("N,d", [(8, 256), (32, 2048)])
def test_norm_of_a_state_whose_sum_of_squares_overflows(N, d):
    """mean(x^2) is infinite: the normalised state is zero and the gates are 1 / N, as in every other kernel."""
    M, L, V = 9, 2, 20
    g = torch.Generator().manual_seed(4)
    luts = torch.empty(L, V, N, d).normal_(0, 0.05, generator=g).to(torch.bfloat16)
    wrs = torch.empty(L, d, N).normal_(0, 0.02, generator=g).to(torch.bfloat16).to(DEV)
    hidden = torch.empty(M, d).normal_(0, 1, generator=g).to(torch.bfloat16)
    hidden[2, 7] = 2e19
    ids = torch.randint(0, V, (M,), generator=g, dtype=torch.int32)
    ones = torch.ones(L, d, dtype=torch.bfloat16, device=DEV)
    h = hidden.to(DEV)
    ref = as_f64(hidden[2])
    for l in range(L):  # each layer's output is rounded once
        ref = as_f64(torch.from_numpy(ref + as_f64(luts[l, int(ids[2])]).mean(axis=0)).to(torch.bfloat16))
    for kernel in (mole.KERNEL_AUTO, mole.KERNEL_RING):
        out = mole.decode_step_args(h, ids.to(DEV), luts.to(DEV), wrs, torch.empty_like(h), mode=mole.STEP_FUSED, norm_weights=ones,
                                    norm_eps=1e-6, kernel=kernel)
        # a rounding tie of a layer may fall the other way: an ulp of bf16 per layer
        assert (np.abs(as_f64(out[2]) - ref) <= L * 2.0 ** -7 * np.maximum(1.0, np.abs(ref))).all(), kernel


@pytest.mark.parametrize("N,d", [(8, 256), (16, 640), (32, 512), (16, 2048), (32, 2048)])
def test_infinite_table_entries(N, d):
    """A numerator of exactly 1 (a router of zeros) has parts that are zero, and zero times infinity is not what one times infinity
    is: an infinite entry of a row stays infinite in its column, of its sign, and touches no other."""
    M, L, V = 11, 2, 20
    g = torch.Generator().manual_seed(6)
    luts = torch.empty(L, V, N, d).normal_(0, 0.05, generator=g).to(torch.bfloat16)
    hidden = torch.empty(M, d).normal_(0, 1, generator=g).to(torch.bfloat16).to(DEV)
    ids = torch.arange(M, dtype=torch.int32).to(DEV)
    want = torch.zeros(M, d)
    for t in range(0, M, 2):
        for col, sign in ((t, 1.0), (d - 1 - 7 * t, -1.0), (d // 2 + t, 1.0)):
            luts[L - 1, t, t % N, col] = want[t, col] = sign * float("inf")
    wrs = torch.zeros(L, d, N, dtype=torch.bfloat16, device=DEV)
    outs = [mole.decode_step_args(hidden, ids, luts.to(DEV), wrs, torch.empty_like(hidden), mode=mole.STEP_FUSED, kernel=k).cpu().float()
            for k in (mole.KERNEL_AUTO, mole.KERNEL_RING)]
    for out in outs:
        assert torch.equal(torch.isinf(out), torch.isinf(want)) and not torch.isnan(out).any()
        assert torch.equal(out[torch.isinf(want)], want[torch.isinf(want)])
    finite = ~torch.isinf(want)
    assert (outs[0] - outs[1])[finite].abs().max() <= 2.0 ** -5  # an ulp of a value of up to 8
