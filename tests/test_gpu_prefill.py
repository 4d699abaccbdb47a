"""The prefill kernel (single layers of many tokens) against the fp64 oracle at the sizes where its groups, warps per
token and column passes have edges: expert counts, widths of one to sixteen slices of 128 columns, ragged token counts
one past the dispatch line, one past a wave and below it, with and without norm, residual and bad ids."""
import numpy as np
import pytest
import torch

from gpu_util import as_f64, bits, check_gates, check_out, oracle_layer, rand_case
from paper_2503_15798_b200 import binding as mole
from test_gpu_norm import check_out_after_flips, oracle_norm_layer

pytestmark = pytest.mark.gpu
DEV = "cuda"
SMS = 148

# N, d, tokens per SM of the dispatch line, further tokens
CASES = [(8, 128, 8, 1), (8, 1152, 6, 5), (8, 2048, 6, 700), (16, 256, 8, 2), (16, 384, 8, 9), (16, 640, 6, 1), (16, 768, 6, 3), (16, 1024, 6, 900),
         (16, 1280, 2, 1), (16, 2048, 2, 300), (32, 512, 6, 1), (32, 1024, 2, 3), (32, 1920, 2, 2), (32, 2048, 2, 1), (32, 2048, 2, 400)]


@pytest.mark.parametrize("N,d,line,more", CASES)
@pytest.mark.parametrize("norm", [False, True])
def test_prefill_layer_against_the_oracle(N, d, line, more, norm):
    M, V = line * SMS + more, 70
    hidden, ids, lut, wr = rand_case(M, N, d, V, seed=N * d + M)
    residual = torch.empty(M, d).normal_(0, 1, generator=torch.Generator().manual_seed(1)).to(torch.bfloat16)
    ids[0], ids[M - 1] = -1, V  # the routed term of neither
    assert mole.variant(M, N, d, norm=norm)[0].startswith(f"tile<{N},{int(norm)},")
    assert mole.variant(line * SMS, N, d, norm=norm)[0].startswith(("step<", "slice_layer<"))  # up to the dispatch line
    gates = torch.zeros(M, N, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    gamma = (1.0 + 0.2 * torch.empty(d).normal_(0, 1, generator=torch.Generator().manual_seed(2))).to(torch.bfloat16) if norm else None
    out = mole.layer_forward(hidden.to(DEV), ids.to(DEV).long(), lut.to(DEV), wr.to(DEV), gates_out=gates, status=status, residual=residual.to(DEV),
                             norm_weight=None if gamma is None else gamma.to(DEV), norm_eps=1e-5)
    torch.cuda.synchronize()
    assert int(status.item()) == mole.STATUS_BAD_ID
    assert np.array_equal(bits(out)[[0, M - 1]], bits(residual)[[0, M - 1]])
    if norm:
        ref, gref, _ = oracle_norm_layer(hidden, ids, lut, wr, gamma, 1e-5, residual=residual)
        check_out_after_flips(out, ref, gates, gref, lut)
    else:
        ref, gref, _ = oracle_layer(hidden, ids, lut, wr, residual=residual)
        check_out(out, ref)
        check_gates(gates, gref)


def test_large_logits_and_in_place_output():
    """Router weights that push logits beyond the range where the maximum has to be subtracted; out is hidden itself."""
    M, N, d, V = 6 * SMS + 40, 16, 768, 50
    hidden, ids, lut, wr = rand_case(M, N, d, V, seed=5, wr_std=3.0)
    ref, gref, _ = oracle_layer(hidden, ids, lut, wr)
    assert gref.max() > 0.999
    h = hidden.to(DEV)
    out = mole.layer_forward(h, ids.to(DEV), lut.to(DEV), wr.to(DEV), out=h)
    torch.cuda.synchronize()
    # logits of ~80 carry 80 * 2^-22 of fp32 rounding, and so do the gates relative to themselves: 2e-5 of the routed term
    err = np.abs(as_f64(out) - ref)
    assert (err <= 2.0 ** -8 * np.abs(ref) + 2e-5 + 4e-5 * float(lut.abs().max()) * N).all(), float(err.max())


@pytest.mark.parametrize("N,d,M", [(16, 768, 6 * SMS + 3), (32, 2048, 2 * SMS + 1)])
def test_norm_of_a_state_whose_sum_of_squares_overflows(N, d, M):
    """mean(x^2) is infinite: the normalised state is zero, the gates are 1 / N, the result is that of the ring kernel."""
    V = 40
    hidden, ids, lut, wr = rand_case(M, N, d, V, seed=9)
    hidden[3, 5], hidden[M - 1, d - 1] = 2e19, -3e38
    gamma = torch.ones(d, dtype=torch.bfloat16, device=DEV)
    h, i, t, w = hidden.to(DEV), ids.to(DEV), lut.to(DEV), wr.to(DEV)
    got, want = [], []
    for r, kernel in ((got, mole.KERNEL_AUTO), (want, mole.KERNEL_RING)):
        gates = torch.zeros(M, N, dtype=torch.float32, device=DEV)
        r += [mole.layer_forward(h, i, t, w, gates_out=gates, norm_weight=gamma, norm_eps=1e-6, kernel=kernel), gates]
    for row in (3, M - 1):
        assert (got[1][row] == 1.0 / N).all() and (want[1][row] == 1.0 / N).all()
        ref = as_f64(hidden[row]) + as_f64(lut[int(ids[row])]).mean(axis=0)
        for out in (got[0], want[0]):  # one rounding of the sum
            assert (np.abs(as_f64(out[row]) - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-6).all()
