"""Gram matrix of binary32 gradients as 8-bit digits on the tensor cores: against binary64 products of the same values.

A value is rounded to fixed point of at most 2^-24 of the largest magnitude of the gradient, half a unit off; by Cauchy-Schwarz
    |G_ij - exact| <= 2^-25 sqrt(D) (max|x_i| |x_j| + max|x_j| |x_i|),
and the sums themselves are exact integers, put together in binary64."""
import pytest
import torch

import paper_2412_18052_b200 as gaf
from paper_2412_18052_b200 import workloads
from parity import check_any_seed, check_filter

pytestmark = pytest.mark.gpu


def _grads(K, D, kind, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shared = torch.randn(D, generator=gen, device="cuda")
    out = []
    for i in range(K):
        x = 0.5 * shared + torch.randn(D, generator=gen, device="cuda")
        if kind == "scales":
            x *= 10.0 ** (i % 7 - 3)
        elif kind == "outlier":                     # far beyond what the sample lets expect
            x[(i * 37) % D] *= 1e6
        elif kind == "segments":
            x *= torch.exp(2.5 * torch.randn((D + 999) // 1000, generator=gen, device="cuda")).repeat_interleave(1000)[:D]
        elif kind == "sparse":                      # most samples see nothing but zeros
            x *= torch.rand(D, generator=gen, device="cuda") < 0.001
        elif kind == "tiny":
            x *= 1e-30
        elif kind == "huge":
            x *= 1e17
        out.append(x.contiguous())
    return out


def _exact(grads):
    G = torch.zeros(len(grads), len(grads), dtype=torch.float64, device="cuda")
    for s in range(0, grads[0].numel(), 1 << 20):
        m = torch.stack([g[s:s + (1 << 20)].double() for g in grads])
        G += m @ m.T
    return G


def _gram(grads, ws):
    K = len(grads)
    return gaf.gaf_pairwise_cosdist(grads, ws, gram_out=torch.empty(K, K, dtype=torch.float64, device="cuda"))[1]


def _check(grads):
    K, D = len(grads), grads[0].numel()
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    G = _gram(grads, ws)
    assert gaf.gaf_read_status(ws) & ~gaf.GAF_STATUS_ZERO_NORM == 0
    assert torch.equal(G, _gram(grads, ws))         # integer sums do not depend on the order the tiles come in
    E = _exact(grads)
    norm, top = E.diagonal().sqrt(), torch.stack([g.abs().max() for g in grads]).double()
    bound = 2.0 ** -25 * D ** 0.5 * (torch.outer(top, norm) + torch.outer(norm, top)) + 1e-12 * torch.outer(norm, norm)
    assert bool(((G - E).abs() <= bound).all()), (K, D, ((G - E).abs() / bound).max().item())


# (up to 16 gradients of fewer than 2^20 elements, and up to 24 of fewer than 327680, go to another kernel)
@pytest.mark.parametrize("K", [9, 16, 17, 24, 25, 32, 33, 40, 41, 48, 49, 56, 57, 64])
def test_tiles_and_remainders(K):
    short = (1, 3, 5, 127, 128, 129, 10_007, 148 * 128 * 3 + 130) if K > 24 else ()
    for D in short + ((1 << 20, (1 << 20) + 3, 148 * 256 * 30 + 130) if K <= 16 else (327_680, 327_683, 148 * 128 * 23 + 130)):
        _check(_grads(K, D, "", K + D))


@pytest.mark.parametrize("K", [15, 23, 31, 39, 47, 55, 63])
def test_one_absent_gradient(K):
    """The warp with the absent gradient loads the other seven under predicates."""
    for D in ((1 << 20) + 129, 148 * 256 * 11 + 5) if K <= 16 else (327_680 + 127, 148 * 128 * 21 + 6):
        _check(_grads(K, D, "", K + D))


def _digits_length(K):
    """A ragged length of several tiles per CTA that goes to the digits."""
    return (1 << 20) + 261 if K <= 16 else 327_680 + 133 if K <= 24 else 50_005


@pytest.mark.parametrize("K", [10, 16, 20, 24, 29, 32, 40, 47, 56, 64])
@pytest.mark.parametrize("bands", [False, True])
def test_whole_numbers_are_exact(K, bands):
    """Whole numbers below 2^23, all four digits of them in use, are whole in fixed point, and so are smaller ones with bands beyond
    their bound (2^5 times 2^15): nothing is rounded but sums in binary64, the reference's among them (sqrt(D) x 2^-53 at the most likely, 1e-13).
    A digit lost or in the wrong place leaves 1e-9 and more."""
    D = _digits_length(K)
    gen = torch.Generator(device="cuda").manual_seed(K)
    top = 15 if bands else 23
    grads = [torch.randint(1 - (1 << top), 1 << top, (D,), generator=gen, device="cuda").float() for _ in range(K)]
    if bands:
        for i, x in enumerate(grads):
            for at in (D // 7 * (i % 5) + 11, D - 300 - i):
                x[at:at + 200] = torch.randint(1 - (1 << 23), 1 << 23, (200,), generator=gen, device="cuda").float()
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    G, E = _gram(grads, ws), _exact(grads)
    norm = E.diagonal().sqrt()
    assert float(((G - E).abs() / torch.outer(norm, norm)).max()) < 1e-12


@pytest.mark.parametrize("K", [9, 16, 24, 32, 40, 48, 56, 64])
def test_rounding_of_normal_values(K):
    """Each value is at most half a unit off, 2^-25 of the gradient's largest, at random: the products' errors add up to a normal variable
    of at most 2^-25 / sqrt(3) (max|x_i| |x_j| + max|x_j| |x_i|); eight times that."""
    grads = _grads(K, _digits_length(K), "", 100 + K)
    ws = gaf.new_workspace(K, grads[0].numel(), gaf.GAF_F32)
    G, E = _gram(grads, ws), _exact(grads)
    norm, top = E.diagonal().sqrt(), torch.stack([g.abs().max() for g in grads]).double()
    bound = 8 / 3 ** 0.5 * 2.0 ** -25 * (torch.outer(top, norm) + torch.outer(norm, top)) + 1e-12 * torch.outer(norm, norm)
    assert bool(((G - E).abs() <= bound).all()), ((G - E).abs() / bound).max().item()


def test_small_elements_beside_large_ones():
    """The stated bound holds where nearly all elements of a gradient are below its unit and all errors have one sign."""
    K, D = 40, 300_001
    grads = [torch.full((D,), 2.0 ** -26.2 * (1 + i / 40), device="cuda") for i in range(K)]
    for i, x in enumerate(grads):
        x[:: 997 + i] = 1.0
    grads[3] = torch.ones(D, device="cuda")
    grads[3][::2] = 0.9
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    G, E = _gram(grads, ws), _exact(grads)
    total, top = torch.stack([g.abs().double().sum() for g in grads]), torch.stack([g.abs().max() for g in grads]).double()
    bound = 2.0 ** -25 * (torch.outer(top, total) + torch.outer(total, top)) + 2.0 ** -49 * D * torch.outer(top, top)
    assert bool(((G - E).abs() <= bound).all()), ((G - E).abs() / bound).max().item()


@pytest.mark.parametrize("K", [12, 15, 17, 20, 24, 30, 40])
def test_filter_on_digits(K):
    """Algorithm 1 and its order-indifferent variant on a Gram matrix of digits, with one scale and with tensors of different scales."""
    D = _digits_length(K)
    sigma = torch.exp(2.0 * torch.randn(40, generator=torch.Generator().manual_seed(K))).repeat_interleave(-(-D // 40))[:D].cuda() * 1e-3
    for scale in (1e-3, sigma):
        rho = ([0.8, 0.7, -0.6, 0.5, 0.0, 0.6, -0.2, 0.4] * 5)[:K]
        grads = workloads.mixture(K, D, "f32", rho, K, device="cuda", sigma=scale).grads
        ws = gaf.new_workspace(K, D, gaf.GAF_F32)
        for tau in (0.9, 2.0):
            check_filter(grads, tau, ws)
            assert gaf.gaf_last_schedule() == gaf.GAF_SCHED_GRAM
        check_any_seed(grads, 0.9, ws)


@pytest.mark.parametrize("kind", ["scales", "outlier", "segments", "sparse", "tiny", "huge"])
@pytest.mark.parametrize("K, D", [(12, 1_100_001), (40, 300_001)])
def test_ranges_of_values(K, D, kind):
    _check(_grads(K, D, kind, 3))


def test_more_products_than_one_integer_sum_holds():
    _check(_grads(9, 2 * 148 * 1023 * 128 + 77, "", 4))
    _check(_grads(1, 148 * 1023 * 128 + 5, "outlier", 4))


@pytest.mark.parametrize("K, D", [(9, 1_100_003), (40, 70_003)])
def test_infinities_and_nans(K, D):
    grads = _grads(K, D, "", 5)
    grads[1][77], grads[3][77], grads[4][4001] = float("inf"), -float("inf"), float("nan")
    grads[5][D - 1], grads[6][10], grads[6][11] = float("inf"), float("inf"), -float("inf")
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    G = _gram(grads, ws)
    assert gaf.gaf_read_status(ws) & gaf.GAF_STATUS_NONFINITE
    E = torch.stack([torch.stack([(x.double() * y.double()).sum() for y in grads]) for x in grads])
    finite = torch.isfinite(E)
    assert torch.equal(torch.isfinite(G), finite) and torch.equal(torch.isnan(G), torch.isnan(E))
    assert torch.equal(G[torch.isinf(E)], E[torch.isinf(E)])
    assert bool(((G - E)[finite].abs() <= 1e-7 * D).all())


@pytest.mark.parametrize("K, D", [(13, 1_100_001), (24, 500_003), (40, 300_001), (64, 150_001)])
@pytest.mark.parametrize("kind", ["points", "bands", "half", "zeros first", "all"])
def test_values_beyond_the_bound(K, D, kind):
    """Tiles with values far beyond what was sampled are left out and come again under other scales: few of them, many, at the
    end, in single gradients, in every tile that was not sampled."""
    grads = _grads(K, D, "", 7)
    pick = torch.Generator(device="cuda").manual_seed(K)
    for i, x in enumerate(grads):
        if kind == "points" and i % 3 == 1:
            x[torch.randint(D, (20,), generator=pick, device="cuda")] *= 1e5
            x[-1] = 3e6
        elif kind == "bands" and i % 2:
            x[D // 3:D // 3 + 7001] *= 1e3
            x[-3001:] *= 1e4
        elif kind == "half":                        # every other 512 elements
            x[: D // 1024 * 1024].view(-1, 2, 512)[:, 1] *= 200.0
        elif kind == "zeros first" and i != 2:
            x[: D * 9 // 10] = 0.0
        elif kind == "all" and i == 5:
            x[torch.rand(D, generator=pick, device="cuda") < 0.99] = 0.0
            x *= torch.exp(4.0 * torch.randn(D, generator=pick, device="cuda"))
    _check(grads)


@pytest.mark.parametrize("K", [9, 17, 33])
def test_second_period(K):
    """More tiles per CTA than one integer sum holds: an outlier, and an infinity, in the second period only."""
    D = 148 * 1023 * 128 + 700_001
    grads = _grads(K, D, "", 11)
    _check(grads)
    grads[3][148 * 1023 * 128 + 300_000] = 1e6
    grads[K - 1][-9] = -1e6
    _check(grads)
    grads[1][D - 4000] = float("inf")
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    G, E = _gram(grads, ws), _exact(grads)
    assert torch.equal(torch.isfinite(G), torch.isfinite(E)) and torch.equal(G[1].sign(), E[1].sign())
    assert bool(((G - E)[torch.isfinite(E)].abs() <= 1e-9 * E[3, 3]).all())


@pytest.mark.parametrize("K, D", [(9, 1_100_003), (24, 400_001), (64, 70_003)])
def test_gradients_of_nans_and_infinities(K, D):
    """A gradient that is NaN throughout, one with infinities of one sign, of both signs, against values of one sign, against zeros;
    with values beyond the bound beside them."""
    grads = _grads(K, D, "", 12)
    grads[0][:] = float("nan")
    grads[2][grads[2] > 2.5] = float("inf")
    grads[4][grads[4].abs() > 2.5] *= float("inf")
    grads[5].abs_()
    grads[6].abs_()
    grads[6][D // 2] = float("inf")
    grads[7].abs_()
    grads[7][(D // 2) // 4 * 4 + 8] = 0.0
    grads[8].abs_()
    grads[8][(D // 2) // 4 * 4 + 8], grads[8][99] = -float("inf"), 1e7
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    G = _gram(grads, ws)
    E = torch.stack([torch.stack([(x.double() * y.double()).sum() for y in grads]) for x in grads])
    finite = torch.isfinite(E)
    assert torch.equal(torch.isfinite(G), finite) and torch.equal(torch.isnan(G), torch.isnan(E))
    assert torch.equal(G[torch.isinf(E)], E[torch.isinf(E)])
    assert torch.isinf(E[5, 6]) and torch.isnan(E[7, 8]) and E[5, 8] == -float("inf")
    assert bool(((G - E)[finite].abs() <= 1e-7 * D).all())
    again = _gram(grads, ws)
    assert torch.equal(again[finite], G[finite])


def _time(grads, ws):
    best = float("inf")
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            gaf.gaf_pairwise_cosdist(grads, ws)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("kind", ["point", "band", "nan"])
def test_time_with_values_beyond_the_bound(kind):
    """What a call costs beyond one on values of one scale is what the tiles beyond their bounds cost, not its share again: measured
    1.0 to 1.3 times; a share done again cost 4 times, a gradient of NaNs 28 times."""
    K, D = 16, 11_000_003
    grads = _grads(K, D, "", 13)
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    plain = _time(grads, ws)
    if kind == "point":
        grads[1][D // 3 + 12345] = 1e6
    elif kind == "band":
        grads[1][D // 3:D // 3 + D // 20] *= 1e3
    else:
        grads[1][:] = float("nan")
    assert _time(grads, ws) < 2.0 * plain


def test_bounded_wait_runs_out():
    grads = _grads(24, 400_000, "", 6)
    ws = gaf.new_workspace(24, 400_000, gaf.GAF_F32)
    want = _gram(grads, ws)
    try:
        gaf.gaf_test_set_wait_fault(2000, 1)
        _gram(grads, ws)
        torch.cuda.synchronize()
        assert gaf.gaf_read_status(ws) & gaf.GAF_STATUS_TIMEOUT
    finally:
        gaf.gaf_test_set_wait_fault(0, 0)
    assert torch.equal(_gram(grads, ws), want) and gaf.gaf_read_status(ws) == 0
