"""The Gram-first forms of the filter from every state a workspace can be in, and decisions and sums that must not depend on the
form or on what ran before: GPU tests, results against the stepwise schedule bit for bit."""
import numpy as np
import pytest
import torch

import paper_2412_18052_b200 as gaf
from paper_2412_18052_b200 import workloads

pytestmark = pytest.mark.gpu

DTYPES = ["f32", "bf16"]
CODE = {"f32": gaf.GAF_F32, "bf16": gaf.GAF_BF16}


def _mix(K, D, dtype, seed, rho, stacked=False):
    return workloads.mixture(K, D, dtype, rho, seed, device="cuda", stacked=stacked).grads


def _predicted_length(K, dtype):
    """A length from which the one-pass kernel predicts the accept pattern: four times what the SMs' shared memory holds."""
    return 4 * 200_000 // (K * (4 if dtype == "f32" else 2)) * 148


def _stepwise(grads, tau, ws):
    return [t.clone() for t in gaf.gaf_filter_accumulate(grads, tau, ws, schedule=gaf.GAF_SCHED_STEPWISE)]


def _same(got, want):
    assert torch.equal(got[1], want[1]) and torch.equal(got[3], want[3])
    assert torch.equal(got[0], want[0])


@pytest.mark.parametrize("K,dtype", [(3, "f32"), (4, "f32"), (8, "f32"), (8, "bf16")])
def test_two_launches_on_a_workspace_initialised_for_every_call(K, dtype):
    """One buffer, initialised anew for every call, as a workspace per step at one address is; the accept patterns alternate, so
    that what the memory still holds from the call before is always the wrong one."""
    D = _predicted_length(K, dtype)
    both = [_mix(K, D, dtype, 3, [0.8] * K), _mix(K, D, dtype, 4, ([0.8] + [0.7, -0.6] * K)[:K])]
    other = gaf.new_workspace(K, D, CODE[dtype])
    want = [_stepwise(g, 0.9, other) for g in both]
    assert not torch.equal(want[0][1], want[1][1])
    ws = gaf.new_workspace(K, D, CODE[dtype])
    for call in range(12):
        gaf.gaf_workspace_init(ws)
        _same(gaf.gaf_filter_accumulate(both[call % 2], 0.9, ws, schedule=gaf.GAF_SCHED_GRAM), want[call % 2])


@pytest.mark.parametrize("before", ["cosdist", "stepwise", "stream", "bucketed", "pairwise16"])
def test_two_launches_first_after_another_operation(before):
    """Whole-numbered gradients: the partial sums that other operations leave in the workspace have empty low words.  The first
    two-launch call behind them."""
    K, D = 4, _predicted_length(4, "f32")
    gen = torch.Generator(device="cuda").manual_seed(9)
    grads = [torch.randint(0, 2, (D,), generator=gen, device="cuda").float() + 1.0 for _ in range(K)]
    grads[2] = -grads[2]
    want = _stepwise(grads, 0.9, gaf.new_workspace(K, D, gaf.GAF_F32))
    assert want[1].tolist() == [1, 1, 0, 1]
    for _ in range(3):
        ws = gaf.new_workspace(16, D, gaf.GAF_F32)
        if before == "cosdist":
            gaf.gaf_cosdist(grads[0], grads[2], ws)
        elif before == "stepwise":
            _stepwise(grads, 0.9, ws)
        elif before == "stream":
            acc = torch.empty(D, device="cuda")
            gaf.gaf_stream_begin(grads[0], acc, ws)
            gaf.gaf_stream_push(grads[1], 1, 0.9, acc, ws)
            gaf.gaf_stream_end(2, acc, ws)
        elif before == "bucketed":
            gaf.gaf_filter_accumulate_bucketed(grads, 0.9, [0, D // 16 * 8, D], ws)
        else:
            gaf.gaf_pairwise_cosdist([g[:100_000].contiguous() for g in grads * 4], ws)
        _same(gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM), want)


@pytest.mark.parametrize("fill", [0.0, 1.0, -3.0, 1e-3])
def test_two_launches_on_memory_that_held_other_data(fill):
    """A workspace whose memory was a binary64 tensor before: zeros, values with an empty low word, any others."""
    K, D = 4, _predicted_length(4, "f32")
    grads = _mix(K, D, "f32", 5, [0.8, 0.7, -0.6, 0.5])
    want = _stepwise(grads, 0.9, gaf.new_workspace(K, D, gaf.GAF_F32))
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    for _ in range(3):
        ws.view(torch.float64).fill_(fill)
        gaf.gaf_workspace_init(ws)
        for _ in range(2):
            _same(gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM), want)


def _lines(ws, table):
    """The lines of 16 words through which the CTAs of the one-pass kernel are told the predicted (0) or decided (1) pattern."""
    return ws[4096 + table * 160 * 128:4096 + (table + 1) * 160 * 128].view(torch.int64).view(160, 16)


@pytest.mark.parametrize("K,dtype", [(4, "f32"), (8, "f32"), (8, "bf16")])
def test_first_call_on_a_workspace_predicts(K, dtype):
    """The first two-launch call on memory that was zero, or held another workspace, writes the result in its first launch
    (word 3 of the workspace says so) like every later one.  A prediction is given up after some tens of microseconds, so one call
    of several counts."""
    D = _predicted_length(K, dtype)
    grads = _mix(K, D, dtype, 5, ([0.8, 0.7, -0.6, 0.5] * 2)[:K])
    ws = gaf.new_workspace(K, D, CODE[dtype])
    for zeroed in (True, False):
        done = 0
        for _ in range(5):
            if zeroed:
                ws.zero_()
            gaf.gaf_workspace_init(ws)
            gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM)
            done += int(ws[:16].view(torch.int32)[3])
        assert done >= 1, zeroed


def test_words_that_only_look_like_a_pattern():
    """Lines that hold a whole valid word of the call's tag with the wrong pattern (two launches: only the comparison of what the
    CTAs wrote can tell), and words whose low half alone is the tag of the call (either form)."""
    K, D = 4, _predicted_length(4, "f32")
    grads = _mix(K, D, "f32", 5, [0.8, 0.7, -0.6, 0.5])
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    want = _stepwise(grads, 0.9, ws)
    wrong = (0x80000004 - (1 << 32)) << 32                      # the third gradient alone
    for whole in (True, False):
        gaf.gaf_workspace_init(ws)
        _lines(ws, 0)[:, 0] = wrong | 1
        _lines(ws, 0)[:, 1] = wrong | 0xFFFFFFFE if whole else 0
        _same(gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM), want)
    for _ in range(3):
        _same(gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM_FUSED), want)
        tag = (int(_lines(ws, 1)[1, 0]) + 1) & 0xFFFFFFFF        # the next call's
        _lines(ws, 1)[:, 0] = wrong | tag
        _lines(ws, 1)[:, 1] = 0


@pytest.mark.parametrize("K,dtype", [(3, "f32"), (5, "f32"), (8, "f32"), (6, "bf16"), (8, "bf16"), (12, "f32"), (12, "bf16")])
def test_everything_is_accepted_from_tau_two_on(K, dtype):
    """tau >= 2 accepts everything, also a gradient that points exactly against a running sum most of which has cancelled: the
    sums' rounding puts that cosine below -1 in about every other case, and Eq. 4 takes it as -1."""
    ws = gaf.new_workspace(16, 1 << 20, gaf.GAF_F32)
    torch.manual_seed(17)
    tdtype = torch.float32 if dtype == "f32" else torch.bfloat16
    for D in (4_001, 60_007):
        for trial in range(24):
            a = torch.randn(D, device="cuda").to(tdtype)
            b = (-a.float() + 4e-3 * torch.randn(D, device="cuda")).to(tdtype)
            c = ((a.double() + b.double()) * -100.0).to(tdtype)
            grads = [a, b, c] + [torch.randn(D, device="cuda").to(tdtype) for _ in range(K - 3)]
            for tau in (2.0, 2.5):
                for schedule in (gaf.GAF_SCHED_STEPWISE, gaf.GAF_SCHED_GRAM, gaf.GAF_SCHED_AUTO):
                    _, mask, _, count = gaf.gaf_filter_accumulate(grads, tau, ws, schedule=schedule)
                    assert mask.tolist() == [1] * K and int(count) == K, (D, trial, tau, schedule)
                if K <= 8:
                    got = gaf.gaf_filter_accumulate_bucketed(grads, tau, [0, D // 16 * 8, D], ws)
                    assert bool((got[1] == 1).all()), (D, trial, tau)
                got = gaf.gaf_filter_accumulate_any_seed(grads, tau, ws)
                assert bool((got[1] == 1).all()) and int(got[4]) == 0, (D, trial, tau)


def _nearly_equal(K, D, dtype, seed):
    """Gradients so close to one another that their distances show the last bits of the sums."""
    torch.manual_seed(seed)
    x = torch.randn(D, device="cuda")
    tdtype = torch.float32 if dtype == "f32" else torch.bfloat16
    return [(x + (1e-5 if dtype == "f32" else 4e-3) * torch.randn(D, device="cuda")).to(tdtype) for _ in range(K)]


@pytest.mark.parametrize("dtype", DTYPES)
def test_two_gradients_same_bits_after_every_history(dtype):
    """What a call of two gradients gives does not depend on how the calls before it on the workspace ended."""
    for D in (_predicted_length(2, dtype) // 4 + 12_345, _predicted_length(2, dtype) + 5):
        ws = gaf.new_workspace(2, D, CODE[dtype])
        for seed in range(4):
            grads = _nearly_equal(2, D, dtype, seed)
            yes, no = grads, [grads[0], -grads[1]]
            seen = []
            for history in ((), (yes, yes), (no, no), (yes, no), (no, yes)):
                gaf.gaf_workspace_init(ws)
                for h in history:
                    gaf.gaf_filter_accumulate(h, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM_FUSED)
                seen.append([t.clone() for t in gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM_FUSED)])
            seen.append([t.clone() for t in gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM)])
            for other in seen[1:]:
                for a, b in zip(seen[0], other):
                    assert torch.equal(a, b), (D, seed)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("K", [3, 4, 5, 6, 7, 8])
def test_one_and_two_launches_same_bits(K, dtype):
    """Both Gram-first forms take the same sums in the same order, short vectors (no prediction) and longer ones."""
    for D in (_predicted_length(K, dtype) // 8 + 12_345, _predicted_length(K, dtype) + 5):
        ws = gaf.new_workspace(K, D, CODE[dtype])
        for seed in range(3):
            grads = _nearly_equal(K, D, dtype, seed)
            one = [t.clone() for t in gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM_FUSED)]
            two = gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM)
            for a, b in zip(one, two):
                assert torch.equal(a, b), (D, seed)


@pytest.mark.parametrize("dtype", DTYPES)
def test_gradients_made_as_they_are_asked_for(dtype):
    """A sequence that makes its tensors on request, and the rows of one tensor: the call holds them until it has been launched,
    so that none of the outputs it allocates lies in their memory."""
    K, D = 4, 300_000
    kept = _mix(K, D, "f32", 3, [0.8, 0.7, -0.6, 0.5])
    tdtype = torch.float32 if dtype == "f32" else torch.bfloat16

    class Made:
        def __len__(self):
            return K

        def __getitem__(self, i):
            if i >= K:
                raise IndexError
            return kept[i].clone().to(tdtype)

    grads = [Made()[i] for i in range(K)]
    ws = gaf.new_workspace(K, D, CODE[dtype])
    want = [t.clone() for t in gaf.gaf_filter_accumulate(grads, 0.9, ws)]
    want_pairs = gaf.gaf_pairwise_cosdist(grads, ws)[0].clone()
    for _ in range(3):
        for given in (Made(), torch.stack(grads)):
            for a, b in zip(gaf.gaf_filter_accumulate(given, 0.9, ws), want):
                assert torch.equal(a, b)
            assert torch.equal(gaf.gaf_pairwise_cosdist(given, ws)[0], want_pairs)


def test_orders_that_are_no_permutation_are_refused():
    K, D = 3, 1000
    grads = _mix(K, D, "f32", 3, [0.8, 0.7, -0.6])
    ws = gaf.new_workspace(K, D, gaf.GAF_F32)
    want = [t.clone() for t in gaf.gaf_filter_accumulate(grads, 0.9, ws, order=[2, 0, 1])]
    for bad in ([], [0], [0, 1], [0, 1, 3], [0, 1, -1], [0, 1, 2 + 2 ** 32], [2 ** 31, 1, 2], [0, 1, 1]):
        for call in (lambda: gaf.gaf_filter_accumulate(grads, 0.9, ws, order=bad),
                     lambda: gaf.gaf_filter_accumulate_bucketed(grads, 0.9, [0, D], ws, order=bad)):
            with pytest.raises(gaf.GafError) as e:
                call()
            assert e.value.code == 1, bad
    for good in ([2, 0, 1], (2, 0, 1), np.array([2, 0, 1]), torch.tensor([2, 0, 1]), [2, 0, 1, 7]):
        for a, b in zip(gaf.gaf_filter_accumulate(grads, 0.9, ws, order=good), want):
            assert torch.equal(a, b)


def test_thresholds_that_float_takes():
    grads = _mix(3, 1000, "f32", 3, [0.8, 0.7, -0.6])
    ws = gaf.new_workspace(3, 1000, gaf.GAF_F32)
    want = [t.clone() for t in gaf.gaf_filter_accumulate(grads, 0.5, ws)]
    for tau in (np.float32(0.5), torch.tensor(0.5), "0.5"):
        for a, b in zip(gaf.gaf_filter_accumulate(grads, tau, ws), want):
            assert torch.equal(a, b)
    for bad in ("half", None, [0.5]):
        with pytest.raises((TypeError, ValueError)):
            gaf.gaf_filter_accumulate(grads, bad, ws)


class _Fault:
    """Limit and withheld signals of the bounded waits, for the calls inside."""

    def __init__(self, limit, withhold):
        self.args = (limit, withhold)

    def __enter__(self):
        gaf.gaf_test_set_wait_fault(*self.args)

    def __exit__(self, *_):
        gaf.gaf_test_set_wait_fault(0, 0)


@pytest.mark.parametrize("tiles", [4, 8])
@pytest.mark.parametrize("K,dtype", [(2, "f32"), (4, "f32"), (5, "bf16"), (8, "f32"), (8, "bf16")])
def test_tiles_that_never_land(K, dtype, tiles):
    """No copy at all, and none from the second lap of the ring on: every warp gives up, touches no tile that it has not seen land,
    and the call ends with GAF_STATUS_TIMEOUT.  Nothing outside the outputs is written, and the next call is right."""
    for D in (_predicted_length(K, dtype) + 5, _predicted_length(K, dtype) // 2 + 64):
        grads = _mix(K, D, dtype, 5, ([0.8, 0.7, -0.6, 0.5] * 2)[:K])
        ws = gaf.new_workspace(K, D, CODE[dtype])
        want = _stepwise(grads, 0.9, ws)
        guarded = torch.full((D + 8192,), 777.0, device="cuda")
        for schedule in (gaf.GAF_SCHED_GRAM, gaf.GAF_SCHED_GRAM_FUSED):
            with _Fault(200, tiles):
                gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=schedule, macro_out=guarded[4096:4096 + D])
                status = gaf.gaf_read_status(ws)
            assert status & gaf.GAF_STATUS_TIMEOUT
            assert bool((guarded[:4096] == 777.0).all()) and bool((guarded[4096 + D:] == 777.0).all())
            _same(gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=schedule), want)
            assert gaf.gaf_read_status(ws) == 0


@pytest.mark.parametrize("K,dtype", [(3, "f32"), (6, "bf16"), (8, "f32"), (8, "bf16")])
def test_prediction_that_does_not_come(K, dtype):
    """The wait for the predicted pattern runs out and nothing else does: a valid call, written after the decision."""
    for D in (_predicted_length(K, dtype) + 5, _predicted_length(K, dtype) // 2 + 64):
        ws = gaf.new_workspace(K, D, CODE[dtype])
        for rho in ([0.8] * K, ([0.8, 0.7, -0.6, 0.5] * 2)[:K]):
            grads = _mix(K, D, dtype, 5, rho)
            want = _stepwise(grads, 0.9, ws)
            for schedule in (gaf.GAF_SCHED_GRAM, gaf.GAF_SCHED_GRAM_FUSED):
                with _Fault(0, 2):
                    got = gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=schedule)
                    assert gaf.gaf_read_status(ws) == 0
                _same(got, want)


@pytest.mark.parametrize("dtype", DTYPES)
def test_two_gradients_prediction_that_does_not_come(dtype):
    """The shortest vectors that two gradients predict on (one tile more than the ring holds), where a sample's tile is among those
    that stay in the ring; the pattern of the calls before is no help, since they ended differently."""
    tile = 1792 if dtype == "f32" else 3584
    ring = 8 * tile * torch.cuda.get_device_properties(0).multi_processor_count
    for D in (ring + 1000, ring + ring // 8, ring + ring // 8 + 1000):
        ws = gaf.new_workspace(2, D, CODE[dtype])
        yes = _mix(2, D, dtype, 5, [0.8, 0.7])
        no = [yes[0], -yes[1]]
        for grads in (yes, no):
            want = _stepwise(grads, 0.9, ws)
            for _ in range(3):
                for h in (yes, no):
                    gaf.gaf_filter_accumulate(h, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM_FUSED)
                with _Fault(0, 2):
                    got = gaf.gaf_filter_accumulate(grads, 0.9, ws, schedule=gaf.GAF_SCHED_GRAM_FUSED)
                    assert gaf.gaf_read_status(ws) == 0
                _same(got, want)
