"""GPU: the plan kernels where their dispatch can go wrong -- runs that end on, just before and just
after a tile border, tiles of mixed depth, unsorted tiles, more undecided pairs than are kept in shared
memory, more query tiles than threads -- against the oracle."""
import numpy as np
import pytest
import torch

from oracle import peagle_oracle as orc
from paper_2602_01469_b200 import binding, inputs
from tests.gpu_common import DeviceCase, check_forward
from tests.test_gpu_backward import check_grads, oracle_all, run_partitioned
from tests.test_gpu_mask_and_tiles import device_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = binding.Context(0)
    yield c
    c.close()


def check_classes(ctx, anchor, depth, K, q, k):
    prob = device_problem([0, anchor.shape[0]], anchor, depth, K)
    got = binding.peagle_classify_tiles(ctx, prob, binding.Partition(0, q, k))
    want, _, _ = orc.classify_tiles(anchor, depth, q[0], q[1], k, 128, 128)
    assert np.array_equal(got, want)
    assert binding.peagle_poll_status(ctx) == 0


@pytest.mark.parametrize("order", ["depth_major", "anchor_major"])
@pytest.mark.parametrize("n,K", [(1, 8), (63, 6), (127, 5), (128, 5), (129, 5), (255, 3), (385, 4), (40, 40)])
def test_classes_at_tile_borders(ctx, n, K, order):
    anchor, depth = inputs.full_grid(n, K)
    perm = inputs.arrange_by_segment(anchor, depth, np.zeros(n * K, np.int32), order)
    anchor, depth = anchor[perm], depth[perm]
    check_classes(ctx, anchor, depth, K, (0, n * K), None)
    if n * K > 40:      # ranges that start inside a run, a one-token range among them
        check_classes(ctx, anchor, depth, K, (7, n * K - 3), [(1, 2), (5, n * K // 2 + 1), (n * K - 9, n * K)])


def test_classes_of_one_anchor_and_of_unsorted_tiles(ctx):
    # 250 depths of one anchor: chain tiles that are FULL without a depth-0 key in them
    check_classes(ctx, np.zeros(250, np.int32), np.arange(250, dtype=np.int32), 250, (0, 250), None)
    # 282 unsorted key tiles: all pairs of a query tile are undecided
    anchor, depth = inputs.full_grid(9000, 4)
    perm = np.random.default_rng(3).permutation(36000)
    check_classes(ctx, anchor[perm], depth[perm], 4, (100, 430), None)


@pytest.mark.parametrize("w", [
    # chain keys of a query tile straddle two key tiles by one token, by half, by all but one
    inputs.Workload("straddle_1", (129,), 6, 4, 2, 64, seed=41),
    inputs.Workload("straddle_64", (192,), 6, 4, 2, 128, seed=42),
    inputs.Workload("straddle_127", (255,), 6, 4, 2, 64, seed=43),
    # thinned chains: neighbouring windows that may and may not be joined
    inputs.Workload("thinned", (391,), 8, 4, 2, 64, seed=44, cod_r=0.8),
], ids=lambda w: w.name)
def test_joined_windows(ctx, w):
    case = DeviceCase(w)
    run_partitioned(ctx, case)
    O, LSE, dQ, dK, dV = oracle_all(case)
    check_forward(case.O.float().cpu().numpy(), case.LSE.t().cpu().numpy(), O, LSE)
    check_grads(case, dQ, dK, dV)


@pytest.mark.parametrize("n,K", [(150, 48), (128, 40), (70, 120)])
def test_more_chain_tiles_than_places_repeat_bit_for_bit(ctx, n, K):
    """From 33 depths on a query tile has more one-key-per-row tiles than the plan keeps: the same ones are
    chosen in every run, so that O and LSE, which are summed in a fixed order, repeat."""
    case = DeviceCase(inputs.Workload("deep", (n,), K, 4, 2, 64, seed=54))
    part = case.bparts[0]
    first = None
    for _ in range(10):
        binding.peagle_attn_fwd(ctx, case.prob, part, case.dQ_, case.dK_, case.dV_, case.O, case.LSE)
        assert binding.peagle_poll_status(ctx) == 0
        if first is None:
            first = (case.O.clone(), case.LSE.clone())
        assert torch.equal(case.O, first[0]) and torch.equal(case.LSE, first[1])
    O, LSE = case.oracle_fwd(case.parts[0])
    check_forward(case.O.float().cpu().numpy(), case.LSE.t().cpu().numpy(), O, LSE)


def test_plan_scratch_per_tile_pair():
    """What grows with the square of the length: class (1 byte), key list (8) and backward items (8) per pair
    of tiles.  A context keeps an eighth more than it needs, and the allocator rounds up to 2 MB."""
    n = 1 << 17
    Q = torch.randn(n, 1, 64, device="cuda").bfloat16()
    K, V, O, LSE = torch.randn_like(Q), torch.randn_like(Q), torch.empty_like(Q), torch.empty(1, n, device="cuda")
    anchor = torch.arange(n, dtype=torch.int32, device="cuda")
    depth = torch.zeros_like(anchor)
    own = binding.Context(0)

    def forward(m):
        prob = binding.Problem(np.array([0, m], np.int32), anchor, depth, 1, 1, 1, 64, 0.125)
        binding.peagle_attn_fwd(own, prob, binding.Partition(0, (0, m), None), Q, K, V, O, LSE)
        assert binding.peagle_poll_status(own) == 0
        return torch.cuda.mem_get_info()[0]

    used = forward(128) - forward(n)
    own.close()
    pairs = (n // 128) ** 2
    linear = n * 4 + n // 128 * (2 * 32 + 2 * 32 + 16 * 128 + 16 * 4 + 64)   # metadata, summaries, SINGLE entries
    assert used <= 1.125 * (17.5 * pairs + linear) + (4 << 20)


def test_more_query_tiles_than_threads(ctx):
    case = DeviceCase(inputs.Workload("long", (8300,), 8, 2, 1, 64, seed=45))
    run_partitioned(ctx, case)
    part = case.parts[0]
    rows = np.sort(np.random.default_rng(1).choice(case.T, 64, replace=False))
    O, LSE = case.oracle_fwd(part, rows=rows)
    idx = torch.as_tensor(rows, device="cuda")
    check_forward(case.O[idx].float().cpu().numpy(), case.LSE[:, idx].t().cpu().numpy(), O, LSE)
    dQ, _, _ = case.oracle_bwd(part, rows=rows)
    got = case.dQ[idx].float().cpu().numpy()
    assert np.linalg.norm(got - dQ) <= 1e-2 * np.linalg.norm(dQ)


@pytest.mark.parametrize("w", [
    inputs.Workload("sums_small", (200,), 3, 4, 2, 64, seed=46),        # cleared beside the plan
    inputs.Workload("sums_above_32mb", (2050,), 8, 2, 2, 128, seed=47),  # by a fill of their own
], ids=lambda w: w.name)
def test_sums_of_an_earlier_call_are_cleared(ctx, w):
    case = DeviceCase(w)
    run_partitioned(ctx, case)
    first = [t.float().cpu().numpy() for t in (case.dQ, case.dK, case.dV)]
    # a partition without rows in front: the next one's plan has to clear them
    empty = binding.Partition(0, (5, 5), case.parts[0]["k"])
    case.bparts = [empty] + case.bparts
    run_partitioned(ctx, case)
    for t, want in zip((case.dQ, case.dK, case.dV), first):
        # two fp32 sums of the same terms in another order, each rounded once to bf16
        assert np.linalg.norm(t.float().cpu().numpy() - want) <= 2.0**-8 * np.linalg.norm(want)
    for none in ([], [empty]):
        case.bparts = none
        run_partitioned(ctx, case)
        assert not case.dK.any() and not case.dV.any()
