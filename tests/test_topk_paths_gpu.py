"""The ways a Top-k selection can be carried out (one kernel with the sweep, a CTA or a cluster per candidate list, a
separate emission, passes over the block) at the sizes where one takes over from another, and Block-Sign at the edges of
its own dispatch: against the oracle, index sets and sign bits exact, floats within the parity tolerance."""
import numpy as np
import pytest
import torch

import oracle
from paper_2205_05632_b200 import BLOCKSIGN, RANDK, TOPK, CompAMS
from parity import Pair, close, unpack_sign_bits

pytestmark = pytest.mark.gpu


def run(n, offs, comp, ratio, draw, steps=5, seed=None):
    d = int(offs[-1])
    gen = torch.Generator(device="cuda").manual_seed(n * 1000003 + d)
    p = Pair(n, d, offs, comp, ratio, seed=seed)
    try:
        p.start(0.1 * torch.randn(d, generator=gen, device="cuda"))
        for t in range(steps):
            p.step(draw(gen, n, d), check_e=t in (1, steps - 1))
        return p.gpu.buffer("status").cpu().tolist()
    finally:
        p.close()


def normal(gen, n, d):
    return torch.randn(n, d, generator=gen, device="cuda")


def levels(gen, n, d):  # few distinct magnitudes: thresholds shared by many entries
    return torch.randint(-400, 401, (n, d), generator=gen, device="cuda").float()


@pytest.mark.parametrize("n,offs", [
    (1, [0, 8192]), (2, [0, 8193]), (4, [0, 65536]), (1, [0, 131072]), (9, [0, 131072]), (10, [0, 131072]), (1, [0, 131073]),
    (3, [0, 1, 3, 2051, 2100, 4150, 12343, 12350, 30001]), (2, [0, 2048, 4097, 8193 + 4097]),
    (5, list(np.cumsum([0] + [700 + 97 * k for k in range(40)]))),
])
@pytest.mark.parametrize("ratio", [0.01, 0.1, 0.3])
@pytest.mark.parametrize("draw", [normal, levels])
def test_sweep_and_selection_in_one_kernel(n, offs, ratio, draw):
    run(n, offs, TOPK, ratio, draw, steps=4)


@pytest.mark.parametrize("n,sizes,ratio", [
    (4, [50000, 2500] * 8, 0.01),                 # topk_small behind topk_select
    (8, [20000, 30] * 9, 0.02),                   # ... for the sake of a short sweep
    (2, [90000, 900, 30, 7] * 3 + [20000] * 9, 0.02),  # in front of it: two orders of kernels, as for the following
    (20, [20000, 2500] * 8, 0.02),                # a wave of selecting CTAs
    (10, [20000] * 33 + [4000, 9] * 24, 0.03),    # more than a wave of both
    (1, [(1 << 21) + 5, 4096, 30], 0.1),          # with an emission kernel
    (3, [30000, 4096, 60000, 17], 0.2),           # without lists
])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_steps_with_small_blocks_do_not_depend_on_what_is_waited_for(n, sizes, ratio, dtype):
    # back to back, in between kernels that write what the step reads, and one at a time: the same bits
    offs = list(np.cumsum([0] + sizes))
    d, steps = int(offs[-1]), 8
    gen = torch.Generator(device="cuda").manual_seed(d)
    batches = [normal(gen, n, d).to(dtype) for _ in range(steps)]
    results = []
    for wait in (False, True):
        opt, theta, G = CompAMS(n, d, offs, TOPK, ratio), torch.zeros(d, device="cuda"), torch.empty_like(batches[0])
        for t in range(steps):
            G.copy_(batches[t])
            theta.add_(0.125)
            if wait:
                torch.cuda.synchronize()
            opt.step(G, theta)
            if t % 3 == 2:  # two steps without anything between them
                opt.step(G, theta)
            if wait:
                torch.cuda.synchronize()
        assert opt.check_status() == 0
        results.append([theta] + [opt.buffer(name).clone() for name in ("E", "m", "v", "vhat")])
        opt.close()
    for name, a, b in zip(("theta", "E", "m", "v", "vhat"), *results):
        assert torch.equal(a, b), name


@pytest.mark.parametrize("n,d,ratio", [
    (1, (1 << 21) + 5, 0.1),    # list emitted by a kernel of its own, 16 CTAs
    (2, 3000001, 0.111),        # the densest selection with a candidate list ...
    (2, 3000001, 0.112),        # ... and one without: always the dense passes
    (3, 1500003, 0.02), (16, 400001, 0.02), (1, 262144, 0.002), (7, 150001, 0.05), (2, (1 << 21) + 3, 0.001),
    (4, 262144, 0.2), (9, 20001, 0.2), (1, 262145, 0.2),  # no list: by its cluster, by the dense passes
])
@pytest.mark.parametrize("draw", [normal, levels])
def test_long_lists(n, d, ratio, draw):
    run(n, [0, d], TOPK, ratio, draw, steps=5)


def test_lists_of_several_rounds_that_one_cta_each_takes():
    # more lists than clusters would fit: 5500 entries per list, a round is 4096
    st = run(16, [40000 * b for b in range(21)], TOPK, 0.11, normal, steps=6)
    assert st[2] > st[1]


def test_long_and_short_lists_side_by_side():
    sizes = [900001, 37, 4096, 4097, 600003, 20000, 1, 70001, 250007, 9000]
    st = run(3, list(np.cumsum([0] + sizes)), TOPK, 0.04, normal, steps=6)
    assert st[2] > st[1]  # most selections inside their lists


@pytest.mark.parametrize("n,offs", [
    (16, [0, 64 * 8192 - 31]), (17, [0, 64 * 8192 - 31]), (1, [0, 256 * 8192]), (1, [0, 256 * 8192 + 1]), (4, [0, 1, 2050, 6150, 10249]),
    (25, [0, 3, 2049, 20001]), (2, [0, 5, 8197, 16391, 24601, 24603]), (16, [0, 160 * 8192]), (16, [0, 160 * 8192 + 1]),
    (17, list(np.cumsum([0] + [611 + 37 * k for k in range(80)]))), (4, [0, 15 * 8192]), (5, [0, 19 * 8192]), (5, [0, 20 * 8192]),
    (9, [0, 36 * 8192 - 32]), (9, [0, 36 * 8192]), (19, [0, 37, 20003]), (20, [0, 37, 20003]), (40, [0, 1000, 1003, 30001]),
    (24, [0, 95 * 8192 - 40]), (24, [0, 96 * 8192 - 40]),
    # 17 workers and more: tables of 4 workers, 32 per round
    (17, [0, 3, 70 * 8192 + 5]), (32, [0, 97 * 8192]), (33, [0, 5, 2054, 97 * 8192 + 3]), (40, list(np.cumsum([0] + [9001] * 90))),
    (65, [0, 4101, 97 * 8192 + 4101]),
])
def test_blocksign_server_kernels_and_who_adds_up_the_scales(n, offs):
    run(n, offs, BLOCKSIGN, 1.0, normal, steps=4)


def test_blocksign_sweep_that_asks_ahead():
    run(3, [0, 31, 9001, 9001 + 3 * 8192, 22369623], BLOCKSIGN, 1.0, normal, steps=2)  # n d just above 2^26


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,sizes", [
    # mostly empty tiles: blocks that end inside a warp's first 128 coordinates, at its edges, at the next warp's, in the last one
    (6, [1, 31, 32, 97, 127, 128, 129, 1023, 1024, 1025, 1151, 7168, 7169, 3] * 5), (2, [200] * 150), (33, [5, 130, 1500] * 4),
])
def test_blocksign_sweep_of_mostly_empty_tiles(n, sizes, dtype):
    run(n, list(np.cumsum([0] + sizes)), BLOCKSIGN, 1.0, lambda gen, n, d: normal(gen, n, d).to(dtype), steps=3)


def test_blocksign_whole_tiles_with_zeros_and_subnormals():
    def draw(gen, n, d):
        g = torch.randn(n, d, generator=gen, device="cuda")
        g[:, ::7] = 0.0
        g[:, 3::11] = -0.0
        g[:, 5::13] *= 2.0 ** -130
        return g
    run(3, [0, 2 * 8192, 5 * 8192 + 70], BLOCKSIGN, 1.0, draw, steps=3)


@pytest.mark.parametrize("d", [8192, 8192 + 5])  # a whole tile; tiles that are not
@pytest.mark.parametrize("beside", [1.0, 0.0, 2.0 ** -130])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_blocksign_an_infinity_adds_the_same_beside_any_values(d, beside, dtype):
    # its pattern read as a number, 2^128, whose quotient by d is the scale: the other values, at most 1 each, are below half an ulp
    opt = CompAMS(1, d, [0, d], BLOCKSIGN)
    g = torch.ones(1, d, device="cuda", dtype=dtype)
    g[0, 4000:4008] = beside
    g[0, 4002] = float("inf")
    opt.compress(g)
    bits, scales = opt.message_buffers()
    assert scales.item() == float(np.float32(2.0 ** 128 / d))
    opt.apply(torch.zeros(d, device="cuda"))
    opt.close()


@pytest.mark.parametrize("n,offs,ratio", [
    (3, [0, 31, 1055, 1056, 9300, 30011], 0.02), (2, [0, 20001], 0.25), (2, [0, 20001], 0.95), (4, [0, 1024, 2048, 10240], 0.125),
])
def test_randk_spans_that_share_words_and_overflow_their_room(n, offs, ratio):
    run(n, offs, RANDK, ratio, normal, steps=4, seed=11)


@pytest.mark.parametrize("n,offs,ratio", [
    # several slots per thread: one block per CTA, blocks that begin inside one, a row whose last CTA is short
    (1, [0, 4 * 757761], 0.05), (2, [0, 1048575], 0.1), (3, [0, 1, 40, 500009, 500010, 520000, 1500001], 0.1),
    (2, list(np.cumsum([0] + [1500 + 7 * k for k in range(700)])), 0.06),
    # two, three, eight and four per thread on 148 SMs, blocks that begin inside a CTA's slots
    (4, [0, 700001, 1600003], 0.1), (8, [0, 4099, 1200007], 0.1), (8, [0, 900001, 900002, 903000, 3300001], 0.1),
    (4, list(np.cumsum([0] + [3000 + 11 * k for k in range(250)])), 0.3),
])
def test_randk_several_slots_per_thread(n, offs, ratio):
    run(n, offs, RANDK, ratio, normal, steps=3, seed=5)


@pytest.mark.parametrize("comp", [TOPK, BLOCKSIGN, RANDK])
def test_messages_are_complete_between_the_two_halves_of_a_step(comp):
    # whatever a whole step leaves to its server side, compress() alone leaves what the step would have sent
    n, offs = 3, [0, 5, 8197, 24601]
    d = offs[-1]
    gen = torch.Generator(device="cuda").manual_seed(5)
    a, b = CompAMS(n, d, offs, comp, 0.02), CompAMS(n, d, offs, comp, 0.02)
    ta, tb = torch.zeros(d, device="cuda"), torch.zeros(d, device="cuda")
    for _ in range(3):
        G = torch.randn(n, d, generator=gen, device="cuda")
        a.step(G, ta)
        b.compress(G)
        first, second = (m.clone() for m in b.message_buffers())
        b.apply(tb)
        want, want2 = a.message_buffers()
        if comp != BLOCKSIGN:  # the pairs of a segment come in any order
            order, order_w = torch.argsort(first, 1), torch.argsort(want, 1)
            first, second = first.gather(1, order), second.gather(1, order)
            want, want2 = want.gather(1, order_w), want2.gather(1, order_w)
        assert torch.equal(first, want) and torch.equal(second, want2)
        assert torch.equal(ta, tb)
    a.close()
    b.close()


@pytest.mark.parametrize("n,offs,ratio", [
    (2, [0, 1500], 0.02), (2, [0, 300, 40300], 0.02),                # one kernel: blocks without and with a list
    (16, [0, 400001], 0.02), (1, [0, (1 << 21) + 5], 0.1),           # clusters; a list emitted by a kernel of its own
    (3, [0, 600003, 604099, 1504100], 0.01),                         # clusters, one CTA per list, a block in shared memory
])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("share", [1.2, 3.0, 1e9])  # of k_b: coordinates that are not finite (1e9: all of them)
def test_gradients_that_are_not_finite_select_by_key_and_index(n, offs, ratio, bad, share):
    # an overflow in a mixed-precision step: more such values in a block than it keeps, in the step after the first (whose
    # selection has a list) and in the first one. Which are kept is unspecified for the caller; here: the lowest indices
    d = offs[-1]
    gen = torch.Generator(device="cuda").manual_seed(d)
    for good_steps in (0, 3):
        opt = CompAMS(n, d, offs, TOPK, ratio)
        theta = torch.zeros(d, device="cuda")
        for _ in range(good_steps):
            opt.step(torch.randn(n, d, generator=gen, device="cuda"), theta)
        G = torch.randn(n, d, generator=gen, device="cuda")
        want = torch.zeros(n, d, dtype=torch.bool, device="cuda")
        for lo, hi in zip(offs, offs[1:]):
            k = max(1, int(ratio * (hi - lo)))
            count = min(hi - lo, int(share * k) + 1)
            for i in range(n):
                where = lo + torch.randperm(hi - lo, generator=gen, device="cuda")[:count].sort().values
                G[i, where] = bad
                want[i, where[:k]] = True
        opt.step(G, theta)
        assert opt.check_status() == 0
        idx = opt.buffer("topk_idx").long()
        got = torch.zeros(n, d, dtype=torch.int32, device="cuda")
        got.scatter_add_(1, idx, torch.ones_like(idx, dtype=torch.int32))
        assert torch.equal(got, want.int())
        for _ in range(2):  # the handle goes on
            opt.step(torch.randn(n, d, generator=gen, device="cuda"), theta)
            assert opt.check_status() == 0
        opt.close()


@pytest.mark.parametrize("n,d,ratio,count", [(1, 131072, 0.02, 2800), (4, 65536, 0.02, 1500), (1, 400001, 0.009, 3700)])
def test_a_short_list_that_cannot_decide_leaves_the_block_to_its_whole_cluster(n, d, ratio, count):
    # a list of at most 4096 entries, which the first CTA of a cluster takes alone, whose k_b-th largest key lies beyond its
    # histogram: `count` nearly all equal magnitudes far above the last threshold. The lowest indices win
    gen = torch.Generator(device="cuda").manual_seed(d)
    opt = CompAMS(n, d, [0, d], TOPK, ratio)
    theta = torch.zeros(d, device="cuda")
    k = int(ratio * d)
    assert k < count <= 4096
    for _ in range(12):
        opt.step(torch.randn(n, d, generator=gen, device="cuda"), theta)
    before = opt.buffer("status").cpu().tolist()
    e = opt.buffer("E").clone()
    G = -e
    for i in range(n):
        where = torch.randperm(d, generator=gen, device="cuda")[:count]
        G[i, where] += 1024.0  # x = (1024 - e) + e is 1024 but for the rounding of the difference, elsewhere it is 0
    x = (G + e).cpu().numpy()
    opt.step(G, theta)
    after = opt.buffer("status").cpu().tolist()
    assert after[0] == 0 and after[1] - before[1] == n and after[5] - before[5] == n
    idx = np.sort(opt.buffer("topk_idx").cpu().numpy(), axis=1)
    for i in range(n):
        assert np.array_equal(idx[i], np.flatnonzero(oracle.topk_keep_mask(x[i], k)))
    opt.close()


@pytest.mark.parametrize("n,offs,ratio", [(3, [0, 5, 8197, 24601], 0.02), (2, [0, 900001], 0.01), (2, [0, 3000, 900001], 0.3)])
@pytest.mark.parametrize("comp", [TOPK, BLOCKSIGN, RANDK])
def test_apply_averages_what_the_message_buffers_hold(n, offs, ratio, comp):
    # the caller works on the messages between the two halves: one worker dropped, another's values halved
    d = offs[-1]
    gen = torch.Generator(device="cuda").manual_seed(9)
    opt = CompAMS(n, d, offs, comp, ratio, record_average=True)
    theta = 0.1 * torch.randn(d, generator=gen, device="cuda")
    want = {"theta": theta.cpu().numpy().copy(), **{k: np.zeros(d, dtype=np.float32) for k in ("m", "v", "vhat")}}
    for t in range(4):
        opt.compress(torch.randn(n, d, generator=gen, device="cuda"))
        first, second = opt.message_buffers()
        second[0] *= 0.5
        second[n - 1] = 0.0
        C = np.zeros((n, d), dtype=np.float64)
        if comp == BLOCKSIGN:
            signs = unpack_sign_bits(first.cpu().numpy(), opt.buffer("sign_word_offsets").cpu().numpy(), np.asarray(offs))
            C[:] = np.where(signs, -1.0, 1.0) * np.repeat(second.cpu().numpy(), np.diff(offs), axis=1)
        else:
            np.put_along_axis(C, first.cpu().numpy().astype(np.int64), second.cpu().numpy().astype(np.float64), 1)
        opt.apply(theta)
        gbar = C.sum(0).astype(np.float32) / np.float32(n)
        oracle.amsgrad(gbar, want["m"], want["v"], want["vhat"], want["theta"], 1e-3, 0.9, 0.999, 1e-8)
        close(opt.buffer("gbar"), gbar, "gbar", t)
        close(theta, want["theta"], "theta", t)
        for name in ("m", "v", "vhat"):
            close(opt.buffer(name), want[name], name, t)
        assert opt.check_status() == 0
    opt.close()


@pytest.mark.parametrize("n,offs,ratio", [(3, [0, 5, 8197, 24601], 0.02), (2, [0, 900001], 0.01), (2, [0, 3000, 900001], 0.3)])
@pytest.mark.parametrize("comp", [TOPK, BLOCKSIGN, RANDK])
def test_apply_sees_what_the_stream_did_to_theta_since_compress(n, offs, ratio, comp):
    # decoupled weight decay in front of the server's update, with the worker side done before or after it
    d = offs[-1]
    gen = torch.Generator(device="cuda").manual_seed(10)
    a, b = CompAMS(n, d, offs, comp, ratio), CompAMS(n, d, offs, comp, ratio)
    ta = 0.1 * torch.randn(d, generator=gen, device="cuda")
    tb = ta.clone()
    for _ in range(6):
        G = torch.randn(n, d, generator=gen, device="cuda")
        ta *= 0.9
        a.step(G, ta)
        b.compress(G)
        tb *= 0.9
        b.apply(tb)
        assert torch.equal(ta, tb)
    a.close()
    b.close()


def test_dense_passes_stand_by_in_the_first_steps_only():
    # one worker's long block: a list that fails is left to the dense passes of the whole GPU while a handle is new, to its
    # cluster afterwards
    n, d = 1, (1 << 21) + 5
    gen = torch.Generator(device="cuda").manual_seed(13)
    p = Pair(n, d, [0, d], TOPK, 0.05)
    try:
        p.start(torch.zeros(d, device="cuda"))
        launches, walks = [], []
        for t in range(38):
            before = p.gpu.buffer("status").cpu().tolist()[1], p.gpu.launch_count()
            p.step((0.2 if t in (20, 36) else 1.0) * torch.randn(n, d, generator=gen, device="cuda"), check_e=t in (0, 20, 21, 36, 37))
            launches.append(p.gpu.launch_count() - before[1])
            walks.append(p.gpu.buffer("status").cpu().tolist()[1] - before[0])
        assert walks[20] == 1 and walks[36] == 1  # the lists did fail
        assert launches[30] == launches[34] + 1
        # a replaced accumulator starts over
        p.gpu.set_state(p.gpu.get_state())
        theta, at = p.theta_gpu.clone(), p.gpu.launch_count()
        p.gpu.step(torch.randn(n, d, generator=gen, device="cuda"), theta)
        assert p.gpu.launch_count() - at == launches[30]
    finally:
        p.close()
