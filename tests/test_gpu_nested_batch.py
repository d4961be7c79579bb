"""Nested decode of several sequences in shared passes: every sequence gets the bits of a launch of its own, at the edges
of its tiles (rows of one vector, of one or two consumer groups, of two vectors per thread; layers smaller than the grid;
empty, whole and one-neuron lists; passes of three to eight sequences and rests, two sequences in a launch each), with any
workspace that was accepted, with inputs out of range, and from a graph whose launches wait for one another."""
import pytest
import torch

from tests._util import launches

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clada():
    from paper_2502_19078_b200 import binding, build
    build.build()
    binding.load()
    return binding


def _case(clada, B, d, F, dtype, act):
    g = torch.Generator(device="cuda").manual_seed(1000 * B + d + F)
    mk = lambda s, *shape: torch.randn(shape, generator=g, device="cuda").mul_(s).to(dtype)
    layer = clada.Layer(mk(0.05, F, d), None if act == 2 else mk(0.05, F, d), mk(0.05, F, d), activation=act)
    order = torch.stack([torch.randperm(F, generator=g, device="cuda") for _ in range(B)]).to(torch.int32)
    counts = torch.randint(0, F + 1, (B, 4), generator=g, device="cuda").to(torch.int32)
    counts[0] = F                                            # everything kept
    counts[1] = 0                                            # nothing kept
    if B > 2:
        counts[2] = 1
    level = (torch.arange(B, device="cuda") % 4).to(torch.int32)
    return layer, order, counts, level, mk(1.0, B, d)


def _run(clada, layer, order, counts, level, x, y_dtype, ws):
    y = torch.full((x.shape[0], x.shape[1]), 7.0, device="cuda").to(y_dtype)
    kept = torch.full((x.shape[0],), -1, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    clada.clada_sparse_ffn_decode_nested(layer, x, order, counts, level, y, ws, kept, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert kept.tolist() == [int(counts[b, int(level[b])]) for b in range(x.shape[0])]
    return y


@pytest.mark.parametrize("B,d,F,dtype,act", [
    (2, 8, 1, torch.bfloat16, 0), (3, 8, 31, torch.float16, 1), (8, 2048, 147, torch.bfloat16, 0),
    (4, 2048, 149, torch.bfloat16, 1), (9, 2056, 500, torch.float16, 0), (5, 2056, 333, torch.bfloat16, 2),
    (2, 1024, 13400, torch.bfloat16, 2), (7, 4096, 1000, torch.bfloat16, 0), (3, 4104, 700, torch.float16, 0),
    (8, 5120, 450, torch.bfloat16, 0), (3, 8192, 300, torch.bfloat16, 0), (6, 8192, 300, torch.float16, 2),
    (3, 512, 1376, torch.float32, 0), (4, 1024, 640, torch.float32, 2), (8, 1032, 640, torch.float32, 1),
    (3, 4096, 200, torch.float32, 0), (10, 256, 40000, torch.bfloat16, 0),
    (3, 8, 1, torch.bfloat16, 0), (3, 1024, 13400, torch.bfloat16, 2), (4, 4104, 700, torch.float16, 0),
    (4, 8192, 300, torch.bfloat16, 2), (4, 2568, 200, torch.float32, 0),
])
def test_batch_bits_are_those_of_single_launches(clada, B, d, F, dtype, act):
    layer, order, counts, level, x = _case(clada, B, d, F, dtype, act)
    ws, one = clada.new_workspace(layer, B, 0), clada.new_workspace(layer, 1, 0)
    y = _run(clada, layer, order, counts, level, x, torch.float32, ws)
    for b in range(B):
        s = slice(b, b + 1)
        assert torch.equal(y[s], _run(clada, layer, order[s], counts[s], level[s], x[s], torch.float32, one)), b
    assert torch.all(y[1] == 0)
    assert torch.equal(y, _run(clada, layer, order, counts, level, x, torch.float32, one))  # the smallest accepted workspace
    h = dtype if dtype != torch.float32 else torch.float16
    assert torch.equal(y.to(h), _run(clada, layer, order, counts, level, x, h, ws))          # 16-bit outputs: one rounding


def test_repeated_indices_count_as_often_as_they_are_listed(clada):
    layer, order, counts, level, x = _case(clada, 3, 512, 300, torch.bfloat16, 0)
    order[0, 10:20] = order[0, 5]
    ws = clada.new_workspace(layer, 3, 0)
    y = _run(clada, layer, order, counts, level, x, torch.float32, ws)
    for b in range(3):
        s = slice(b, b + 1)
        assert torch.equal(y[s], _run(clada, layer, order[s], counts[s], level[s], x[s], torch.float32, ws))


def test_launches_do_not_grow_with_the_batch(clada):
    """Four launches whatever the batch, not one per sequence."""
    layer, order, counts, level, x = _case(clada, 8, 512, 1000, torch.bfloat16, 0)
    ws, y = clada.new_workspace(layer, 8, 0), torch.empty(8, 512, device="cuda")
    names = [n for n, _ in launches(lambda: clada.clada_sparse_ffn_decode_nested(layer, x, order, counts, level, y, ws))]
    assert len(names) == 4 and not any("sparse_ffn_kernel" in n for n in names), names


@pytest.mark.parametrize("B,d,F,dtype,act,singles,passes", [
    (2, 1024, 300, torch.bfloat16, 0, 2, 0),                                            # two: a launch each
    (3, 2048, 300, torch.float16, 2, 0, 1), (3, 2056, 300, torch.float16, 2, 3, 0),     # three, no gate: rows of 256, 257,
    (3, 4088, 300, torch.float16, 2, 3, 0), (3, 4096, 300, torch.float16, 2, 0, 1),     # 511 and 512 vectors
    (3, 2560, 16384, torch.bfloat16, 0, 0, 1), (3, 2560, 16385, torch.bfloat16, 0, 3, 0),  # gated: 80 MB a matrix
    (3, 7168, 300, torch.bfloat16, 0, 0, 1), (3, 7680, 300, torch.bfloat16, 0, 3, 0),   # six ring stages beside x, and five
    (5, 7168, 300, torch.bfloat16, 0, 0, 1), (6, 7168, 300, torch.bfloat16, 0, 1, 1),   # five, and four: a pass of five
    (4, 8192, 300, torch.bfloat16, 0, 4, 0), (8, 8192, 300, torch.float16, 2, 0, 1),
    (4, 2560, 300, torch.float32, 0, 0, 1), (4, 4096, 300, torch.float32, 1, 4, 0),
    (11, 512, 300, torch.bfloat16, 1, 0, 2), (17, 512, 300, torch.float32, 0, 1, 2),
])
def test_which_batches_take_a_pass(clada, B, d, F, dtype, act, singles, passes):
    """Both sides of each line of the rule, and the same bits from a launch per sequence."""
    layer, order, counts, level, x = _case(clada, B, d, F, dtype, act)
    ws, y = clada.new_workspace(layer, B, 0), torch.empty(B, d, device="cuda")
    names = [n for n, _ in launches(lambda: clada.clada_sparse_ffn_decode_nested(layer, x, order, counts, level, y, ws))]
    assert sum("sparse_ffn_kernel" in n for n in names) == singles and sum("nested_sums_kernel" in n for n in names) == passes
    assert len(names) == singles + 4 * passes
    y = _run(clada, layer, order, counts, level, x, torch.float32, ws)
    for b in range(B):
        s = slice(b, b + 1)
        assert torch.equal(y[s], _run(clada, layer, order[s], counts[s], level[s], x[s], torch.float32, ws)), b


@pytest.mark.parametrize("d,dtype", [(512, torch.bfloat16), (1032, torch.float32)])
@pytest.mark.parametrize("B,bad", [(3, 0), (3, 2), (8, 7)])
@pytest.mark.parametrize("kind", ["level below", "level above", "count below", "count above", "indices"])
def test_inputs_out_of_range_are_clamped_and_reported(clada, B, bad, d, dtype, kind):
    """One sequence's level, count or indices outside the layer: reported, made harmless as a launch of its own makes them,
    and nothing to the other sequences."""
    F = 700
    layer, order, counts, level, x = _case(clada, B, d, F, dtype, 0)
    counts[bad] = torch.tensor([60, 300, 100, 200])
    clean = _run(clada, layer, order, counts, level, x, torch.float32, clada.new_workspace(layer, B, 0))
    if kind.startswith("level"):
        level[bad] = -1 if kind == "level below" else 6
    elif kind.startswith("count"):
        counts[bad] = -3 if kind == "count below" else F + 5
    else:
        order[bad, :60:7] = torch.tensor([-7, F, F + 100, -2 ** 31, 2 ** 31 - 1, -1, F, F, 2 * F], dtype=torch.int32, device="cuda")

    def run(s, ws):
        y, kept = torch.full((B, d), 7.0, device="cuda")[s], torch.full((B,), -1, dtype=torch.int32, device="cuda")[s]
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        clada.clada_sparse_ffn_decode_nested(layer, x[s], order[s], counts[s], level[s], y, ws, kept, status)
        return y, kept, int(status.item())

    y, kept, status = run(slice(0, B), clada.new_workspace(layer, B, 0))
    assert status == 8  # CLADA_STATUS_BAD_INDEX
    one = clada.new_workspace(layer, 1, 0)
    for b in range(B):
        yb, kb, sb = run(slice(b, b + 1), one)
        assert torch.equal(y[b:b + 1], yb) and torch.equal(kept[b:b + 1], kb) and (sb != 0) == (b == bad)
        if b != bad:
            assert torch.equal(y[b], clean[b])


@pytest.mark.parametrize("B,d,F,dtype", [(4, 2048, 1500, torch.bfloat16), (3, 1024, 4100, torch.float16), (9, 512, 700, torch.bfloat16)])
def test_a_graph_that_feeds_each_launch_from_the_one_before(clada, B, d, F, dtype):
    """Two of a pass's launches read ahead of their wait: in a graph that makes the lists, decodes over them and decodes
    again from that output, replayed with other inputs each time, every read comes after what writes it."""
    layer, order, counts, _, x = _case(clada, B, d, F, dtype, 1)
    ws, status = clada.new_workspace(layer, B, 0), torch.zeros(1, dtype=torch.int32, device="cuda")
    scores, tau = torch.empty(B, F, device="cuda"), torch.full((B,), 0.75, device="cuda")
    logits, token = torch.empty(B, 3000, device="cuda"), torch.arange(B, dtype=torch.int32, device="cuda")
    level = torch.zeros(B, dtype=torch.int32, device="cuda")
    s, h = torch.empty(B, device="cuda"), torch.empty(B, device="cuda")
    y, z = torch.empty(B, d, dtype=dtype, device="cuda"), torch.empty(B, d, device="cuda")

    def step(sync):
        for part in (lambda: clada.clada_nested_build(scores, tau, 0.4, 0.2, order, counts),
                     lambda: clada.clada_cogload_level(logits, token, 8.0, 7.4, s, h, level),
                     lambda: clada.clada_sparse_ffn_decode_nested(layer, x, order, counts, level, y, ws, None, status),
                     lambda: clada.clada_sparse_ffn_decode_nested(layer, y, order, counts, level, z, ws, None, status)):
            part()
            if sync:
                torch.cuda.synchronize()

    g = torch.Generator(device="cuda").manual_seed(5)

    def inputs():
        scores.uniform_(0.5, 1.5, generator=g)
        logits.normal_(0.0, 3.0, generator=g)
        x.normal_(0.0, 1.0, generator=g)

    inputs()
    step(True)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step(False)
    for _ in range(20):
        inputs()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got = y.clone(), z.clone(), order.clone(), level.clone()
        step(True)
        for a, b in zip(got, (y, z, order, level)):
            assert torch.equal(a, b)
        assert torch.isfinite(z).all() and z.abs().max() > 0
    assert int(status.item()) == 0
