"""Decode launches whose CTAs cannot all be resident at a time: beside a kernel that keeps half of the SMs for longer than
a decode takes, and beside another decode on a second stream.  Every launch ends, its control words are back at zero and
its outputs are the bits of an undisturbed run.  (Five sequences over lists take passes that do not meet; they are there
for their chained launches.)  How far two kernels overlap is the scheduler's affair, so who leaves a meeting, who shares the
parts and how a group waits for a late member is checked in self-tests whose CTAs are made to begin late."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clada():
    from paper_2502_19078_b200 import binding, build
    build.build()
    binding.load()
    return binding


def _layer(clada, d, F, dtype):
    g = torch.Generator(device="cuda").manual_seed(d + F)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda").mul_(0.05).to(dtype)
    return clada.Layer(mk(F, d), mk(F, d), mk(F, d))


class _Decode:
    def __init__(self, clada, B, d, F, dtype, nested, tau=0.8):
        self.clada, self.layer, self.nested = clada, _layer(clada, d, F, dtype), nested
        g = torch.Generator(device="cuda").manual_seed(B)
        self.x = torch.randn(B, d, generator=g, device="cuda").to(dtype)
        self.scores = torch.rand(B, F, generator=g, device="cuda") + 0.5
        self.tau = torch.full((B,), tau, device="cuda")
        self.order = torch.empty(B, F, dtype=torch.int32, device="cuda")
        self.counts = torch.empty(B, 4, dtype=torch.int32, device="cuda")
        clada.clada_nested_build(self.scores, self.tau, 0.25, 0.1, self.order, self.counts)
        self.level = torch.zeros(B, dtype=torch.int32, device="cuda")
        self.ws, self.status = clada.new_workspace(self.layer, B, 0), torch.zeros(1, dtype=torch.int32, device="cuda")

    def run(self):
        y = torch.full(self.x.shape, float("nan"), device="cuda")
        if self.nested:
            self.clada.clada_sparse_ffn_decode_nested(self.layer, self.x, self.order, self.counts, self.level, y, self.ws,
                                                      None, self.status)
        else:
            self.clada.clada_sparse_ffn_decode(self.layer, self.x, self.scores, self.tau, 1, y, self.ws, status=self.status)
        return y

    def clean(self):
        return int(self.status.item()) == 0 and int(self.ws[:256].view(torch.int32).abs().sum().item()) == 0


FORMS = [(1, 1024, 2400, torch.bfloat16, False), (1, 512, 1376, torch.float32, False), (2, 1024, 2400, torch.bfloat16, False),
         (2, 512, 1376, torch.float32, False), (4, 512, 1376, torch.float32, False), (6, 1024, 2400, torch.float16, False),
         (20, 1024, 2400, torch.bfloat16, False), (1, 1024, 2400, torch.bfloat16, True), (5, 1024, 2400, torch.bfloat16, True)]
NOTHING_KEPT = [(1, 1024, 2400, torch.bfloat16, False, 9.0), (1, 512, 1376, torch.float32, True, 9.0)]


@pytest.mark.parametrize("B,d,F,dtype,nested", FORMS)
def test_beside_a_kernel_that_keeps_half_of_the_sms(clada, B, d, F, dtype, nested):
    dec = _Decode(clada, B, d, F, dtype, nested)
    want = dec.run()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    other_layer = _layer(clada, 8192, 128 * (sms // 2), torch.bfloat16)  # one persistent CTA per 128 neurons of one token tile
    norm = torch.empty(other_layer.d_ff, device="cuda")
    clada.clada_down_norms(other_layer, norm)
    other_layer.set_down_norm(norm)
    X, ws = torch.randn(128, 8192, device="cuda").to(torch.bfloat16), clada.new_workspace(other_layer, 1, 128)
    scores = torch.empty(1, other_layer.d_ff, device="cuda")
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    outs = []
    for _ in range(20):
        with torch.cuda.stream(other):
            clada.clada_prefix_scores(other_layer, X, [0, 128], scores, ws)
        outs += [dec.run(), dec.run()]
        torch.cuda.synchronize()
    assert dec.clean()
    for y in outs:
        assert torch.equal(y, want)


@pytest.mark.parametrize("first", range(len(FORMS)))
def test_two_streams(clada, first):
    """Launches of two streams that share the SMs as they come."""
    decs = [_Decode(clada, *FORMS[first]), _Decode(clada, *FORMS[(first + 2) % len(FORMS)])]
    want = [d.run() for d in decs]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    outs = [[], []]
    for _ in range(40):
        for i in (0, 1):
            with torch.cuda.stream(streams[i]):
                outs[i].append(decs[i].run())
    torch.cuda.synchronize()
    for i in (0, 1):
        assert decs[i].clean()
        for y in outs[i]:
            assert torch.equal(y, want[i])


@pytest.mark.parametrize("form", NOTHING_KEPT)
def test_launches_that_keep_nothing(clada, form):
    """They take their counts back without a meeting: y is zero, and the control words are zero for the dense pass behind each, which
    numbers its CTAs by one of them.  On two streams, so that launches begin a few CTAs at a time."""
    none, dense = [_Decode(clada, *form) for _ in (0, 1)], [_Decode(clada, 6, 1024, 2400, torch.bfloat16, False) for _ in (0, 1)]
    want = dense[0].run()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for i in (0, 1):
        none[i].ws = dense[i].ws  # one workspace for both kinds
    torch.cuda.synchronize()
    outs = []
    for _ in range(40):
        for i in (0, 1):
            with torch.cuda.stream(streams[i]):
                outs.append((none[i].run(), dense[i].run()))
    torch.cuda.synchronize()
    for i in (0, 1):
        assert none[i].clean() and dense[i].clean()
    for zero, y in outs:
        assert torch.all(zero == 0) and torch.equal(y, want)


@pytest.mark.parametrize("n,late", [(1, 0), (1, 1), (5, 0), (5, 5), (5, 2), (64, 1), (64, 40), (64, 63)])
def test_parts_of_a_meeting(clada, n, late):
    """Who leaves and who does what, with CTAs made to begin late: no part is lost and none is done twice, and the parts of
    CTAs that left are shared by all that came later."""
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(20):
        report = torch.full((n, 2), -9, dtype=torch.int32, device="cuda")
        clada.clada_selftest_meeting(ws, n, late, report, status)
        got = report.tolist()
        if late in (0, n):
            assert got == [[c, n] for c in range(n)]
        else:
            assert [parts for _, parts in got[:n - late]] == [0] * (n - late)
            assert sorted(got[n - late:]) == [[c, late] for c in range(late)]
        assert int(status.item()) == 0 and int(ws.view(torch.int32).abs().sum().item()) == 0


@pytest.mark.parametrize("limit", [100, 1000])
def test_a_group_waits_for_a_member_that_begins_late(clada, limit):
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    status, report = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.full((4,), -9, dtype=torch.int32, device="cuda")
    clada.clada_selftest_late_member(ws, limit, report, status)
    assert report.tolist() == [1, 1, 1, 1]
    assert int(status.item()) == 0 and int(ws.view(torch.int32).abs().sum().item()) == 0
