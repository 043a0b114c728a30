"""The tcgen05 convolution kernels' warps are whole where an instruction needs them
whole (csrc/conv_tcgen05.cu, read as text).

tcgen05.ld is .sync.aligned and elect.sync names all lanes, but a wait on an
mbarrier is a loop that ends lane by lane, and the last strip of a row whose length
is no multiple of 128 lets only some lanes of a warp store.  So a role goes on from
every wait through a vote of the whole warp, `together`, which brings the lanes
together and makes them give up together; the waits without one only drain copies or
MMAs before the end of the CTA."""
import os
import re

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_0902_3921_gb300", "csrc", "conv_tcgen05.cu")
POLL = "auto poll = [&](uint32_t bar, uint32_t parity) { return mbar_poll(bar, parity, abort_flag); };"
VOTE = "auto together = [](bool got) { return __all_sync(0xffffffffu, got) != 0; };"


def _kernels():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    out = {}
    for m in re.finditer(r"__global__\s+void\s+__launch_bounds__\([^)]*\)\s+(\w+)\(", text):
        nxt = text.find("\ntemplate", m.end())
        out[m.group(1)] = text[m.start():nxt if nxt > 0 else len(text)]
    assert set(out) == {"conv_tc_kernel", "wgrad_tc_kernel"}
    return out


def _args(text, at):
    depth, k = 1, at
    while depth:
        depth += {"(": 1, ")": -1}.get(text[k], 0)
        k += 1
    return text[at:k - 1]


def test_every_wait_is_voted_on_or_a_drain():
    for name, body in _kernels().items():
        assert body.count(POLL) == 1 and body.count(VOTE) == 1
        body = body.replace(POLL, "").replace(VOTE, "")
        for m in re.finditer(r"\bmbar_(?:wait|poll|wait_long)\(", body):
            if not body[:m.start()].endswith("together("):
                assert _args(body, m.end()).endswith("nullptr"), (name, body[m.start():m.start() + 80])
                assert body[:m.start()].rstrip()[-1] in ";{)", (name, body[m.start() - 40:m.start() + 40])
        # polls: no lane leaves, and nothing needs the whole warp, before the next vote
        polls = [m.start() for m in re.finditer(r"\bpoll\(", body)]
        assert polls
        for at in polls:
            rest = body[at:body.index("together(got", at)]
            assert not re.search(r"\bbreak\b|\bcontinue\b|\breturn\b|elect_lane|mma_|tmem_ld", rest), (name, rest)
            # copies of a row whose wait gave up are not issued
            for b in re.finditer(r"\bif \(lane < [^\n]*\n|lane == 0 [^\n]*\n", rest):
                assert "&& got" in b.group(0), (name, b.group(0))


def test_each_tensor_memory_load_follows_a_vote():
    for name, body in _kernels().items():
        loads = [m.start() for m in re.finditer(r"\btmem_ld(?:16|32)\(", body)]
        assert loads
        for at in loads:
            vote = body.rindex("together(mbar_wait", 0, at)
            # nothing between the vote and the load leaves lanes behind
            assert not re.search(r"\bcontinue\b|\bmine\b", body[vote:at]), name
