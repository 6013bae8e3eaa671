"""Rules that the kernels' sources keep and that no run shows reliably: a read that is too early, or a wait that may
never end, would be a race or a hang on the GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_14352_b200", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _body(text, function):
    """The text between the braces of the function's definition."""
    at = text.index("{", text.index(")", re.search(r"\b%s\(" % function, text).end()))
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i]
    raise AssertionError(function)


@pytest.mark.parametrize("name,function", [("router.cuh", "router_logits"), ("router.cuh", "router_logits_one"),
                                           ("router.cuh", "router_logits_batch"), ("decode_layer.cu", "decode_layer_kernel")])
def test_router_reads_its_inputs_after_the_kernels_in_front_are_done(name, function):
    """The kernel in front of a call's first one may be the one that writes x: griddepcontrol.wait comes before the first
    load (prefetches into L2, and the body of a loading lambda, which runs where it is called, aside)."""
    body = re.sub(r"auto \w+ = \[&\]\(int \w+\) \{.*?\n\s*\};", "", _body(_source(name), function), flags=re.S)
    reads = [m.start() for m in re.finditer(r"__ldg\(|__ldcg\(|\*>\((a\.)?x\)\[|fetch_[wx]\(|\bx8\(", body)]
    assert reads and body.index("pdl_wait();") < min(reads)


BARRIER = r"(?:\b|\\[nt])(?:bar|barrier)(?:\.cta)?\.(?:sync|red|arrive)\b"  # (also right behind an escape in a string)


@pytest.mark.parametrize("name", ["ffn_tma.cu", "ffn_i8.cu", "pipe.cuh", "umma.cuh"])
def test_no_unbounded_barrier_among_the_warps_of_the_pipelined_kernels(name):
    """A warp whose bounded wait has run out leaves its role; a named barrier that its neighbours stand at would then never
    open.  (Barriers of the whole CTA stand only where every role passes: at the start and, behind all roles, at the end.)"""
    assert not re.search(BARRIER, _source(name))


def test_the_storing_warps_of_the_grouped_gemm_leave_together():
    """They have named barriers: each stands behind the set's vote on the unit's waits, and nothing between the vote and
    the end of the unit waits or leaves."""
    text = _source("ffn_umma.cu")
    assert len(re.findall(BARRIER, text)) == 2  # inside set_agrees and set_sync
    kernel = _body(text, "ffn_umma_kernel")
    vote = kernel.index("if (!set_agrees(part, ok)) break;")
    assert kernel.count("set_agrees(") == 1 and kernel.index("set_sync(") > vote
    unit_end = kernel.index("if (*abort_flag)", vote)
    assert not re.search(r"mbar_wait|\bbreak;|\breturn\b|\bcontinue;", kernel[vote + len("if (!set_agrees(part, ok)) break;"):unit_end])


@pytest.mark.parametrize("name", ["common.cuh", "ffn_gemv.cu", "ffn_i8.cu", "ffn_tma.cu", "ffn_umma.cu", "route.cu"])
def test_limits_of_dynamic_shared_memory_are_set_once(name):
    """The limit belongs to a kernel on a device and is shared by the contexts of all host threads: a launch that sets its own
    size may lower it between another thread's setting and its launch, which is then refused."""
    text = _source(name)
    for m in re.finditer(r"cudaFuncSetAttribute\(", text):
        assert re.search(r"raised\[dev\]\.load|if \(!(ctas_per_device|sms_of_device)\[dev\]\) \{", text[:m.start()][-400:])


def test_waits_beside_the_kernel_in_front_count_no_time():
    """The second projection of the grouped GEMM starts while the first is running, which may take longer than a wait is bounded
    by: until its producer of the activations is past its own wait for the first, the CTA says so beside its abort flag and
    no wait counts (pipe.cuh checks the count itself when it is compiled).  Every kernel with such waits sets both words."""
    kernel = _body(_source("ffn_umma.cu"), "ffn_umma_kernel")
    assert "wait_words[PIPE_FRONT] = a.phase != 0;" in kernel
    released = [m.start() for m in re.finditer(r"abort_flag\[PIPE_FRONT\] = 0;", kernel)]
    assert len(released) == 1 and kernel.rindex("pdl_wait();") < released[0] < kernel.index("walk.next(")
    assert "waited_ns(waited, before, now, front)" in _body(_source("pipe.cuh"), "mbar_wait_parked")
    for name in sorted(n for n in os.listdir(CSRC) if n.endswith(".cu")):
        text = _source(name)
        if re.search(r"mbar_wait(_warp|_parked)?\(", text):
            assert "__shared__ int wait_words[PIPE_WORDS];" in text and re.search(r"wait_words\[PIPE_FRONT\] = ", text), name


def test_reads_in_front_of_the_wait_rest_on_a_kernel_that_waited_before_its_trigger():
    """The CUDA-core kernel and the second tcgen05 projection read inputs before griddepcontrol.wait: those are older than the kernel
    directly in front, which has to have waited before it lets this one start, and nothing is launched between."""
    permute = _body(_source("route.cu"), "permute_kernel")
    assert permute.index("pdl_wait();") < permute.index("pdl_trigger();")
    gemv = _body(_source("ffn_gemv.cu"), "ffn_gemv_kernel")
    first = gemv.index("if (a.phase == 0)")
    assert re.findall(r"pdl_\w+", gemv) == ["pdl_wait", "pdl_trigger"] * 2 and gemv.index("pdl_wait") > first
    assert re.findall(r"a\.(?:experts|off|x|perm|hidden|o)\b", gemv[:first]) == ["a.experts"]
    umma = _body(_source("ffn_umma.cu"), "ffn_umma_kernel")
    empty, rest = umma[:umma.index("UmBars b;")], umma[umma.index("UmBars b;"):]
    assert empty.index("pdl_wait();") < empty.index("a.plan") < empty.index("return;")  # with this wait the others are no-ops
    assert rest.index("if (a.phase == 0) pdl_wait();") < rest.index("pdl_trigger();") < rest.index("walk.open(a.plan")
    for name in ("api.cu", "noalloc.cu"):
        launches = re.findall(r"launch_(\w+)\((\d?)", _source(name))
        for i, launch in enumerate(launches):
            if launch == ("ffn_gemv", "0"):
                assert launches[i + 1] == ("ffn_gemv", "1")
            if launch == ("ffn_umma", "0"):
                assert launches[i + 1] == ("ffn_umma", "1")
        assert ("ffn_gemv", "0") in launches
