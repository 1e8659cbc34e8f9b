"""Every wait between the roles of the prefill kernel has a limit: a named barrier would wait for ever for a warpgroup
that gave up, and a role that went on after a wait ran out would overwrite what others still read."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_02647_b200", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_roles_of_the_prefill_kernel_meet_only_at_bounded_waits():
    src = source("prefill_sm100.cu")
    assert not re.search(r"\b(bar|barrier)\.(sync|red|arrive)|__syncthreads_|named_barrier", src)
    # block barriers: set-up, teardown, the self-test; none while the roles run
    kernel = src[src.index("prefill_sm100_kernel(const"):src.index("position_tables_kernel(const")]
    assert [len(re.findall("__syncthreads", x)) for x in kernel.split("if (warp == kProducerWarp) {\n        asm volatile(\"setmaxnreg")] == [1, 1]
    # polls of a barrier stand in a loop with a limit, or behind one that is not (the phase may be over already)
    for poll in re.finditer(r"mbar_try_wait\(", src):
        line = src[src.rindex("\n", 0, poll.start()) + 1:src.index("\n", poll.start())]
        before = src[:poll.start()].rsplit("\n", 2)[-2]
        assert "bool mbar_try_wait" in line or re.search(r"for \(uint32_t \w+ = 0; \w+ < \w+", before + line), line


def test_producer_stops_when_a_wait_ran_out():
    src = source("prefill_sm100.cu")
    producer = src[src.index("setmaxnreg.dec"):src.index("} else if (warp == kMmaWarp)")]
    main = producer[:producer.rindex("item_info")]                # (the end marker is published whatever happened)
    for wait in re.finditer(r"mbar_wait_call\(", main[:main.rindex("break;")]):
        line = main[main.rindex("\n", 0, wait.start()) + 1:main.index("\n", wait.start())]
        assert re.search(r"(ok|q_free) = mbar_wait_call|!mbar_wait_call\(.*\) break;", line), line
