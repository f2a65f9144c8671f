"""Rules that the kernels of csrc/em_screen.cu keep and that no run can show to be broken without risking the device: read from the source."""
import re
from pathlib import Path

SOURCE = (Path(__file__).resolve().parent.parent / "paper_2606_10896_b200" / "csrc" / "em_screen.cu").read_text()


def _body(start):
    """Text of the braces that open behind ``start``."""
    first = SOURCE.index("{", start)
    depth = 0
    for i in range(first, len(SOURCE)):
        depth += {"{": 1, "}": -1}.get(SOURCE[i], 0)
        if depth == 0:
            return SOURCE[first:i + 1]
    raise AssertionError("unbalanced braces")


def _kernels():
    for m in re.finditer(r"__global__ void __launch_bounds__\([^;{]*?\)\s+(screen_\w+)\(", SOURCE):
        yield m.group(1), _body(m.end())


def test_a_verdict_that_a_kernel_can_give_is_read_once_per_cta():
    writes = re.compile(r"ctl\[SC_DENSE\] = 1")
    by_call = [m.group(1) for m in re.finditer(r"__device__ (?:__forceinline__ )?void (screen_\w+)\(", SOURCE) if writes.search(_body(m.end()))]
    assert "screen_convert" in by_call
    seen = set()
    for name, body in _kernels():
        if writes.search(body) or any(re.search(rf"\b{f}\s*[<(]", body) for f in by_call):
            seen.add(name)
            assert not re.search(r"if \((p\.)?ctl\[SC_DENSE\] != 0\) return", body), f"{name}: every thread decides for itself whether to leave"
    assert {"screen_sweep_kernel", "screen_transform_kernel", "screen_rows_kernel", "screen_group_sort_kernel"} <= seen


def test_a_warpgroup_changes_its_registers_with_one_instruction():
    """The sweep's roles: softmax warps (two warpgroups), converting warps (one), and three roles that share the last."""
    body = dict(_kernels())["screen_sweep_kernel"]
    give = body.index("auto give_registers")
    assert body.count("setmaxnreg.dec") == 1 and give < body.index("setmaxnreg.dec") < body.index(";\n", give)
    softmax, converting, last = (body.index(s) for s in ("if (warp < S::CONVERTER)", "else if (CONVERT && warp < S::PRODUCER)", "else if (give_registers(), role == S::PRODUCER)"))
    assert softmax < body.index("setmaxnreg.inc") < converting < last and body.count("setmaxnreg.inc") == 1
    assert body[converting:last].count("give_registers()") == 1 and body[last:].count("give_registers()") == 1


def test_the_sweeps_loads_have_landed_before_it_ends_whoever_leaves_first():
    """The softmax warps can leave (another CTA's verdict) when the producer has asked for everything and has seen no reason to leave itself."""
    body = dict(_kernels())["screen_sweep_kernel"]
    producer = body[body.index("role == S::PRODUCER)"):body.index("role == S::FETCH)")]
    drain = producer.index("BAR(S::PFULL + h % S::PS)")
    depth = producer[producer.index("{"):drain].count("{") - producer[producer.index("{"):drain].count("}")
    assert depth == 2, "the loop over the last stages stands in the producer's own block, under no condition"
    assert "if (!CONVERT && ut > 0 && lane == 0) bar_wait(BAR(S::UFULL)" in producer[drain:]
