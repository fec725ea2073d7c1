"""Rules that the CUDA sources keep and that no run can show to be broken."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_04929_b200", "csrc")


def _kernels():
    """name -> (parameters, body) of every kernel."""
    out = {}
    for fn in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, fn)).read())
        for part in text.split("__global__")[1:]:
            m = re.search(r"(k_\w+|\w+_kernel)\s*\(", part)
            if not m:
                continue
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(part[i], 0)
                i += 1
            start = end = part.index("{", i)
            while True:
                depth += {"{": 1, "}": -1}.get(part[end], 0)
                end += 1
                if not depth:
                    break
            out[m.group(1)] = (part[m.end():i - 1], part[start:end])
    return out


def test_kernels_that_start_early_promise_nothing_about_what_they_wait_for():
    """A kernel that is launched ahead of the end of the one before (it calls pdl_wait) must not declare its operands
    unchanged for its lifetime: the compiler may then load them ahead of the wait."""
    early = {k: v for k, v in _kernels().items() if "pdl_wait()" in v[1]}
    assert {"k_sweep_rows", "k_rank_rows", "k_compensate", "k_row_range", "k_grid_score", "k_grid_pick"} <= set(early)
    for name, (params, body) in early.items():
        assert "__restrict__" not in params and "__restrict__" not in body, name
        for arg in re.findall(r"__ldg\(([^()]*)", body):  # read-only loads: the factors alone
            assert re.match(r"(U|Pm|uo|po)\b", arg.strip()), (name, arg)
