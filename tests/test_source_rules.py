"""Rules of the CUDA sources that no run can show to be kept, read from the sources."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_23569_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _functions(src, qualifier):
    """name -> (parameters, body) of the functions declared with `qualifier`."""
    out = {}
    for m in re.finditer(qualifier + r"\b", src):
        n = re.compile(r"(\w+)\s*\(").search(src, m.end())
        while n.group(1) in ("__launch_bounds__", "__align__"):
            n = re.compile(r"(\w+)\s*\(").search(src, src.index(")", n.end()))
        depth, i = 1, n.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(src[i], 0)
            i += 1
        params = src[n.end():i - 1]
        b = re.compile(r"[;{]").search(src, i)
        if b.group() == ";":
            continue  # a declaration
        depth, j = 1, b.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[j], 0)
            j += 1
        p, q = out.get(n.group(1), ("", ""))
        out[n.group(1)] = (p + params, q + src[b.end():j])
    return out


def _loop_before(src, pos):
    """The text from the start of the innermost loop body around `pos` up to it."""
    depth = 0
    for i in range(pos, -1, -1):
        if src[i] == "}":
            depth += 1
        elif src[i] == "{":
            if depth == 0:
                head = src[max(0, i - 200):i].rstrip()
                if re.search(r"\b(for|while) \([^{}]*\)$", head):
                    return src[i:pos]
            else:
                depth -= 1
    raise AssertionError("no loop")


def test_tensor_memory_loads_start_from_a_converged_warp():
    """tcgen05.ld is .sync.aligned: in the loop body that makes it, the warp is converged before it and after the
    last poll, which its lanes leave one by one."""
    calls = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        src = _source(os.path.basename(path))
        assert "tcgen05.ld." not in src  # only through the helpers
        for m in re.finditer(r"tc::tmem_ld\d+\(", src):
            before = _loop_before(src, m.start())
            at = before.rfind("tc::converge();")
            assert at >= 0 and not re.search(r"bar_wait|wait_bar\(", before[at:]), (path, src[m.start() - 80:m.end()])
            calls += 1
    assert calls >= 10


def test_tensor_memory_waits_name_their_registers():
    for path in glob.glob(os.path.join(CSRC, "*.*")):
        assert not re.search(r"\btmem_wait_ld\(\s*\)", _source(os.path.basename(path))), path


def test_overlapping_kernels_read_nothing_as_constant():
    """Kernels launched over the end of the one before (launch_chained): that one still writes their input after they
    have begun, so neither they nor the functions they call read it as data constant for their lifetime."""
    seen = set()
    for name in ("cnn.cu", "cnn_tc.cu"):
        src = _source(name)
        chained = set(re.findall(r"launch_chained\(\s*\"\w+\",\s*(\w+)", src))
        funcs = _functions(src, "__global__")
        helpers = _functions(src, "__device__")
        for k in chained:
            params, body = funcs[k]
            assert "grid_wait();" in body, k
            for h, (hp, hb) in helpers.items():
                if re.search(r"\b%s\s*(<[^;{}]*>)?\(" % h, body):
                    params, body = params + "," + hp, body + hb
            assert "__ldg" not in body, k
            assert not re.search(r"const[^,]*\*\s*__restrict__", params), k
            seen.add(k)
    assert {"k_conv_tc", "k_conv_tma", "k_conv_wgrad", "k_wgrad_reduce", "k_loss"} <= seen


def test_the_votes_bounds_check_keeps_the_warp_together():
    """The check build's test is made by each lane for its own member: a lane that fails it may not leave the others to
    the warp's barriers that follow."""
    _, body = _functions(_source("sigma.cu"), "__global__")["k_vote"]
    assert body.count("HTS_IN_BOUNDS") == len(re.findall(r"__all_sync\(\s*FULL,[^;]*HTS_IN_BOUNDS", body)) > 0
    assert "continue;" not in body
