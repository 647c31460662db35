"""Which loads the digit sorts use, read from the source.  A wave pass lets the
next pass start while it still writes (pdl_trigger), so that pass must not read
the keys, payloads or histograms through the read-only path: `__ldg` and `const
__restrict__` loads need memory that no one writes while the kernel is alive, and
may be moved over the wait.  No run shows the difference."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def kernel(name):
    """(parameters, body) of a __global__ function of radix.cu, comments dropped."""
    with open(os.path.join(ROOT, "paper_2409_03970_gb300", "csrc", "radix.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    m = re.search(r"__global__[^;{]*?\b" + name + r"\(([^{]*)\) \{(.*?)\n\}\n", text, re.S)
    return m.group(1), m.group(2)


def writer(body, call):
    """Who writes what `call` reads, as each of its uses says."""
    return re.findall(rf"\b{call}<([^>]+)>\(", body)


def test_wave_passes():
    params, body = kernel("radix_pass_kernel")
    assert "if constexpr (WAVE) pdl_trigger();" in body
    for p in params.split(","):
        if p.strip().startswith("const"):
            assert "__restrict__" not in p, p
    assert "__ldg" not in body
    for call in ("load", "move_values"):
        assert writer(body, call) == ["WAVE ? PREDECESSOR : NOBODY"], call
    # the histogram; a look-back pass's first tile, after its predecessor's end, may read it plainly
    assert [x.strip() for x in re.findall(r"[^;{}\n]*\bhist\b[^;\n]*;", body)] == [
        "if constexpr (WAVE && CL > 1) digit_total = load_from<PREDECESSOR>(hist + (tid >> 1));",
        "if constexpr (WAVE && CL == 1) digit_total = load_from<PREDECESSOR>(hist + d);",
        "excl = t.sum_below(hist[d]);"]
    assert body.rindex("} else {", 0, body.index("hist[d]")) > body.rindex("if constexpr (WAVE) {")


def test_cluster_sort():
    params, body = kernel("radix_cluster_kernel")
    assert "__restrict__" not in params and "__ldg" not in body
    for call in ("load", "move_values"):
        assert writer(body, call) == ["THIS_KERNEL"], call
