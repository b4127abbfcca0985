"""Rules of the kernel sources that no run can show reliably."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2007_07760_gb300", "csrc")


def kernels():
    """(name, parameters, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+_kernel)\s*\(([^{]*)\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield m.group(1), m.group(2), text[m.end():i]


def test_dependent_kernels_read_with_ordered_loads():
    """A kernel launched with programmatic serialization may be resident while the kernel ahead of it
    still writes. A __restrict__ parameter promises memory that nothing writes while the kernel is
    there, which lets its loads pass the wait: no kernel that waits takes one."""
    found = {name: "__restrict__" in params for name, params, body in kernels()
             if re.search(r"\bpdl_wait\(\)|march_strip<|dvm_strip<", body)}
    assert {"step_march_kernel", "batch_march_kernel", "batch_advance_kernel", "dvm_march_kernel", "step_fast_kernel",
            "mass_final_kernel"} <= set(found)
    assert not [k for k, bad in found.items() if bad]


def test_mass_sum_triggers_before_it_reads_an_argument():
    """The next step is placed when the sum's one CTA triggers: 0.11 us later where an argument is loaded first."""
    params, body = next((p, b) for name, p, b in kernels() if name == "mass_final_kernel")
    before = body[:body.index("pdl_trigger()")]
    assert not [w for w in re.findall(r"(\w+)\s*(?:,|$)", params) if re.search(rf"\b{w}\b", before)]


def test_batch_constants_are_read():
    """Every constant that a batch sends with each launch is read by its kernel."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "dugks_march.cuh")).read())
    fields = re.search(r"struct BatchUniform \{(.*?)\};", text, flags=re.S).group(1)
    names = [w for line in fields.split(";") for w in re.findall(r"\*?(\w+)\s*(?:,|$)", line.strip())]
    host = open(os.path.join(CSRC, "dugks_batch.cu")).read()
    assert "be1" in names and "status" in names
    for n in names:
        assert re.search(rf"\bu\.{n}\b", text) or re.search(rf"\bu\.{n}\b(?!\s*=)", host), n
