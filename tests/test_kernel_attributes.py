"""Function attributes (a kernel's limit of dynamic shared memory) belong to the device, not to a context.  A launch that set
one to the size of its own call could lower it under the larger launch that another context's thread is about to make, which
is then refused half-way through a call.  The window between the two is too narrow to be hit on demand, so the rule itself
is checked: attributes are set by the prepare functions, which ltri_create runs, and nowhere else.

In the same way a refused launch has to end its call where it happens: nothing on a GPU refuses one on demand."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2412_04757_b200", "csrc")
FILES = sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu*")))
# a definition at the start of a line: its name, then everything up to the closing brace in the first column
FUNCTION = re.compile(r"^[A-Za-z][^\n;=]*?\b(\w+)\([^;{}]*\)\s*\{.*?^\}", re.M | re.S)


@pytest.mark.parametrize("name", FILES)
def test_attributes_are_set_when_a_context_is_created_only(name):
    text = open(os.path.join(CSRC, name)).read()
    calls = text.count("cudaFuncSetAttribute(") + text.count("allow_smem(")
    inside = 0
    for f in FUNCTION.finditer(text):
        n = f.group(0).count("cudaFuncSetAttribute(") + f.group(0).count("allow_smem(")
        assert n == 0 or f.group(1).startswith("prepare_") or f.group(1) == "allow_smem", f"{name}: {f.group(1)} sets a limit"
        inside += n
    assert inside == calls, f"{name}: an attribute is set outside the functions seen here"


def test_every_prepare_function_runs_at_creation():
    text = {f: open(os.path.join(CSRC, f)).read() for f in FILES}
    parts = set(re.findall(r"^cudaError_t (prepare_\w+)\([^;]*;", text["common.cuh"], re.M)) - {"prepare_kernels"}
    body = [f.group(0) for f in FUNCTION.finditer(text["ltri_api.cu"]) if f.group(1) == "prepare_kernels"]
    assert len(body) == 1 and parts and all(p + "(" in body[0] for p in parts)
    create = [f.group(0) for f in FUNCTION.finditer(text["ltri_api.cu"]) if f.group(1) == "ltri_create"]
    assert len(create) == 1 and "prepare_kernels(ctx->d" in create[0]


@pytest.mark.parametrize("name", FILES)
def test_the_result_of_every_launch_is_looked_at(name):
    # a statement that begins with the launch drops its result, and the kernels behind it run on what it did not write
    text = open(os.path.join(CSRC, name)).read()
    assert not re.search(r"(^|[;{}]|\)|\belse)\s*\n\s*launch(_chained(_cluster)?)?\(", text), name


def test_the_pull_kernel_fits_beside_the_large_kernels():
    # 18 warps of 96 registers a thread leave 1024 registers on two of an SM's four partitions: a warp of 32 a thread.  What a
    # kernel may use follows from its launch bounds: 65536 registers over the threads of the CTAs that an SM has to hold.
    text = open(os.path.join(CSRC, "kernels_state.cu")).read()
    threads = int(re.search(r"kPullThreads = (\d+);", text).group(1))
    m = re.search(r"__launch_bounds__\(kPullThreads(?:, ([^;{}]*?))?\)\s+k_pull_pack\(", text)
    ctas = eval((m.group(1) or "1").replace("kPullThreads", str(threads)).replace("/", "//"))
    assert 65536 // (ctas * threads) <= 32
