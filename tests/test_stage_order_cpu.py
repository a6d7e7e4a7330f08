"""The kernels that refill a shared-memory stage by tensor copies store into it with ordinary
instructions first; each of them releases the stage between the two (generic and async proxy)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_14130_gb300", "csrc")


def _body(src, at):
    """The text between the braces of the function whose parameter list starts at `at`."""
    k = src.index("{", src.index(")", at))
    depth, i = 1, k + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    return src[k:i]


def staged_kernels():
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        src = re.sub(r"//[^\n]*", "", src)
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(", src):
            body = _body(src, m.end() - 1)
            if re.search(r"\bissue_\w+<", body):
                yield f, m.group(1), body


def test_every_refilled_stage_is_released_before_the_barrier():
    found = {}
    for f, name, body in staged_kernels():
        loop = body[re.search(r"\bfor \(;;|\bfor \(; t < a.ntiles|\bfor \(int k = 0; t < a.ntiles", body).start():]
        found[name] = len(re.findall(r"^\s*stage_release\(\);", loop, re.M))
    assert set(found) == {"k_step_tma", "k_adj_tma", "k_adj_scaled_tma", "k_step_tile", "k_adj_tile"}
    assert all(n == 1 for n in found.values()), found


@pytest.mark.parametrize("name", ["stage_release", "fence_proxy_async_smem"])
def test_release_is_the_proxy_fence(name):
    src = open(os.path.join(CSRC, "tma.cuh")).read()
    body = _body(src, src.index(f"void {name}("))
    assert ("fence_proxy_async_smem()" if name == "stage_release" else "fence.proxy.async.shared::cta") in body
