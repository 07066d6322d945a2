"""Operands that cp.async copies into shared memory (generic proxy) are fenced before
the tensor cores read them (async proxy). An mbarrier orders threads, not proxies, so
without a fence.proxy.async after the wait a tcgen05.mma may read what the slot held
before; no result shows that reliably, so the order is checked in the source. Operands
that TMA writes need none. No GPU is touched."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2301_13601_gb300", "csrc")


def kernels_with_copied_operands():
    """(name, body) of each kernel that issues MMAs and copies with cp.async inside its roles."""
    out = []
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for part in re.split(r"(?=__global__ )", text)[1:]:
            body = part[:part.find("\n}\n")]
            if "mma_bf16_leader(" in body and "cp_async_arrive_noinc(" in body:
                out.append((re.search(r"(\w+)\(const", body).group(1), body))
    return out


def test_the_kernels_are_found():
    assert [k for k, _ in kernels_with_copied_operands()] == ["conv3x3_tc_kernel", "wgrad_tc_kernel"]


@pytest.mark.parametrize("name, operands, copied", [
    ("conv3x3_tc_kernel", ("full_bar",), "!L::SWZ"),            # the 16-channel input rows
    ("wgrad_tc_kernel", ("xf_bar", "gf_bar"), "!(SWX && SWG)"),  # 16-channel x or g rows
])
def test_mma_warp_fences_after_its_waits(name, operands, copied):
    body = dict(kernels_with_copied_operands())[name]
    issuer = body[body.index("warp == CONV_MMA_WARP) {", body.index("CONV_LOAD_WARP")):]
    waits = [issuer.index(f"mbar_wait(&{bar}") for bar in operands]
    fence = issuer.find(f"if constexpr ({copied}) tc::fence_proxy_async();")
    mma = min(i for i in (issuer.find("mma_bf16_leader("), issuer.find("conv_row_mmas<")) if i >= 0)
    assert max(waits) < fence < mma
