"""Kernels that are set up while the kernel before them still runs."""
import glob
import os
import re

from paper_2411_05799_gb300 import build


def _early_kernels():
    text = "".join(open(p).read() for p in sorted(glob.glob(os.path.join(build.CSRC, "*.cu"))))
    for name in sorted(set(re.findall(r"launch_early\((\w+)", text))):
        head = re.search(r"\n%s\(|\s%s\(const|void[^;{]*\b%s\(" % (name, name, name), text)
        assert head, name
        body = text[head.start() + 1:]
        yield name, body[:body.index("\n}\n")]


def test_early_kernels_wait_and_promise_no_constant_memory():
    """Such a kernel waits before it touches memory that another wrote, and takes no pointer as const
    __restrict__ and no value by __ldg: both promise that the memory stays as it is for as long as the
    kernel lives, which begins before its predecessor has written its results, and let the loads be
    moved ahead of the wait."""
    kernels = dict(_early_kernels())
    assert {"pack_input_kernel", "loss_grad_kernel", "grads_finish_kernel", "adam_kernel", "gemm_tn_kernel"} <= set(kernels)
    for name, body in kernels.items():
        assert "early_wait()" in body, name
        assert "__restrict__" not in body and "__ldg" not in body and "ld.global.nc" not in body, name
