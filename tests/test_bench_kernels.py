"""The benchmark takes a chain's kernel from the library and keys recorded traffic
by that kernel's own sources."""
from __future__ import annotations

import importlib.util
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1804_07250_gb300", "csrc")


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_kernels_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_every_kernel_name_has_the_sources_that_define_it(bench):
    with open(os.path.join(CSRC, "tl_host.cpp")) as f:
        body = re.search(r"const char\* tl_chain_kernel\(tl_chain\* c\)\n\{(.*?)\n\}", f.read(), re.S).group(1)
    names = set(re.findall(r'"(\w+_kernel)"', body))
    assert names == set(bench.CHAIN_KERNELS)
    for name, sources in bench.CHAIN_KERNELS.items():
        text = "".join(open(os.path.join(ROOT, s)).read() for s in sources)
        assert re.search(r"__global__ void[^;{]*\b%s\(" % name, text), name


@pytest.mark.gpu
def test_names(bench):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1804_07250_gb300 as T
    ctx, half, other = T.Context(0), T.thresholds(scalar=1 << 31), T.thresholds(scalar=3 << 29)

    def chain(dom, th, **plan):
        c = T.Chain(ctx, dom, seed=1, th=th)
        if plan:
            c.set_plan(**plan)
        return c
    assert chain(T.Domain.aztec(100), half).kernel == "small_kernel"
    assert chain(T.Domain.rect(100, 600), half).kernel == "regdom_kernel"     # narrow, but not small
    c = chain(T.Domain.aztec(100), half)
    c.density_begin(1, 0)
    assert c.kernel == "regdom_kernel"
    assert chain(T.Domain.aztec(500), half, kernel=2).kernel == "resident_kernel"
    assert chain(T.Domain.aztec(500), other).kernel == "words_kernel"
    assert chain(T.Domain.aztec(500), other, kernel=1).kernel == "pass_global_kernel"
    assert chain(T.Domain.rect(2000, 2000), T.thresholds(scalar=1 << 30)).kernel == "resident_kernel"
