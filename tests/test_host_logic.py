"""Host-side algebra of the package that needs no GPU."""
import os
import re

import numpy as np
import torch

import oracle
from paper_2509_09679_b200.composite import cayley_pullback


def test_cayley_pullback_matches_central_differences_of_the_oracle():
    rng = np.random.default_rng(0)
    for n1 in (2, 5, 9):
        par = rng.standard_normal(n1 * (n1 - 1) // 2) * 0.4
        Gq = rng.standard_normal((n1, n1))  # dL/dQ1 of L = sum(Gq * Q1)
        loss = lambda q: float(np.sum(Gq * oracle.cayley(q, n1)))
        fd = np.zeros_like(par)
        for k in range(par.size):
            e = np.zeros_like(par)
            e[k] = 1e-6
            fd[k] = (loss(par + e) - loss(par - e)) / 2e-6
        got = cayley_pullback(torch.from_numpy(par), n1, torch.from_numpy(Gq)).numpy()
        assert np.abs(got - fd).max() <= 1e-7 * max(1.0, np.abs(fd).max())


def _bodies(text):
    """(signature, body) of every kernel of a CUDA source."""
    at = text.find("__global__")
    while at >= 0:
        start = text.index("{", at)
        depth, end = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
        yield text[at:start], text[start:end]
        at = text.find("__global__", end)


def test_kernels_that_start_early_read_by_plain_loads():
    """A kernel that waits for the one before it (grid_dep_wait) may be alive while its inputs are written: no loads that are for
    memory which does not change meanwhile (__ldg, ld.global.nc, const __restrict__ parameters), in it and in what it is built from."""
    csrc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_09679_b200", "csrc")
    seen = 0
    for name in sorted(os.listdir(csrc)):
        with open(os.path.join(csrc, name)) as f:
            text = f.read()
        kernels = list(_bodies(text))
        early = [(sig, body) for sig, body in kernels if "grid_dep_wait()" in body]
        seen += len(early)
        for sig, body in early:
            assert "__ldg(" not in body and "ld.global.nc" not in body, (name, sig)
            assert not re.search(r"const [\w:]+\s*\*\s*__restrict__", sig), (name, sig)
        if name in ("bfq_n4096.cuh", "bfq_row_again.cuh", "bfq_regroup.cuh") or (early and len(early) == len(kernels)):
            assert "__ldg(" not in text and "ld.global.nc" not in text, name
    assert seen >= 12
