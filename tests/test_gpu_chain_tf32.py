"""The forward's chain with one CTA per chain: calls of more than 74 chains.  Copies of two heads' rows fill the batch, so that the
oracle has two chains to walk."""
import numpy as np
import pytest

import mdn_workloads as wl
from helpers import rel_err, run_oracle, to_torch

pytestmark = pytest.mark.gpu

COPIES = 38   # of two chains each: 76


@pytest.fixture(scope="module")
def mdn():
    import paper_2605_05838_b200 as m
    m.lib()
    return m


def run_copies(mdn, t, inp, **kw):
    """(o, S, M) of a batch of copies, each checked to be the same bits for all of them."""
    many = lambda x: x.expand(COPIES, *x.shape[1:]).contiguous()
    got = mdn.chunk_fwd(*(many(t[n]) for n in ("q", "k", "v", "beta", "log_alpha", "log_mu", "eta")), scale=inp["scale"],
                        initial_S=many(t["initial_S"]), initial_M=many(t["initial_M"]), **kw)
    got = [x.double().cpu().numpy() for x in got]
    assert all(np.array_equal(x, np.broadcast_to(x[:1], x.shape)) for x in got)
    return [x[:1] for x in got]


REGIMES = [(0.999, 0.8, 0.001), (0.99, 0.9, 0.01), (0.98, 0.97, 0.01), (0.97, 0.98, 0.015), (0.9, 0.95, 0.1), (0.995, 0.6, 0.01),
           (0.999, 0.999, 0.0002), (0.95, 0.999, 0.015), (0.3, 0.5, 0.3)]


@pytest.mark.parametrize("T,alpha,mu,beta", [(t, *r) for r in REGIMES for t in (64 * 6 + 9, 64)])
def test_products_that_read_an_accumulator_wait_for_it(mdn, T, alpha, mu, beta):
    """Chunks that all stay lazy, all rescale the masters, or mix: every product of the chain reads what another one has accumulated.
    76 chains, ten times the same bits, 2e-2 to the oracle as everywhere on this path."""
    import torch
    w = wl.Workload("tf32_regime", B=1, T=T, H=2, dk=128, dv=128, dtype="bf16", init_state_std=0.05, seed=91)
    inp = wl.make_inputs(w)
    for n, x in zip(("log_alpha", "log_mu", "beta"), (np.log(alpha), np.log(mu), beta)):
        inp[n][:] = np.float32(x)
    inp["log_alpha"][0, 30:40, 1] = np.float32(np.log(0.2))      # a burst of fast forgetting in one head
    inp["log_mu"][0, 50:52, 0] = -np.inf                         # and a few mu = 0 tokens in the other
    ref, t = run_oracle(inp), to_torch(inp)
    first = None
    for _ in range(10):
        got = run_copies(mdn, t, inp, o_dtype=torch.float32)
        first = first or got
        assert all(np.array_equal(x, y) for x, y in zip(got, first))
    assert max(rel_err(x, y) for x, y in zip(first, ref)) <= 2e-2


@pytest.mark.parametrize("segments,T", [(3, 64 * 9), (4, 64 * 13 + 17), (5, 64 * 3 + 5)])
def test_forced_scan(mdn, segments, T):
    """38 chains: every phase of the scan has more than 74 runs, the serial chain two CTAs for each.  The first segment's tokens are
    the same bits on both kernels; a ragged tail, and more segments than chunks."""
    import torch
    from helpers import run_gpu
    w = wl.Workload("tf32_scan", B=1, T=T, H=38, dk=128, dv=128, dtype="bf16", init_state_std=0.3, seed=50 + segments)
    inp = wl.make_inputs(w)
    ref = run_oracle(inp)
    got = run_gpu(mdn, inp, path="tensor", o_dtype=torch.float32, segments=segments)
    assert mdn.last_launch_count() == 5
    assert max(rel_err(x, y) for x, y in zip(got, ref)) <= 2e-2
    per = ((T + 63) // 64 + segments - 1) // segments * 64
    one = run_gpu(mdn, inp, path="tensor", o_dtype=torch.float32, segments=1)
    assert np.array_equal(got[0][:, :per], one[0][:, :per])
