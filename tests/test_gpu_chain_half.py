"""The forward's chain on two CTAs per chain (up to 74 runs at once) against the oracle and against the kernel with one CTA per
chain, which a batch of 38 copies of the same rows (76 chains) takes."""
import numpy as np
import pytest

import mdn_workloads as wl
from helpers import rel_err, run_gpu, run_oracle, to_torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdn():
    import paper_2605_05838_b200 as m
    m.lib()
    return m


# (tokens, preset): chunk edges, two and more chunks; preset F forgets fast: the masters are rescaled in every chunk
CASES = [(T, "S") for T in (1, 63, 64, 65, 128, 200, 449)] + [(65, "F"), (333, "F")]


@pytest.mark.parametrize("T,preset", CASES)
def test_two_ctas_per_chain(mdn, T, preset):
    """Both kernels make the same products and the same roundings in the same order: the same bits; 2e-2 to the oracle as everywhere
    on this path (a bf16 o carries its own rounding besides: half a place, 2^-8 of the largest value)."""
    import torch
    w = wl.Workload("half", B=1, T=T, H=2, dk=128, dv=128, dtype="bf16", init_state_std=0.2, seed=T, preset=preset)
    inp = wl.make_inputs(w)
    ref = run_oracle(inp)
    t = to_torch(inp)
    names = ("q", "k", "v", "beta", "log_alpha", "log_mu", "eta")
    for o_dtype in (torch.float32, torch.bfloat16):
        got = run_gpu(mdn, inp, o_dtype=o_dtype)
        half_place = 0.0 if o_dtype == torch.float32 else 2.0 ** -8 * np.abs(ref[0]).max() / np.sqrt(np.mean(ref[0] ** 2))
        assert rel_err(got[0], ref[0]) <= 2e-2 + half_place and max(rel_err(x, y) for x, y in zip(got[1:], ref[1:])) <= 2e-2
        many = mdn.chunk_fwd(*(t[n].expand(38, *t[n].shape[1:]).contiguous() for n in names), scale=inp["scale"], o_dtype=o_dtype,
                             initial_S=t["initial_S"].expand(38, -1, -1, -1).contiguous(),
                             initial_M=t["initial_M"].expand(38, -1, -1, -1).contiguous())
        for x, y in zip(got, many):
            y = y.double().cpu().numpy()
            assert np.array_equal(x, y[:1]) and np.array_equal(y[:1], y[37:])


def test_two_ctas_per_chain_packed(mdn):
    """Sequences of one token, of one chunk, of chunks and a rest in one row, each with its own start state."""
    lens = np.array([1, 64, 130, 63, 200])
    w = wl.Workload("half_packed", B=1, T=int(lens.sum()), H=3, dk=128, dv=128, dtype="bf16", varlen=True, init_state_std=0.2, seed=5)
    inp = wl.make_inputs(w, lengths=lens)
    import torch
    got, ref = run_gpu(mdn, inp, o_dtype=torch.float32), run_oracle(inp)
    assert max(rel_err(x, y) for x, y in zip(got, ref)) <= 2e-2


def eager_chunks(inp, h):
    """Which chunks of head h rescale the masters: the rule of the lazily scaled state (limits 2^-64 and 1), on G in 64 bits."""
    g11, g12, g22, out = 1.0, 0.0, 1.0, []
    for c in range(0, inp["beta"].shape[1], 64):
        al, mu, be = (inp[n][0, c:c + 64, h].astype(np.float64) for n in ("log_alpha", "log_mu", "beta"))
        for a, m, b in zip(np.exp(al), np.exp(mu), be):
            g22 *= m
            g11, g12 = a * g11, a * g12 - b * g22
        out.append(not (g11 >= 2.0 ** -64 and g22 >= 2.0 ** -64 and abs(g12) <= g22))
        if out[-1]:
            g11, g12, g22 = 1.0, 0.0, 1.0
    return out


# (tokens, constant gates alpha, mu, beta or None for preset S, mu = 0 at the last token, which chunks are eager)
EAGER_ENDS = [(1, (0.99, 0.9, 0.05), True, [1]), (17, (0.999, 0.5, 0.05), False, [1]), (64, (0.999, 0.8, 0.01), False, [1]),
              (64, (0.3, 0.5, 0.3), False, [1]), (65, None, True, [0, 1]), (128, (0.3, 0.5, 0.3), False, [1, 1]),
              (64 * 4, None, True, [0, 0, 0, 1]), (64 * 4 + 9, None, True, [0, 0, 0, 0, 1])]


@pytest.mark.parametrize("T,gates,cut,eager", EAGER_ENDS)
def test_last_chunk_rescales(mdn, T, gates, cut, eager):
    """A run that ends in a chunk that rescales the masters: its output product is the only one with no later product of the state
    in front of it.  The same bits as the kernel with one CTA per chain, every time."""
    import torch
    w = wl.Workload("half_eager", B=1, T=T, H=2, dk=128, dv=128, dtype="bf16", init_state_std=0.2, seed=T)
    inp = wl.make_inputs(w)
    if gates:
        for n, x in zip(("log_alpha", "log_mu", "beta"), (np.log(gates[0]), np.log(gates[1]), gates[2])):
            inp[n][:] = np.float32(x)
    if cut:
        inp["log_mu"][:, -1] = -np.inf
    assert eager_chunks(inp, 0) == eager_chunks(inp, 1) == [bool(e) for e in eager]
    ref, t = run_oracle(inp), to_torch(inp)
    names = ("q", "k", "v", "beta", "log_alpha", "log_mu", "eta")
    copies = lambda x: x.expand(38, *x.shape[1:]).contiguous()
    for o_dtype in (torch.float32, torch.bfloat16):
        many = mdn.chunk_fwd(*(copies(t[n]) for n in names), initial_S=copies(t["initial_S"]), initial_M=copies(t["initial_M"]),
                             scale=inp["scale"], o_dtype=o_dtype)
        want = [x[0].double().cpu().numpy() for x in many]
        for _ in range(10):
            got = run_gpu(mdn, inp, o_dtype=o_dtype)
            assert all(np.array_equal(x[0], y) for x, y in zip(got, want))
        if o_dtype == torch.float32:
            assert max(rel_err(x, y) for x, y in zip(got, ref)) <= 2e-2


@pytest.mark.parametrize("T,H,launches", [(64 * 29, 1, 2), (64 * 48 - 3, 16, 2), (64 * 51, 16, 5)])
def test_serial_chain_where_it_beats_the_scan(mdn, T, H, launches):
    """Both sides of the rule: a workspace with room for the scan, and the serial chain's kernels (intra-chunk, chain) and bits
    where two CTAs per chain are the faster way, the scan's five kernels otherwise.  A call that keeps its states is always split."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(T)
    unit = lambda x: (x / x.norm(dim=-1, keepdim=True)).bfloat16()
    q, k, v = (torch.randn((1, T, H, 128), device="cuda", generator=g) for _ in range(3))
    gates = [s * torch.rand((1, T, H), device="cuda", generator=g) for s in (0.05, -0.05, -0.05, 1.0)]
    args = (unit(q), unit(k), v.bfloat16(), *gates)
    assert mdn.workspace_layout(mdn.make_params(args[0], args[2], path="tensor")).segments > 1
    got = mdn.chunk_fwd(*args, path="tensor")
    assert mdn.last_launch_count() == launches
    one = mdn.chunk_fwd(*args, path="tensor", segments=1)
    assert mdn.last_launch_count() == 2
    if launches == 2:
        assert all(torch.equal(x, y) for x, y in zip(got, one))
    mdn.chunk_fwd(*args, path="tensor", keep_chunk_states=True)
    assert mdn.last_launch_count() == 5
