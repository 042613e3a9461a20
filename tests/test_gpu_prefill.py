"""GPU parity of the prefill expert path (tcgen05 grouped GEMM, token blocks of
128 pairs, A operand dequantised into tensor memory) against the CPU oracle:
ragged token blocks, empty and overloaded experts, an odd number of W2 row
blocks, both group sizes, fractional zeros, ODP with protected tokens, the
automatic path switch, many work items per CTA, the narrow and the wide geometry,
expired waits, and the Mixtral-8x7b-shaped prefill layer on sampled tokens."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from helpers import assert_close, boundary_tokens, condition_routing, flat, oracle_layer, oracle_mats, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

PATH_GEMV, PATH_GEMM = 1, 2  # mc_set_path: the mma.sync GEMV, the tcgen05 grouped GEMM


@pytest.fixture(scope="module")
def mc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_06270_gb300 import build
    build.build()
    import paper_2410_06270_gb300 as m
    m.load()
    m.set_debug(0, 1_000_000_000)
    return m


def _run(mc, L, path, tokens=None):
    condition_routing(L, L.mu)
    shape = mc.Shape(L.E, L.H, L.F, L.group)
    packed = mc.pack_experts(shape, L.bits, flat(L, "codes"), flat(L, "scale"), flat(L, "zero"))
    x, g, p = to_dev(L)
    ws = mc.alloc_workspace(shape, L.T)
    old = mc.set_path(path)
    try:
        y = mc.moe_forward(x, g, shape, L.bits, packed, L.mu, p, workspace=ws)
        mc.check_status(ws)
    finally:
        mc.set_path(old)
    torch.cuda.synchronize()
    got = y.float().cpu().numpy()
    return got if tokens is None else got[list(tokens)]


def _check(mc, L, path=PATH_GEMM, tokens=None):
    got = _run(mc, L, path, tokens)
    ref, *_ = oracle_layer(L, oracle_mats(L), tokens)
    return assert_close(got, ref, "prefill path=%d T=%d H=%d F=%d g=%d bits=%s mu=%g" % (
        path, L.T, L.H, L.F, L.group, list(map(int, L.bits)), L.mu))


@pytest.mark.parametrize("group", [64, 128])
def test_prefill_small_layer(mc, group):
    """H 384 (three W2 row blocks: one pair plus a lone block), ragged blocks."""
    L = synth.make_layer(300, 384, 512, 8, group, [3, 2, 1, 3, 2, 2, 1, 3], 301 + group, gate_std=0.1, mu=0.4,
                         protect_frac=0.2, zero_mode="fractional")
    _check(mc, L)


@pytest.mark.parametrize("bits", [[1] * 8, [2] * 8, [3] * 8])
def test_prefill_single_bit_width(mc, bits):
    L = synth.make_layer(260, 256, 256, 8, 64, bits, 320 + bits[0], gate_std=0.1)
    _check(mc, L)


def test_prefill_skewed_loads(mc):
    """Skewed routing: some experts get several full 128-pair blocks, some none."""
    L = synth.make_layer(700, 256, 384, 8, 128, [3, 3, 2, 2, 1, 2, 3, 1], 330, gate_std=0.05, skew=(3.0, 0.9))
    _check(mc, L)


def test_prefill_sixteen_experts(mc):
    L = synth.make_layer(400, 256, 256, 16, 64, [1, 2, 3] * 5 + [2], 340, gate_std=0.1, mu=0.5)
    _check(mc, L)


def test_automatic_switch_agrees_with_gemv(mc):
    """T = 256 (512 pairs; the GEMM from 240 pairs) takes the GEMM automatically;
    the GEMV path on the same inputs agrees with it and with the oracle."""
    L = synth.make_layer(256, 256, 512, 8, 64, [3, 2, 2, 1, 3, 2, 2, 3], 350, gate_std=0.1, mu=0.3,
                         protect_frac=0.1)
    auto = _run(mc, L, 0)
    gemv = _run(mc, L, 1)
    ref, *_ = oracle_layer(L, oracle_mats(L))
    assert_close(auto, ref, "automatic path")
    assert_close(gemv, ref, "GEMV path")
    assert_close(auto, gemv.astype(np.float64), "automatic vs GEMV")


def test_bounded_wait_reports_timeout_and_context_survives(mc):
    """With the weight producer starved every wait of both GEMM launches runs out: the
    call returns, the status word says so, and the next call is right again."""
    L = synth.make_layer(300, 256, 384, 8, 64, [3, 2, 1, 3, 2, 2, 1, 3], 360, gate_std=0.1)
    condition_routing(L)
    shape = mc.Shape(L.E, L.H, L.F, L.group)
    packed = mc.pack_experts(shape, L.bits, flat(L, "codes"), flat(L, "scale"), flat(L, "zero"))
    x, g, p = to_dev(L)
    ws = mc.alloc_workspace(shape, L.T)
    old = mc.set_path(PATH_GEMM)
    try:
        mc.set_debug(1, 20_000_000)  # the producer issues nothing; waits give up after 20 ms
        try:
            mc.moe_forward(x, g, shape, L.bits, packed, workspace=ws)
            with pytest.raises(mc.MCError) as ei:
                mc.check_status(ws)
            assert ei.value.code == mc.ERR_TIMEOUT
        finally:
            mc.set_debug(0, 1_000_000_000)
        y = mc.moe_forward(x, g, shape, L.bits, packed, workspace=ws)
        mc.check_status(ws)
    finally:
        mc.set_path(old)
    torch.cuda.synchronize()
    ref, *_ = oracle_layer(L, oracle_mats(L))
    assert_close(y.float().cpu().numpy(), ref, "GEMM after an expired wait")


@pytest.mark.parametrize("T,H,F,E,group", [
    (2560, 128, 8192, 8, 128),   # W1,W3 items of one column step, 64 per token block; lone W2 blocks
    (300, 128, 16384, 16, 64),   # the same with token blocks of at most 64 pairs
    (2300, 1408, 1024, 8, 64),   # W2: five block pairs and a lone block per token block
    (2300, 1408, 1024, 8, 128),
])
def test_prefill_many_items_per_cta(mc, T, H, F, E, group):
    """Several items per CTA in both launches, so that every ring and barrier goes round:
    thousands of one-step W1,W3 items (the item ring's tight case), wide and narrow, and a
    lone W2 block followed by another item.  The tokens at the edges of the experts'
    token blocks against the oracle, all of them against the GEMV path."""
    L = synth.make_layer(T, H, F, E, group, [1, 2, 3, 2] * (E // 4), 370 + T, gate_std=0.05)
    condition_routing(L)
    idx, _, pr = oracle.route(L.x_f32(), L.gate_f32(), 0.0)
    pairs = np.diff(oracle.permute(idx, pr, E)[0])
    assert (pairs.max() <= 64) == (T == 300)
    tokens = boundary_tokens(L, blocks=(128,))
    got = _run(mc, L, PATH_GEMM)
    ref, *_ = oracle_layer(L, oracle_mats(L), tokens)
    assert_close(got[tokens], ref, "GEMM T=%d H=%d F=%d g=%d" % (T, H, F, group))
    assert_close(got, _run(mc, L, PATH_GEMV).astype(np.float64), "GEMM vs GEMV")


def test_prefill_narrow_and_wide_agree(mc):
    """The longest prefixes of a batch whose largest expert has 64 and 65 pairs: one takes
    the narrow geometry (two accumulator sets), the other the wide one.  Both against the
    oracle, and bit for bit the same on the tokens they share."""
    L = synth.make_layer(300, 384, 2048, 8, 128, [3, 2, 1, 3, 2, 2, 1, 3], 380, gate_std=0.05)
    condition_routing(L)
    idx, *_ = oracle.route(L.x_f32(), L.gate_f32(), 0.0)
    largest = np.stack([np.cumsum((idx == e).any(axis=1)) for e in range(L.E)]).max(axis=0)
    out = []
    for most in (64, 65):
        T = int(np.searchsorted(largest, most, side="right"))
        assert largest[T - 1] == most
        P = dataclasses.replace(L, T=T, x=L.x[:T])
        out.append(_run(mc, P, PATH_GEMM))
        ref, *_ = oracle_layer(P, oracle_mats(P))
        assert_close(out[-1], ref, "largest expert %d pairs" % most)
    assert np.array_equal(out[1][:len(out[0])], out[0])


def test_prefill_mixtral_shape(mc):
    """Mixtral-8x7b-shaped prefill layer, 4096 tokens with skewed expert loads
    (the prefill workload), outputs checked on the tokens of every expert's
    first and last pair in its first and last (ragged) 128-pair token block,
    from the oracle's permutation, plus the first and last token."""
    L = synth.config_prefill(T=4096)
    tokens = sorted(set(boundary_tokens(L, 0.0, blocks=(128,)) + [0, L.T - 1]))
    assert len(tokens) >= 2 * L.E
    _check(mc, L, path=0, tokens=tokens)
