"""GPU parity of the gradient of the forward pass (vig_bigla_bwd_*) against the fp64 gradient oracle
(oracle/backward.py) on the same seeded inputs.  Bars as for the forward pass, per gradient tensor:
max|gpu - oracle| <= 1e-4 (fp32) / 2e-2 (bf16) of max|oracle|."""
import numpy as np
import pytest
import torch

import paper_2405_18425_b200 as vig
from paper_2405_18425_b200 import synth

from helpers import TOL, device_to_f64, oracle_log_alpha, oracle_out, random_problem, rel_err, to_device, to_stored

pytestmark = pytest.mark.gpu

NAMES = ("dq", "dk", "dv", "dlog_alpha_fwd", "dlog_alpha_bwd")


def _run(oracle, cfg, x, d_out, units=None):
    """GPU gradient of the whole problem; the oracle on `units` (a slice of the flattened (b, h) units) or on all."""
    la_f = oracle_log_alpha(oracle, x["g_fwd"], cfg.dtype, cfg.tau)
    la_b = oracle_log_alpha(oracle, x["g_bwd"], cfg.dtype, cfg.tau)
    host = dict(q=x["q"], k=x["k"], v=x["v"], f=la_f, b=la_b, g=d_out)
    d = {n: to_device(a, cfg.dtype) for n, a in host.items()}
    outs = [torch.full_like(d[n], float("nan")) for n in ("q", "k", "v", "f", "b")]
    vig.vig_bigla_bwd(d["q"], d["k"], d["v"], d["f"], d["b"], d["g"], *outs)
    torch.cuda.synchronize()
    assert vig.vig_last_device_status() == 0
    for n, a in host.items():   # inputs are never written
        np.testing.assert_array_equal(to_stored(d[n], cfg.dtype), a)
    sel = (lambda a: a) if units is None else (lambda a: a.reshape((-1, 1) + a.shape[2:])[units])
    f = lambda a: synth.stored_to_f64(sel(a), cfg.dtype)
    ref = oracle.bigla_bwd(f(x["q"]), f(x["k"]), f(x["v"]), f(la_f), f(la_b), f(d_out))
    got = [sel(device_to_f64(o, cfg.dtype)) for o in outs]
    return got, ref


def _check(got, ref, dtype, label=""):
    for name, g, r in zip(NAMES, got, ref):
        assert np.isfinite(g).all(), name
        err = rel_err(g, r)
        if label:
            print(f"observed {label} {name}: max|gpu-oracle|/max|oracle| = {err:.3e} (bar {TOL[dtype]:g})")
        assert err <= TOL[dtype], (name, err)


@pytest.mark.parametrize("dk,dv", [(16, 32), (24, 48), (32, 64), (8, 16), (40, 72), (64, 128)])
@pytest.mark.parametrize("L", [1, 2, 15, 16, 17, 100, 196, 300])
def test_bf16_gradient_small_and_ragged(oracle, dk, dv, L):
    """Lengths below, at and across the sixteen-token staging, one and two tokens, head sizes on and off the
    tensor-core gradient's."""
    cfg, x = random_problem(4000 + L, 2, 2, L, dk, dv, "bf16", gate_mean=1.0)
    got, ref = _run(oracle, cfg, x, synth.make_grad_input(cfg))
    _check(got, ref, "bf16")


@pytest.mark.parametrize("dk,dv,L", [(16, 32, 7), (5, 3, 33), (32, 64, 130), (24, 48, 50), (3, 2, 6), (128, 128, 20)])
def test_f32_gradient_shapes(oracle, dk, dv, L):
    cfg, x = random_problem(4100 + L, 2, 2, L, dk, dv, "f32", gate_mean=0.5)
    got, ref = _run(oracle, cfg, x, synth.make_grad_input(cfg))
    _check(got, ref, "f32")


def test_gradient_strong_gates(oracle):
    """Gates far below one (log alpha down to about -1 per token): states die within a few tokens, the gate
    gradients are sums of strongly cancelling terms."""
    cfg, x = random_problem(4200, 2, 2, 150, 32, 64, "f32", gate_mean=-3.0, tau=4.0)
    got, ref = _run(oracle, cfg, x, synth.make_grad_input(cfg))
    _check(got, ref, "f32")


def test_bf16_gradient_with_a_unit_beyond_the_tensor_core_range(oracle):
    """One unit whose gates sum to about -80 over a chunk: the tensor-core gradient hands that unit to the walks in the
    kernel (the counter says so); all five gradients must still meet the bar."""
    cfg, x = random_problem(4300, 2, 3, 196, 32, 64, "bf16", gate_mean=1.0)
    g = synth.stored_to_f64(x["g_bwd"], "bf16").copy()
    g[1, 1, 10:140] = -10.0            # log alpha< = -10 / 16 per token
    x["g_bwd"] = synth.store(g, "bf16")
    vig.vig_test_take_fallback_count()
    got, ref = _run(oracle, cfg, x, synth.make_grad_input(cfg))
    assert vig.vig_test_take_fallback_count() == 1
    _check(got, ref, "bf16")


@pytest.mark.parametrize("idx", [0, 1, 3, 4], ids=[synth.CONFIGS[i].name for i in (0, 1, 3, 4)])
def test_gradient_benchmark_config_full_size(oracle, idx):
    """Configurations at full size through the entry point the benchmark times; the oracle (which keeps every state of
    the sequence) on a sample of units spread over the batch: units are independent."""
    cfg = synth.CONFIGS[idx]
    x, g = synth.make_inputs(cfg), synth.make_grad_input(cfg)
    step = max(1, cfg.units // 6)
    units = slice(0, cfg.units, step) if cfg.L <= 256 else slice(0, cfg.units, max(1, cfg.units // 2))
    got, ref = _run(oracle, cfg, x, g, units)
    _check(got, ref, cfg.dtype, cfg.name)


def test_gradient_entry_point_validates_arguments():
    lib = vig.load()
    buf = torch.zeros(1 << 16, device="cuda", dtype=torch.bfloat16)
    p = buf.data_ptr()
    before = vig.vig_kernel_launch_count()
    args = [p + 8192 * n for n in range(11)]   # eleven separate 4096-element regions
    assert lib.vig_bigla_bwd_bf16(*args, 1, 1, 8, 16, 32, None) == 0
    torch.cuda.synchronize()
    launched = vig.vig_kernel_launch_count() - before
    assert launched >= 3                                                        # gates moved, forward pass for dv, the walks
    for missing in range(11):
        a = list(args)
        a[missing] = None
        assert lib.vig_bigla_bwd_bf16(*a, 1, 1, 8, 16, 32, None) == -1
    a = list(args)
    a[7] = p + 2
    assert lib.vig_bigla_bwd_bf16(*a, 1, 1, 8, 16, 32, None) == -4
    assert lib.vig_bigla_bwd_bf16(*args, 1, -1, 8, 16, 32, None) == -2
    assert lib.vig_bigla_bwd_bf16(*args, 1, 1, 8, 200, 32, None) == -3          # head size beyond the kernel's
    assert lib.vig_bigla_bwd_bf16(*args, 0, 1, 8, 16, 32, None) == 0            # empty
    assert vig.vig_kernel_launch_count() - before == launched


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("shape", [(2, 3, 196, 32), (1, 1, 1, 8), (1, 2, 5, 3), (3, 1, 33, 20)])
def test_gate_prep_gradient_matches_oracle(oracle, dtype, shape):
    """dg = dlog_alpha * sigmoid(-g) / tau against the oracle, vector body and scalar tail, separately and in place."""
    r = np.random.default_rng(sum(shape))
    g = [synth.store(r.standard_normal(shape) * 3, dtype) for _ in range(2)]
    d = [synth.store(r.standard_normal(shape), dtype) for _ in range(2)]
    f = lambda a: synth.stored_to_f64(a, dtype)
    tg = [to_device(a, dtype) for a in g]
    td = [to_device(a, dtype) for a in d]
    out = [torch.full_like(t, float("nan")) for t in td]
    vig.vig_gate_prep_bwd(tg[0], tg[1], td[0], td[1], out[0], out[1], 16.0)
    vig.vig_gate_prep_bwd(tg[0], tg[1], td[0], td[1], td[0], td[1], 16.0)   # in place over the incoming gradients
    torch.cuda.synchronize()
    for x in range(2):
        ref = oracle.gate_prep_bwd(f(g[x]), f(d[x]), 16.0)
        assert rel_err(device_to_f64(out[x], dtype), ref) <= (2.0 ** -8 if dtype == "bf16" else 1e-6)
        np.testing.assert_array_equal(to_stored(out[x], dtype), to_stored(td[x], dtype))


@pytest.mark.parametrize("B,H,L,dk,dv", [(16, 4, 196, 32, 64), (2, 2, 1100, 24, 48), (3, 2, 300, 40, 72)])
def test_gradient_is_bitwise_reproducible(B, H, L, dk, dv):
    """A pair of chunks, chunks through scratch and the walks: four calls on the same inputs give the same bytes (the
    asynchronous staging and the in-place results leave no room for a race that this would not show sooner or later)."""
    cfg, x = random_problem(4400 + L, B, H, L, dk, dv, "bf16", gate_mean=1.0)
    d = {n: to_device(a, "bf16") for n, a in x.items()}
    d["d_out"] = to_device(synth.make_grad_input(cfg), "bf16")
    la_f, la_b = torch.empty_like(d["g_fwd"]), torch.empty_like(d["g_bwd"])
    vig.vig_gate_prep_bf16(d["g_fwd"], d["g_bwd"], la_f, la_b, cfg.tau)
    first = None
    for _ in range(4):
        outs = [torch.full_like(d[n], float("nan")) for n in ("q", "k", "v", "q", "q")]
        vig.vig_bigla_bwd(d["q"], d["k"], d["v"], la_f, la_b, d["d_out"], *outs)
        torch.cuda.synchronize()
        got = [to_stored(o, "bf16") for o in outs]
        if first is None:
            first = got
        for a, b in zip(first, got):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("dk,dv", [(16, 32), (24, 48), (32, 64), (32, 48)])
@pytest.mark.parametrize("L", [16, 31, 32, 112, 127, 128, 129, 143, 144, 145, 208, 223, 224, 225, 256, 288, 289, 577])
def test_bf16_gradient_chunk_edges(oracle, dk, dv, L):
    """The tensor-core gradient at the edges of its tiles (16 tokens), of one chunk (128), of a pair of chunks (224) and of
    the chunks of longer sequences (96)."""
    cfg, x = random_problem(4500 + L, 2, 3, L, dk, dv, "bf16", gate_mean=0.5)
    got, ref = _run(oracle, cfg, x, synth.make_grad_input(cfg))
    _check(got, ref, "bf16")


@pytest.mark.parametrize("L", [60, 100, 200, 400])
@pytest.mark.parametrize("direction", ["g_fwd", "g_bwd"])
def test_bf16_gradient_out_of_range_unit_per_form(oracle, L, direction):
    """One unit with closed gates (log alpha = -40 over three tokens) in each form of the tensor-core gradient - one chunk,
    a pair, chunks through scratch: that unit alone takes the recurrence, and every gradient meets the bar."""
    cfg, x = random_problem(4600 + L, 2, 2, L, 24, 48, "bf16", gate_mean=1.0)
    g = synth.stored_to_f64(x[direction], "bf16").copy()
    g[1, 0, 20:23] = -640.0
    x[direction] = synth.store(g, "bf16")
    vig.vig_test_take_fallback_count()
    got, ref = _run(oracle, cfg, x, synth.make_grad_input(cfg))
    assert vig.vig_test_take_fallback_count() == 1
    _check(got, ref, "bf16")


@pytest.mark.parametrize("units,L", [(1, 1), (2, 5), (1, 9), (3, 63), (48, 196), (700, 37), (1, 511), (1, 512), (2, 1030)])
@pytest.mark.parametrize("dk,dv", [(32, 64), (24, 48), (13, 31), (70, 100)])
def test_f32_walks_in_segments(oracle, units, L, dk, dv):
    """fp32 forward and gradient where the walks change form: one segment, a ragged last one, eight of them, units enough to
    walk whole sequences, segments in blocks of their own (512 tokens and more); rows of whole pieces and odd ones."""
    if units * L * dk > 40000 * 32:
        dk, dv = min(dk, 32), min(dv, 64)
    cfg, x = random_problem(4700 + L, units, 1, L, dk, dv, "f32", gate_mean=0.5)
    got, ref = _run(oracle, cfg, x, synth.make_grad_input(cfg))
    _check(got, ref, "f32")
    la = [oracle_log_alpha(oracle, x[n], "f32", cfg.tau) for n in ("g_fwd", "g_bwd")]
    d = [to_device(a, "f32") for a in (x["q"], x["k"], x["v"], *la)]
    out = torch.full_like(d[2], float("nan"))
    vig.vig_bigla_fwd_f32(*d, out)
    torch.cuda.synchronize()
    f = lambda a: synth.stored_to_f64(a, "f32")
    assert rel_err(device_to_f64(out, "f32"), oracle.bigla_fwd(f(x["q"]), f(x["k"]), f(x["v"]), f(la[0]), f(la[1]), nthreads=4)) <= TOL["f32"]


@pytest.mark.parametrize("units,L", [(3, 100), (200, 196), (4, 700)])
def test_chain_of_dependent_launches_sees_what_the_last_one_wrote(units, L):
    """Gate preparation, forward (one launch: a block a unit, or a cluster) and gradient (one launch, or three) back to back on the
    same buffers, the contents changing from pass to pass: each kernel starts while the one before it, which writes its inputs, may
    still be running.  Forward passes of three launches: the test below."""
    rng = torch.Generator(device="cuda").manual_seed(L)
    mk = lambda d: torch.randn(1, units, L, d, generator=rng, device="cuda").bfloat16()
    sets = [dict(q=mk(24) * 24 ** -0.5, k=mk(24), v=mk(48), gf=mk(24), gb=mk(24), g=mk(48)) for _ in range(3)]
    now = {n: torch.empty_like(t) for n, t in sets[0].items()}
    la = [torch.empty_like(now["gf"]) for _ in range(2)]

    def step(keep):
        out = [torch.empty_like(now[n]) for n in ("v", "q", "k", "v", "gf", "gb")] if keep is None else keep
        vig.vig_gate_prep_bf16(now["gf"], now["gb"], la[0], la[1], 16.0)
        vig.vig_bigla_fwd_bf16(now["q"], now["k"], now["v"], la[0], la[1], out[0])
        vig.vig_bigla_bwd(now["q"], now["k"], now["v"], la[0], la[1], now["g"], *out[1:])
        return out

    alone = []
    for s in sets:
        for n in now:
            now[n].copy_(s[n])
        torch.cuda.synchronize()
        alone.append(step(None))
        torch.cuda.synchronize()
    outs = [[[torch.empty_like(t) for t in alone[0]] for _ in sets] for _ in range(8)]
    for rep in outs:
        for s, keep in zip(sets, rep):
            for n in now:
                now[n].copy_(s[n])
            step(keep)
    torch.cuda.synchronize()
    for rep in outs:
        for got, want in zip(rep, alone):
            assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(got, want))


@pytest.mark.parametrize("units,L,dk,dv", [(4, 1300, 24, 64), (9, 2100, 24, 32), (2, 4096, 32, 64), (3, 1200, 16, 48)])
def test_chain_of_chunked_calls_on_reused_buffers_and_scratch(units, L, dk, dv):
    """Forward from logits, forward from log gates and gradient in three launches each, back to back on the same buffers and the
    same scratch, the contents changing from pass to pass; in one of the passes a unit's gates are closed, so that its chunks are
    told to leave it to the walks.  The last of the three launches reads ahead of its own wait: nothing of the pass before may
    come through."""
    rng = torch.Generator(device="cuda").manual_seed(L)
    mk = lambda d: torch.randn(1, units, L, d, generator=rng, device="cuda").bfloat16()
    sets = [dict(q=mk(dk) * dk ** -0.5, k=mk(dk), v=mk(dv), gf=mk(dk), gb=mk(dk), g=mk(dv)) for _ in range(3)]
    sets[1]["gf"][0, 1, 700:703] = -640.0          # log alpha = -40 a token: outside the range of the factorised tiles
    now = {n: torch.empty_like(t) for n, t in sets[0].items()}
    la = [torch.empty_like(now["gf"]) for _ in range(2)]
    names = ("v", "v", "q", "k", "v", "gf", "gb")

    def counted(call, *a):
        before = vig.vig_kernel_launch_count()
        call(*a)
        assert vig.vig_kernel_launch_count() - before == 3

    def step(out):
        counted(vig.vig_bigla_fwd_gates_bf16, now["q"], now["k"], now["v"], now["gf"], now["gb"], out[0], 16.0)
        vig.vig_gate_prep_bf16(now["gf"], now["gb"], la[0], la[1], 16.0)
        counted(vig.vig_bigla_fwd_bf16, now["q"], now["k"], now["v"], la[0], la[1], out[1])
        counted(vig.vig_bigla_bwd, now["q"], now["k"], now["v"], la[0], la[1], now["g"], *out[2:])
        return out

    empty = lambda: [torch.empty_like(now[n]) for n in names]
    alone = []
    for s in sets:
        for n in now:
            now[n].copy_(s[n])
        torch.cuda.synchronize()
        vig.vig_test_take_fallback_count()
        alone.append(step(empty()))
        assert vig.vig_test_take_fallback_count() == (3 if s is sets[1] else 0)
    outs = [[empty() for _ in sets] for _ in range(6)]
    for rep in outs:
        for s, keep in zip(sets, rep):
            for n in now:
                now[n].copy_(s[n])
            step(keep)
    torch.cuda.synchronize()
    assert vig.vig_last_device_status() == 0
    for rep in outs:
        for got, want in zip(rep, alone):
            assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(got, want))


def _gradient_call(L):
    cfg, x = random_problem(4800 + L, 2, 2, L, 24, 48, "bf16", gate_mean=1.0)
    d = {n: to_device(a, "bf16") for n, a in x.items()}
    d["d_out"] = to_device(synth.make_grad_input(cfg), "bf16")
    la = [torch.empty_like(d["g_fwd"]) for _ in range(2)]
    vig.vig_gate_prep_bf16(d["g_fwd"], d["g_bwd"], *la, cfg.tau)

    def call():
        outs = [torch.full_like(d[n], 7.0) for n in ("q", "k", "v", "q", "q")]
        vig.vig_bigla_bwd(d["q"], d["k"], d["v"], *la, d["d_out"], *outs)
        torch.cuda.synchronize()
        return outs
    return call


@pytest.mark.parametrize("L", [60, 196, 400])
def test_gradient_whose_wait_expires_stores_nothing(L):
    """One chunk, a pair, chunks through scratch (where the first of three launches lets its wait run out, and the last must
    not go by what that did not write): the status word says so once, and the next call is as before."""
    call = _gradient_call(L)
    want = call()
    assert vig.vig_last_device_status() == 0
    vig.vig_test_expire_next_wait()
    assert all(bool((o == 7.0).all()) for o in call())
    assert vig.vig_last_device_status() == -7 and vig.vig_last_device_status() == 0
    assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(call(), want))


def test_pair_whose_exchange_expires_stores_no_gate_gradients():
    """The left chunk of a pair (112 of 196 tokens) without the right one's sums: its gate gradients stay unwritten."""
    call = _gradient_call(196)
    want = call()
    vig.vig_test_expire_next_exchange()
    got = call()
    assert vig.vig_last_device_status() == -7 and vig.vig_last_device_status() == 0
    same = lambda a, b: torch.equal(a.view(torch.int16), b.view(torch.int16))
    for a, b in zip(got[:3], want[:3]):
        assert same(a, b)
    for a, b in zip(got[3:], want[3:]):
        assert bool((a[:, :, :112] == 7.0).all()) and same(a[:, :, 112:].contiguous(), b[:, :, 112:].contiguous())


@pytest.mark.parametrize("units,L,dk,dv", [(1, 13, 4, 4), (3, 97, 12, 20), (12, 400, 24, 48), (2, 784, 32, 64), (2, 2047, 16, 32), (47, 61, 32, 64), (60, 30, 32, 32)])
def test_fp32_walks_of_few_and_of_more_units(oracle, units, L, dk, dv):
    """Sixteen warps a block where every block has an SM of its own, blocks with two columns a lane otherwise, ragged last segments;
    forward and gradient, the latter with dv in the same launch below 512 tokens."""
    cfg, x = random_problem(4100 + L, units, 1, L, dk, dv, "f32", gate_mean=1.0)
    la = [oracle_log_alpha(oracle, x[n], "f32", cfg.tau) for n in ("g_fwd", "g_bwd")]
    d = {n: to_device(a, "f32") for n, a in dict(q=x["q"], k=x["k"], v=x["v"], f=la[0], b=la[1]).items()}
    out = torch.empty_like(d["v"])
    vig.vig_bigla_fwd_f32(d["q"], d["k"], d["v"], d["f"], d["b"], out)
    assert rel_err(device_to_f64(out, "f32"), oracle_out(oracle, x["q"], x["k"], x["v"], la[0], la[1], "f32")) <= TOL["f32"]
    g = np.random.default_rng(L).standard_normal(x["v"].shape).astype(np.float32)
    grads = [torch.empty_like(d[n]) for n in ("q", "k", "v", "q", "q")]
    before = vig.vig_kernel_launch_count()
    vig.vig_bigla_bwd(d["q"], d["k"], d["v"], d["f"], d["b"], to_device(g, "f32"), *grads)
    assert (vig.vig_kernel_launch_count() - before == 1) == (L < 512)   # longer ones of few units: segments in blocks of their own
    f64 = lambda a: a.astype(np.float64)
    ref = oracle.bigla_bwd(f64(x["q"]), f64(x["k"]), f64(x["v"]), f64(la[0]), f64(la[1]), f64(g))
    for t, r in zip(grads, ref):
        assert rel_err(device_to_f64(t, "f32"), r) <= TOL["f32"]


@pytest.mark.parametrize("cpl,L,dk,dv,dtype", [(4, 61, 32, 64, "f32"), (4, 97, 16, 64, "f32"), (4, 30, 32, 32, "f32"), (4, 50, 24, 128, "f32"),
                                               (4, 45, 8, 64, "bf16"), (4, 33, 20, 28, "bf16"), (3, 61, 32, 64, "f32"), (3, 50, 16, 48, "f32"),
                                               (3, 41, 12, 20, "f32"), (3, 37, 28, 40, "bf16")])
def test_forward_walks_of_three_and_four_columns_a_lane(oracle, cpl, L, dk, dv, dtype):
    """As many units as give every SM one block at this width and more than one at any smaller, widths of whole slabs and ragged ones."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    slabs = lambda x: -(-dv // (8 * x))
    units = sms // slabs(cpl)
    assert units * slabs(cpl) <= sms and all(units * slabs(x) > sms for x in range(2, cpl))
    cfg, x = random_problem(4900 + L, units, 1, L, dk, dv, dtype, gate_mean=1.0)
    la = [oracle_log_alpha(oracle, x[n], dtype, cfg.tau) for n in ("g_fwd", "g_bwd")]
    d = [to_device(a, dtype) for a in (x["q"], x["k"], x["v"], *la)]
    out = torch.full_like(d[2], float("nan"))
    (vig.vig_bigla_fwd_f32 if dtype == "f32" else vig.vig_bigla_fwd_bf16)(*d, out)
    torch.cuda.synchronize()
    got = device_to_f64(out, dtype)
    assert np.isfinite(got).all()
    assert rel_err(got, oracle_out(oracle, x["q"], x["k"], x["v"], la[0], la[1], dtype)) <= TOL[dtype]


@pytest.mark.parametrize("L,dk,dv", [(6200, 32, 64), (6240, 32, 48), (9000, 24, 64), (10300, 24, 32)])
def test_gradient_fold_over_runs_of_more_chunks_than_it_keeps(oracle, L, dk, dv):
    """65 to 108 chunks of one unit: eight runs of nine to fourteen chunks, read twice, a last run of fewer, or sixteen runs."""
    cfg, x = random_problem(5000 + L, 1, 1, L, dk, dv, "bf16", gate_mean=2.0)
    got, ref = _run(oracle, cfg, x, synth.make_grad_input(cfg))
    _check(got, ref, "bf16")


@pytest.mark.parametrize("L,dk,dv", [(8300, 32, 64), (11600, 32, 64), (13000, 24, 64)])
def test_forward_fold_over_runs_of_more_chunks_than_it_keeps(oracle, L, dk, dv):
    """The same of the forward pass, from log gates and from logits: chunks of 128 tokens and fewer."""
    cfg, x = random_problem(5100 + L, 1, 1, L, dk, dv, "bf16", gate_mean=2.0)
    la = [oracle_log_alpha(oracle, x[n], "bf16", cfg.tau) for n in ("g_fwd", "g_bwd")]
    d = {n: to_device(a, "bf16") for n, a in dict(x, f=la[0], b=la[1]).items()}
    ref = oracle_out(oracle, x["q"], x["k"], x["v"], la[0], la[1], "bf16")
    for call in (lambda o: vig.vig_bigla_fwd_bf16(d["q"], d["k"], d["v"], d["f"], d["b"], o),
                 lambda o: vig.vig_bigla_fwd_gates_bf16(d["q"], d["k"], d["v"], d["g_fwd"], d["g_bwd"], o, cfg.tau)):
        out = torch.full_like(d["v"], float("nan"))
        before = vig.vig_kernel_launch_count()
        call(out)
        assert vig.vig_kernel_launch_count() - before == 3
        got = device_to_f64(out, "bf16")
        assert np.isfinite(got).all() and rel_err(got, ref) <= TOL["bf16"]
