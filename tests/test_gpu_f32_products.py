"""The float32 layer's expert products on the tensor cores, each against float64 products of the operands that the call left
in its workspace, at the edges of the kernel's tiles and chunks; and values that bfloat16 parts cannot hold."""
import math

import pytest
import torch

from paper_2101_03961_b200 import inputs as si
from paper_2101_03961_b200 import switch_moe as sm
from tests.gpu_helpers import TOL_F32
from tests.test_gpu_parity import _check_layer, _check_top2

pytestmark = pytest.mark.gpu


def _layer(T, d, f, E, cf, path, residual=False, seed=1, spoil=None, events=None):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(*shape):
        return torch.empty(shape, device="cuda").normal_(generator=g)

    t = {"x": normal(T, d), "dy": normal(T, d), "W_in": normal(E, d, f) * (0.1 / d) ** 0.5,
         "W_out": normal(E, f, d) * (0.1 / f) ** 0.5, "W_r": torch.zeros(d, E, device="cuda"), "noise": 2.0 * normal(T, E)}
    if spoil is not None:
        spoil(t)
    cfg = sm.make_config(T, d, f, E, cf, dtype=sm.F32, residual=residual, gemm_path=path)
    cfg.router_noise = t["noise"].data_ptr()                   # W_r = 0: the noise decides the routing, dx has no router term
    ws = sm.allocate_workspace(cfg)
    ws.fill_(0xFF)                                             # stale rows read as NaN
    for k in ("y", "dx"):
        t[k] = torch.empty_like(t["x"])
    for k in ("W_r", "W_in", "W_out"):
        t["d" + k] = torch.empty_like(t[k])
    aux = torch.empty(1, device="cuda")
    if events:
        events[0].record()
    sm.switch_moe_fwd(cfg, t["x"], t["W_r"], None, t["W_in"], t["W_out"], t["y"], aux, ws)
    sm.switch_moe_bwd(cfg, t["dy"], 1.0, t["x"], t["W_r"], t["W_in"], t["W_out"], t["y"], ws, t["dx"], t["dW_r"], t["dW_in"],
                      t["dW_out"])
    if events:
        events[1].record()
    sm.switch_moe_check_device_status(cfg, ws)
    C = sm.switch_moe_capacity(cfg)
    view = lambda region: sm.switch_moe_workspace_view(cfg, ws, region)  # noqa: E731
    for name, region, cols in (("X", sm.WS_XD, d), ("H", sm.WS_H, f), ("dY", sm.WS_DYD, d), ("dH", sm.WS_DH, f)):
        t[name] = view(region).view(torch.float32).view(E, C, cols)
    t["kept"] = view(sm.WS_KEPT).tolist()
    t["tokens"] = view(sm.WS_TOKEN_OF_SLOT).view(E, C).long()
    t["gate"] = view(sm.WS_GATE)
    return t


def _errors(t, residual):
    """Relative Frobenius error of each product, and the contraction lengths of the weight gradients."""
    num, den = {}, {}

    def add(name, got, want):
        num[name] = num.get(name, 0.0) + float(((got.double() - want) ** 2).sum())
        den[name] = den.get(name, 0.0) + float((want ** 2).sum())

    for e, n in enumerate(t["kept"]):
        x, h, dy, dh = (t[k][e, :n].double() for k in ("X", "H", "dY", "dH"))
        w_in, w_out, tok = t["W_in"][e].double(), t["W_out"][e].double(), t["tokens"][e, :n]
        add("gemm1", t["H"][e, :n], (x @ w_in).clamp(min=0))
        skip_y, skip_dx = (t["x"][tok].double(), t["dy"][tok].double()) if residual else (0.0, 0.0)
        add("gemm2", t["y"][tok], (h @ w_out) * t["gate"][tok].double()[:, None] + skip_y)
        add("dgrad2", t["dH"][e, :n], (dy @ w_out.T) * (h > 0))
        add("dgrad1", t["dx"][tok], dh @ w_in.T + skip_dx)
        add("wgrad2", t["dW_out"][e], h.T @ dy)
        add("wgrad1", t["dW_in"][e], x.T @ dh)
    return {k: math.sqrt(num[k] / den[k]) for k in num}


FIRST, SECOND, WEIGHTS = ("gemm1", "dgrad2"), ("gemm2", "dgrad1"), ("wgrad2", "wgrad1")
SHAPES = [                                 # and the products that are large enough for the tensor cores
    (1024, 128, 512, 4, 1.25, False, FIRST + SECOND + WEIGHTS),      # whole tiles of m, several tiles of tokens
    (4100, 72, 1000, 16, 1.25, True, FIRST + SECOND + WEIGHTS),      # remainders of m, of a chunk and of 16 tokens; the skip path
    (5000, 8, 3000, 8, 2.0, False, SECOND + WEIGHTS),                # eight rows of a tile, many chunks
    (3000, 520, 24, 60, 2.0, True, FIRST),                           # 24 rows of a tile, about 50 tokens per expert
    (4096, 512, 2048, 16, 1.0, False, FIRST + SECOND + WEIGHTS),     # a full capacity of 256
    (1500, 264, 1032, 50, 1.25, False, FIRST + SECOND + WEIGHTS),    # about 30 tokens per expert: a chunk, less and more
    (1100, 264, 1032, 50, 1.25, False, FIRST + SECOND),              # and 22
]


@pytest.mark.parametrize("T,d,f,E,cf,residual,parts", SHAPES)
def test_products_of_exact_parts(T, d, f, E, cf, residual, parts):
    """Bound: of n = ceil(K / 32) chunks each truncates two sums at the size of the chunk (2^-23 each; chunks are independent,
    together 4 2^-24 of the result), and the float32 sum over the chunks rounds n times at the size of a running sum of random
    terms (2^-24 sqrt(n / 2)); one more rounding for the gate and the skip path each.  Fused multiply-adds round K times, each
    by up to 2^-24 (2^-24 / sqrt(3) in the mean) of a running sum, together 0.41 sqrt(K) 2^-24.  The error also says which kernel
    a product went to: the same on both paths, or well below the chain's (from 60 steps on by more than a quarter; with the skip
    path the sum's own rounding is most of either)."""
    t = _layer(T, d, f, E, cf, sm.GEMM_DEFAULT, residual)
    errs = _errors(t, residual)
    fma = _errors(_layer(T, d, f, E, cf, sm.GEMM_SIMT, residual), residual)
    tokens = max(t["kept"])
    for name, K in (("gemm1", d), ("gemm2", f), ("dgrad2", d), ("dgrad1", f), ("wgrad2", tokens), ("wgrad1", tokens)):
        assert fma[name] <= 2.0 ** -24 * (2.0 + 0.5 * math.sqrt(K)), (name, fma)
        if name in parts:
            assert errs[name] <= 2.0 ** -24 * (6.0 + math.sqrt(math.ceil(K / 32) / 2.0)), (name, errs)
            assert errs[name] <= (0.95 if residual else 0.85) * fma[name], (name, errs, fma)
        else:
            assert abs(errs[name] - fma[name]) <= 0.02 * fma[name], (name, errs, fma)
    again = _layer(T, d, f, E, cf, sm.GEMM_DEFAULT, residual)
    for k in ("y", "dx", "dW_in", "dW_out"):
        assert torch.equal(t[k], again[k])


def test_weight_gradients_of_few_tokens():
    """Contractions of 1 to 39 tokens (one MMA step, one chunk, two): no less exact than a chain of fused multiply-adds.  One
    token: both round one product once, but of operands whose last bits differ between the paths (measured: up to 0.4%)."""
    E, d, f, T = 40, 512, 1024, 2000
    counts = list(range(1, E)) + [T - sum(range(E))]
    expert = torch.cat([torch.full((n,), e) for e, n in enumerate(counts)])
    expert = expert[torch.randperm(T, generator=torch.Generator().manual_seed(3))].cuda()

    def spoil(t):
        t["noise"].zero_()[torch.arange(T, device="cuda"), expert] = 4.0

    errs = []
    for path in (sm.GEMM_DEFAULT, sm.GEMM_SIMT):
        t = _layer(T, d, f, E, 40.0, path, seed=3, spoil=spoil)
        assert t["kept"] == counts
        errs.append({})
        for e, n in enumerate(counts):
            x, h, dy, dh = (t[k][e, :n].double() for k in ("X", "H", "dY", "dH"))
            for name, got, want in (("wgrad2", t["dW_out"][e], h.T @ dy), ("wgrad1", t["dW_in"][e], x.T @ dh)):
                errs[-1][name, n] = float((got.double() - want).norm() / want.norm())
    for k, fma in errs[1].items():
        assert errs[0][k] <= fma * (1.0 + (2.0 ** -6 if k[1] == 1 else 0.0)), (k, errs[0][k], fma)


@pytest.mark.parametrize("scale", [
    dict(x=-118, W_in=74, W_out=46, dy=-46), dict(dy=-118, W_out=74), dict(W_out=-118, W_in=33, dy=33),
    dict(W_in=-118, x=60, W_out=60, dy=-50), dict(x=-59, W_in=-59, W_out=60), dict(dy=-59, W_out=-59, W_in=60)],
    ids=["x", "dy", "W_out", "W_in", "H", "dH"])
def test_products_of_small_operands(scale):
    """Operands around 2^-118, subnormal ones among them, in every product that has such an operand: a power of two changes no
    rounding, so the bound of ordinary operands holds."""
    def spoil(t):
        for name, e in scale.items():
            t[name] *= 2.0 ** e

    shape = (2048, 128, 512, 8, 1.25)
    t = _layer(*shape, sm.GEMM_DEFAULT, spoil=spoil)
    errs, fma, tokens = _errors(t, False), _errors(_layer(*shape, sm.GEMM_SIMT, spoil=spoil), False), max(t["kept"])
    for name, K in (("gemm1", 128), ("gemm2", 512), ("dgrad2", 128), ("dgrad1", 512), ("wgrad2", tokens), ("wgrad1", tokens)):
        assert errs[name] <= 2.0 ** -24 * (6.0 + math.sqrt(math.ceil(K / 32) / 2.0)), (name, errs)
        assert errs[name] <= fma[name], (name, errs, fma)


def test_values_that_the_parts_cannot_hold():
    """Infinities, NaN and the largest floats come out as they do from fused multiply-adds, and stay where they belong."""
    def spoil(t):
        t["W_in"][0, 3, 5] = math.inf
        t["W_in"][1, 4, 6] = math.nan
        t["W_out"][2, 7, 9] = -math.inf
        t["W_out"][0, 100, 2] = 3.4028234e38
        t["W_in"][3, 10, 7] = 3.4e38
        t["dy"][17, 11] = math.inf
        t["dy"][18, 12] = math.nan

    a, b = (_layer(2048, 128, 512, 8, 1.25, path, residual=True, spoil=spoil) for path in (sm.GEMM_DEFAULT, sm.GEMM_SIMT))
    for k in ("y", "dx", "dW_in", "dW_out"):
        ra, rb = a[k], b[k]
        assert torch.equal(torch.isnan(ra), torch.isnan(rb)), k
        assert torch.equal(torch.isposinf(ra), torch.isposinf(rb)) and torch.equal(torch.isneginf(ra), torch.isneginf(rb)), k
        fin = torch.isfinite(rb) & (rb.abs() < 1e30)
        assert float((ra[fin] - rb[fin]).norm()) <= 1e-5 * float(rb[fin].norm()), k


def test_a_value_that_is_not_finite_changes_no_other_result():
    """Tokens that share a tile with a bad one, and rows of a weight gradient beside a bad one, keep their bits."""
    def spoil(t):
        t["dy"][17, 11] = math.inf
        t["dy"][18, 12] = math.nan
        t["W_in"][2, 5, 40] = math.inf

    shape = (2048, 128, 512, 8, 1.25, sm.GEMM_DEFAULT)
    clean, bad = _layer(*shape), _layer(*shape, spoil=spoil)
    assert clean["kept"] == bad["kept"] and torch.equal(clean["tokens"], bad["tokens"])
    for k in ("H", "dH"):                                      # rows of the other tokens, and the other hidden units
        for e, n in enumerate(clean["kept"]):
            a, b = clean[k][e, :n], bad[k][e, :n]
            other = (clean["tokens"][e, :n] != 17) & (clean["tokens"][e, :n] != 18)
            units = torch.arange(a.shape[1], device="cuda") != (40 if e == 2 else -1)
            assert torch.equal(a[other][:, units], b[other][:, units]), (k, e)
    tokens = torch.ones(2048, dtype=torch.bool, device="cuda")
    tokens[17] = tokens[18] = False
    tokens[clean["tokens"][2, :clean["kept"][2]]] = False      # every token of the expert with the bad weight
    for k in ("y", "dx"):
        assert torch.equal(clean[k][tokens], bad[k][tokens]), k
    for k in ("dW_in", "dW_out"):
        for e in (0, 1, 3):
            fin = torch.isfinite(bad[k][e])
            assert fin.float().mean() > 0.4 and torch.equal(clean[k][e][fin], bad[k][e][fin]), (k, e)


@pytest.mark.parametrize("spoiled", ["dy", "W_in", "W_out"])
def test_time_of_results_that_are_not_finite(spoiled):
    """Every element of an operand NaN: all of up to four products are formed again, which takes a bounded multiple of the fused
    multiply-add kernels' time (measured: 3 to 10.5 for a whole step)."""
    def spoil(t):
        t[spoiled].fill_(math.nan)

    best = {}
    for path in (sm.GEMM_DEFAULT, sm.GEMM_SIMT):
        start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        times = []
        for _ in range(3):
            torch.cuda.synchronize()
            t = _layer(8192, 256, 1024, 4, 1.25, path, spoil=spoil, events=(start, end))
            times.append(start.elapsed_time(end))
        best[path] = min(times)
    assert best[sm.GEMM_DEFAULT] <= 20.0 * best[sm.GEMM_SIMT], best


def _call_times(T, d, f, E, geglu):
    """Median times (us) of a forward pass and of a step on the default path and on the FMA kernels, four calls in a row."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1)

    def normal(*shape):
        return torch.empty(shape, device="cuda").normal_(generator=g)

    x, dy, W_r = normal(T, d), normal(T, d), normal(d, E) * (0.1 / d) ** 0.5
    W_in, W_out = normal(E, d, 2 * f if geglu else f) * (0.1 / d) ** 0.5, normal(E, f, d) * (0.1 / f) ** 0.5
    cfg = sm.make_config(T, d, f, E, 1.25, dtype=sm.F32, geglu=geglu)
    ws, aux = sm.allocate_workspace(cfg), torch.empty(1, device="cuda")
    y, dx, dW_r, dW_in, dW_out = (torch.empty_like(t) for t in (x, x, W_r, W_in, W_out))

    def forward():
        sm.switch_moe_fwd(cfg, x, W_r, None, W_in, W_out, y, aux, ws)

    def step():
        forward()
        sm.switch_moe_bwd(cfg, dy, 1.0, x, W_r, W_in, W_out, y, ws, dx, dW_r, dW_in, dW_out)

    times = {}
    for _ in range(9):
        for cfg.gemm_path in (sm.GEMM_DEFAULT, sm.GEMM_SIMT):
            for call in (step, forward):
                call()
                start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                torch.cuda.synchronize()
                start.record()
                for _ in range(4):
                    call()
                end.record()
                torch.cuda.synchronize()
                times.setdefault((call.__name__, cfg.gemm_path), []).append(250.0 * start.elapsed_time(end))
        step()
    sm.switch_moe_check_device_status(cfg, ws)
    return {k: sorted(v)[4] for k, v in times.items()}


@pytest.mark.parametrize("T,d,f,E,geglu", [
    (160, 120, 3744, 3, True),             # few long rows to gate behind the products
    (9651, 8, 2120, 5, False),             # short contractions: GEMM1
    (23182, 1144, 8, 35, False),           # and GEMM2, dgrad1
    (22440, 120, 32, 44, False),           # narrow outputs
    (27995, 64, 104, 55, False),           # half a tile wide
    (5650, 72, 96, 226, False),            # 25 tokens per expert and little else
    (13764, 16, 472, 2, True),             # weight gradients of few tiles
    (600, 232, 1160, 150, False),          # and of few tokens
])
def test_calls_are_no_slower_than_with_fused_multiply_adds(T, d, f, E, geglu):
    """Shapes at which the tensor cores have little to win or the FMA kernels much to lose: 8% for the clock and the timing."""
    t = _call_times(T, d, f, E, geglu)
    for call in ("forward", "step"):
        assert t[call, sm.GEMM_DEFAULT] <= 1.08 * t[call, sm.GEMM_SIMT] + 1.0, t


@pytest.mark.parametrize("kw", [
    dict(geglu=True), dict(geglu=True, dropout=0.3, residual=True), dict(dropout=0.3), dict(dropout=0.3, noise_eps=0.3),
    dict(reroute=True), dict(reroute=True, reroute_stages=3, geglu=True), dict(groups=2, residual=True), dict(jitter_eps=0.2)],
    ids=lambda kw: "-".join(kw))
def test_options_on_tensor_core_products_match_oracle(kw):
    """Every product on the tensor cores (256 tokens per expert, f not a multiple of a tile), checked like every other layer."""
    _check_layer(si.SwitchConfig("f32_options", 2048, 128, 352, 8, 1.0, bias_std=0.5, dtype=si.DTYPE_F32), sm.GEMM_DEFAULT,
                 TOL_F32, d_aux=0.7, **kw)


@pytest.mark.parametrize("residual", [False, True])
def test_top2_on_tensor_core_products_matches_oracle(residual):
    _check_top2(si.SwitchConfig("f32_top2", 2048, 128, 352, 8, 1.0, bias_std=0.5, dtype=si.DTYPE_F32), sm.GEMM_DEFAULT, TOL_F32,
                residual=residual, expect_mix=False)
