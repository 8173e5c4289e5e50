"""GPU parity of each hot-path step, called through the C ABI, against the oracle.

Sizes span several 128-row tiles with ragged tails.  16-bit outputs compare at
|err| <= 1e-2 + 1e-2 |ref| against the exact fp64 result of the same inputs,
fp32 outputs at 1e-4 + 1e-4 |ref|; integer outputs compare exactly.
"""
import json
import os

import numpy as np
import pytest
import torch

import oracle
import synth
from tests.helpers import at_16, check_close, cuda, host, i32, tdtype, to_dev

pytestmark = pytest.mark.gpu

S = pytest.importorskip("paper_2607_14557_gb300.seer")
GOLDEN = os.path.join(os.path.dirname(__file__), "golden")


@pytest.fixture(autouse=True)
def _device_clean():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    assert S.seer_check_device() == 0


def _rng(seed):
    return np.random.default_rng(seed)


def _store(a, dt):
    """Values representable in storage type dt (f16 via torch's converter)."""
    if dt == "f16":
        return torch.from_numpy(np.asarray(a, dtype=np.float32)).to(torch.float16).float().numpy()
    return synth.round_storage(a, dt)


# ------------------------------------------------------------------ linear (S6, S8, S11)
@pytest.mark.parametrize("M,N,K", [(300, 512, 256), (128, 256, 64), (1, 256, 128), (777, 768, 512), (129, 256, 4096)])
@pytest.mark.parametrize("op,res,out", [("bf16", None, "bf16"), ("bf16", "bf16", "bf16"), ("f16", "bf16", "f16"),
                                        ("f16", "f16", "bf16")])
def test_linear_16bit(M, N, K, op, res, out):
    rng = _rng(M + N + K)
    a, w = _store(rng.standard_normal((M, K)), op), _store(0.05 * rng.standard_normal((N, K)), op)
    r = _store(rng.standard_normal((M, N)), res) if res else None
    ref = a.astype(np.float64) @ w.astype(np.float64).T + (r if res else 0.0)
    c = torch.full((M, N), float("nan"), dtype=tdtype(out), device=cuda())
    S.seer_linear(to_dev(a, op), to_dev(w, op), op, to_dev(r, res) if res else None, res or out, c, out, M, None, N, K)
    check_close(host(c), ref, "bf16", f"linear {M}x{N}x{K} {op}/{res}/{out}")


def test_linear_device_row_count_leaves_tail_untouched():
    rng = _rng(5)
    M_cap, M, N, K = 512, 333, 256, 128
    a, w = _store(rng.standard_normal((M_cap, K)), "f16"), _store(0.05 * rng.standard_normal((N, K)), "f16")
    c = torch.full((M_cap, N), 7.0, dtype=torch.float16, device=cuda())
    S.seer_linear(to_dev(a, "f16"), to_dev(w, "f16"), "f16", None, "f16", c, "f16", M_cap, i32([M]), N, K)
    out = host(c)
    check_close(out[:M], a[:M].astype(np.float64) @ w.astype(np.float64).T, "bf16", "linear M_dev")
    assert (out[M:] == 7.0).all()   # zero work past the device row count


def test_linear_f32():
    rng = _rng(6)
    M, N, K = 70, 52, 36
    a, w, r = (x.astype(np.float32) for x in (rng.standard_normal((M, K)), rng.standard_normal((N, K)),
                                              rng.standard_normal((M, N))))
    c = torch.empty((M, N), dtype=torch.float32, device=cuda())
    S.seer_linear(to_dev(a, "f32"), to_dev(w, "f32"), "f32", to_dev(r, "f32"), "f32", c, "f32", M, None, N, K)
    check_close(host(c), a.astype(np.float64) @ w.astype(np.float64).T + r, "f32", "linear f32")


@pytest.mark.parametrize("M,N,K", [
    (1, 256, 64), (127, 4096, 128), (128, 256, 4096),              # one row tile: one SM per tile, narrow tiles
    (129, 256, 192), (255, 2304, 128), (257, 512, 64),             # pairs; a last pair with one row tile
    (700, 4096, 256), (1100, 12288, 64), (842, 4096, 4096),        # last column tile narrower than the others
    (2600, 4096, 128), (4500, 2304, 64)])                          # several waves, both raster orders
@pytest.mark.parametrize("res", [False, True])
def test_linear_tile_choices(M, N, K, res):
    """Every tile shape the GEMM's plan picks (one SM or a pair, 32 .. 256 columns):
    small integers, so every product and sum is exact in fp32 (|sum| <= 4 K < 2^24)
    and the result is the fp64 one rounded once to bf16."""
    rng = _rng(M + N + K)
    a, w = rng.integers(-2, 3, (M, K)).astype(np.float32), rng.integers(-2, 3, (N, K)).astype(np.float32)
    r = rng.integers(-8, 9, (M, N)).astype(np.float32)
    ad, wd, rd = to_dev(a, "f16"), to_dev(w, "f16"), to_dev(r, "f16")
    c = torch.full((M + 1, N), float("nan"), dtype=torch.bfloat16, device=cuda())
    S.seer_linear(ad, wd, "f16", rd if res else None, "f16", c, "bf16", M, None, N, K)
    ref = ad.double() @ wd.double().T + (rd.double() if res else 0.0)
    assert torch.equal(c[:M], ref.to(torch.bfloat16))
    assert torch.isnan(c[M]).all()                                  # nothing past the last row


@pytest.mark.parametrize("M", [1, 45, 300])                          # rows stored lane by lane, alone and after full slabs
def test_gemm_outputs_on_16_byte_boundaries(M):
    """Operands, residual and outputs need 16-byte alignment, not 32: the same bits as
    from buffers on larger boundaries."""
    N, K = 256, 128
    g = torch.Generator(device="cuda").manual_seed(M)
    r = lambda *s: torch.randn(s, generator=g, device="cuda").half()
    a, w, w2, res = r(M, K), 0.1 * r(N, K), 0.1 * r(N, K), r(M, N)
    out = []
    for place in (lambda t: t, at_16):
        c = [place(torch.zeros((M, N), dtype=torch.float16, device="cuda")) for _ in range(3)]
        a_, w_, w2_, res_ = place(a), place(w), place(w2), place(res)
        S.seer_linear(a_, w_, "f16", None, "f16", c[0], "f16", M, None, N, K)
        S.seer_linear(a_, w_, "f16", res_, "f16", c[1], "f16", M, None, N, K)
        S.seer_swiglu(a_, w_, w2_, "f16", c[2], "f16", M, None, N, K)
        out.append(c)
    assert all(torch.equal(p, q) for p, q in zip(*out))


@pytest.mark.parametrize("M,N,K", [(127, 1024, 12288), (300, 4096, 12288)])
def test_linear_repeats_bit_for_bit_over_a_long_k_loop(M, N, K):
    """Each tile runs the operand ring around dozens of times; called back to back on
    narrow tiles (two k-blocks a stage) and wide ones, every call stores the same bits."""
    rng = _rng(M + N)
    a, w = (to_dev(rng.integers(-2, 3, s).astype(np.float32), "f16") for s in ((M, K), (N, K)))
    ref = (a.double() @ w.double().T).to(torch.bfloat16)              # |sums| <= 4 K < 2^24: exact in fp32
    out = torch.full((100, M, N), float("nan"), dtype=torch.bfloat16, device=cuda())
    for c in out:
        S.seer_linear(a, w, "f16", None, "f16", c, "bf16", M, None, N, K)
    assert (out == ref).all()


@pytest.mark.parametrize("M_cap,N,K", [(100, 256, 64), (640, 12288, 128), (640, 4096, 192), (900, 4096, 64), (1049, 4096, 128),
                                       (1500, 4096, 64), (1500, 12288, 64), (1500, 4096, 1024)])
@pytest.mark.parametrize("fill", [0.0, 0.01, 0.25, 0.4, 0.5, 0.78, 0.8, 0.82, 1.0])
def test_linear_second_tile_choice_for_fewer_device_rows(M_cap, N, K, fill):
    """Calls whose device row count is below the size they are planned for use the
    plan's second tile width up to four fifths of the row tiles: exact on integers,
    rows past the count untouched."""
    M = int(M_cap * fill)
    rng = _rng(M_cap + N + K)
    a, w = (to_dev(rng.integers(-2, 3, s).astype(np.float32), "f16") for s in ((M_cap, K), (N, K)))
    r = to_dev(rng.integers(-8, 9, (M_cap, N)).astype(np.float32), "f16")
    c = torch.full((M_cap, N), float("nan"), dtype=torch.bfloat16, device=cuda())
    S.seer_linear(a, w, "f16", r, "f16", c, "bf16", M_cap, i32([M]), N, K)
    assert torch.equal(c[:M], (a[:M].double() @ w.double().T + r[:M].double()).to(torch.bfloat16))
    assert torch.isnan(c[M:]).all()


@pytest.mark.parametrize("M,F,K", [(1, 128, 64), (127, 1280, 64), (200, 384, 128), (300, 12288, 64), (900, 1408, 64)])
def test_swiglu_tile_choices(M, F, K):
    """Gate/up tiles of every width, the last one narrower than the others."""
    rng = _rng(M + F + K)
    a = _store(rng.standard_normal((M, K)), "f16")
    wg, wu = (_store(0.2 * rng.standard_normal((F, K)), "f16") for _ in range(2))
    act = torch.full((M + 1, F), float("nan"), dtype=torch.float16, device=cuda())
    S.seer_swiglu(to_dev(a, "f16"), to_dev(wg, "f16"), to_dev(wu, "f16"), "f16", act, "f16", M, None, F, K)
    g, u = (a.astype(np.float64) @ w.astype(np.float64).T for w in (wg, wu))
    check_close(host(act[:M]), g / (1.0 + np.exp(-g)) * u, "bf16", "swiglu")
    assert torch.isnan(act[M]).all()


@pytest.mark.parametrize("M,N,K", [(1, 4, 4), (31, 33, 17), (33, 96, 768), (65, 260, 35), (130, 3000, 20),
                                   (300, 1000, 100), (1300, 1030, 36), (2000, 2050, 6)])
@pytest.mark.parametrize("offset", [0, 1])
def test_linear_f32_tile_choices(M, N, K, offset):
    """Every fp32 tile size at ragged edges, 16-byte copies and (odd K or operands
    one float past a 16-byte boundary) 4-byte copies; small integers: exact."""
    rng = _rng(M + N + K)
    a, w, r = (torch.from_numpy(rng.integers(-4, 5, (m, n)).astype(np.float32)).to(cuda())
               for m, n in ((M, K), (N, K), (M, N)))
    off = lambda t: torch.cat([t.new_zeros(offset), t.flatten()])[offset:].view(t.shape)
    c = torch.full((M + 1, N), float("nan"), dtype=torch.float32, device=cuda())
    S.seer_linear(off(a), off(w), "f32", r, "f32", c, "f32", M, None, N, K)
    assert torch.equal(c[:M], (a.double() @ w.double().T + r.double()).float())
    assert torch.isnan(c[M]).all()


@pytest.mark.parametrize("M,F,K", [(9, 36, 20), (70, 130, 33), (200, 1540, 12), (900, 2052, 20), (1300, 2052, 20)])
def test_swiglu_f32_tile_choices(M, F, K):
    """fp32 gate/up tiles of every size with the count hook; activations against
    fp64, counts against the kernel's own activations."""
    rng = _rng(M + F + K)
    a, wg, wu = (rng.standard_normal(s).astype(np.float32) * c for s, c in (((M, K), 1.0), ((F, K), 0.3), ((F, K), 0.3)))
    act = torch.full((M + 1, F), float("nan"), dtype=torch.float32, device=cuda())
    counts = torch.zeros(M, dtype=torch.int32, device=cuda())
    S.seer_swiglu(to_dev(a, "f32"), to_dev(wg, "f32"), to_dev(wu, "f32"), "f32", act, "f32", M, None, F, K, i32([0, M]), 1,
                  i32([0]), M, 0.05, counts)
    g, u = (a.astype(np.float64) @ w.astype(np.float64).T for w in (wg, wu))
    check_close(host(act[:M]), g / (1.0 + np.exp(-g)) * u, "f32", "swiglu f32")
    assert torch.isnan(act[M]).all()
    eps = torch.tensor(0.05, dtype=torch.float32, device=cuda())
    assert torch.equal(counts, (act[:M].abs() < eps).sum(1, dtype=torch.int32))


@pytest.mark.parametrize("H,dh,lens,kv", [
    (2, 64, [1, 15, 16, 17], [1, 15, 9, 17]),                       # 16-row tiles, 256 threads
    (3, 4, [5, 64, 65], [5, 64, 1]), (2, 28, [70, 3, 129], [70, 2, 128]), (1, 100, [200], [130]), (2, 128, [131], [131]),
    (16, 64, [150, 31], [97, 31]), (12, 128, [200], [129]),
    (24, 20, [400], [390]),                                         # 16-row tiles, 128 threads
    (32, 32, [400, 63, 257], [399, 63, 64]),                        # 32-row tiles
    (40, 128, [300, 129, 64], [300, 65, 64]), (40, 12, [500, 33], [461, 33])])
@pytest.mark.parametrize("offset", [0, 1])
def test_attention_f32_tile_choices(H, dh, lens, kv, offset):
    """fp32 attention at the edges of its query and key tiles and head widths, rows
    16-byte aligned and not; keys past kv_len hold NaN and must not be read."""
    D, T = H * dh, sum(lens)
    rng = _rng(H + dh + T)
    x = rng.standard_normal((T, 3 * D)).astype(np.float32)
    cu = np.concatenate([[0], np.cumsum(lens)])
    dirty = x.copy()
    for a, b, k in zip(cu[:-1], cu[1:], kv):
        dirty[a + k:b, D:] = np.nan
    buf = torch.from_numpy(np.concatenate([np.zeros(offset, np.float32), dirty.ravel()])).to(cuda())
    o = torch.full((T + 1, D), float("nan"), dtype=torch.float32, device=cuda())
    S.seer_attention(buf[offset:], o, "f32", i32(cu), i32(kv), len(lens), T, H, dh)
    ref = np.concatenate([oracle.attention(*(x[a:a + n, c * D:(c + 1) * D].astype(np.float64)
                                             for c, n in ((0, b - a), (1, k), (2, k))), H)
                          for a, b, k in zip(cu[:-1], cu[1:], kv)])
    check_close(host(o[:T]), ref, "f32", "attention f32")
    assert torch.isnan(o[T]).all()


@pytest.mark.parametrize("H,dh,T", [(2, 128, 1000), (8, 64, 353), (40, 64, 400), (4, 32, 121)])
def test_attention_f32_error_at_large_scores(H, dh, T):
    """Scores of magnitude ~9 (up to ~45): a score summed in blocks is off by about sqrt(7)
    roundings of 2^-24 / sqrt(3) of it, 9e-8 x 9 = 8e-7 in the exponent and less in a row's
    result, where its keys' errors average out; one chain over the head's dims is off by
    three times as much at 128 dims (measured 1.8e-6, in blocks 0.6e-6)."""
    D = H * dh
    g = torch.Generator(device="cuda").manual_seed(T)
    qkv = torch.randn((T, 3 * D), generator=g, device="cuda")
    qkv[:, :2 * D] *= 3.0
    o = torch.empty((T, D), device="cuda")
    S.seer_attention(qkv, o, "f32", i32([0, T]), None, 1, T, H, dh)
    q, k, v = (t.view(T, H, dh).transpose(0, 1) for t in qkv.double().split(D, 1))
    ref = (torch.softmax(q @ k.transpose(1, 2) / dh ** 0.5, -1) @ v).transpose(0, 1).reshape(T, D)
    assert ((o.double() - ref).norm() / ref.norm()).item() < 8e-7


# ------------------------------------------------------------------ SwiGLU + count hook (S10, S1)
@pytest.mark.parametrize("op", ["bf16", "f16"])
def test_swiglu_counts_at_the_threshold_follow_the_ieee_quotient(op):
    """Every operand is a dyadic number and every weight row one power of two, so
    both GEMM paths form the same g and u exactly; with eps set to values of the
    fp32 path's own activations (ties, and g < -87 where the fast quotient may be
    0) the 16-bit path's counts must equal the fp32 path's."""
    rng = _rng(9)
    M, F, K, B, N = 200, 256, 64, 1, 200
    a = rng.integers(-96, 97, (M, K)).astype(np.float32) / 2
    a[:, 0], a[:, 1] = -88.0, -100.0
    one = lambda: np.eye(K, dtype=np.float32)[rng.integers(0, K, F)] * 2.0 ** rng.integers(-6, 2, F)[:, None]
    wg, wu = one(), one()
    wg[:2] = np.eye(K, dtype=np.float32)[:2]
    cu, rs = i32([0, M]), i32([0])

    def counts(dt, eps):
        act = torch.empty((M, F), dtype=tdtype(dt), device=cuda())
        c = torch.zeros(B * N, dtype=torch.int32, device=cuda())
        S.seer_swiglu(to_dev(a, dt), to_dev(wg, dt), to_dev(wu, dt), dt, act, dt, M, None, F, K, cu, B, rs, N, eps, c)
        return act, c.cpu().numpy()

    act, _ = counts("f32", 1.0)
    values = np.unique(np.abs(act.cpu().numpy()))
    for eps in [0.0, *rng.choice(values[(values > 0) & (values < 6e4)], 12), float(values[values > 0].min())]:
        np.testing.assert_array_equal(counts(op, float(eps))[1], counts("f32", float(eps))[1], err_msg=f"eps={eps}")


@pytest.mark.parametrize("op,act,up", [("bf16", "bf16", 3.0), ("f16", "bf16", 3.0), ("bf16", "f16", 2.0 ** 116),
                                      ("f16", "f16", 3.0)])
def test_swiglu_stores_what_the_ieee_quotient_gives_at_very_negative_gates(op, act, up):
    """Gates of -88 and -87.5, whose approximate quotient is 0: the fp32 path's activation
    (of about -5e-37 times u) rounded once to the output's type, nonzero where that type
    or a large u can show it; gates of 1 in the same chunk of columns stay right."""
    M, F, K = 130, 128, 64
    a, wg, wu = (np.zeros(s, dtype=np.float32) for s in ((M, K), (F, K), (F, K)))
    a[:, 0], a[:, 1], a[:, 2] = -88.0, -87.5, 1.0
    wg[np.arange(F), np.arange(F) % 3] = 1.0
    wu[:, 2] = up
    out = {}
    for dt, ot in (("f32", "f32"), (op, act)):
        o = torch.empty((M, F), dtype=tdtype(ot), device=cuda())
        S.seer_swiglu(to_dev(a, dt), to_dev(wg, dt), to_dev(wu, dt), dt, o, ot, M, None, F, K)
        out[ot] = o
    if (op, act) == ("bf16", "f16"):                                  # silu(1) * 2^116 is beyond f16, and recorded
        assert S.seer_check_device() == 6
    want, low = out["f32"].to(tdtype(act)), np.arange(F) % 3 < 2
    assert torch.equal(out[act][:, low], want[:, low])
    assert (out[act][:, low] != 0).all() == (act == "bf16" or op == "bf16")
    ref, got = out["f32"][:, ~low].double(), out[act][:, ~low].double()
    assert ((got - ref).abs() <= 1e-2 * ref.abs()).all() or act == "f16" and op == "bf16"


@pytest.mark.parametrize("op", ["bf16", "f16", "f32"])
def test_swiglu_with_count_hook(op):
    rng = _rng(7)
    M, F, K = 400, 384, 256
    x = _store(rng.standard_normal((M, K)), op)
    wg = _store(0.02 * rng.standard_normal((F, K)), op)
    wu = _store(0.02 * rng.standard_normal((F, K)), op)
    cu = np.array([0, 150, 290, 400])
    resp = np.array([100, 200, 350])
    Nw, eps = 64, 3e-4
    ref_act = oracle.swiglu_activation(x, wg, wu)
    ref_cnt = np.zeros((3, Nw), dtype=np.int64)
    for b in range(3):
        for t in range(Nw):
            r = resp[b] + t
            if r < cu[b + 1]:
                ref_cnt[b, t] = oracle.sparsity_counts(x[r:r + 1], wg, wu, eps)[0]
    act = torch.empty((M, F), dtype=tdtype(op), device=cuda())
    counts = torch.full((3 * Nw,), -1, dtype=torch.int32, device=cuda())
    S.seer_swiglu(to_dev(x, op), to_dev(wg, op), to_dev(wu, op), op, act, op, M, None, F, K, i32(cu), 3,
                  i32(resp), Nw, eps, counts)
    check_close(host(act), ref_act, "f32" if op == "f32" else "bf16", "swiglu act")
    got = counts.cpu().numpy().reshape(3, Nw)
    assert np.abs(got - ref_cnt).max() <= 0.005 * F
    assert ref_cnt.sum() > 0 and np.mean(got == ref_cnt) > 0.9


# ------------------------------------------------------------------ RMSNorm (S5, S9)
# 16-bit rows up to 4096 wide run the register-resident kernel (4, 8 or 16 vectors
# per lane, ragged widths masked); wider rows and fp32 the streaming one
@pytest.mark.parametrize("x_dt,y_dt,d", [("bf16", "f16", 4096), ("f16", "f16", 256), ("bf16", "bf16", 256),
                                         ("f32", "f32", 264), ("bf16", "f16", 1024), ("bf16", "f16", 3072),
                                         ("f16", "f16", 264), ("bf16", "f16", 8192)])
def test_rmsnorm(x_dt, y_dt, d):
    rng = _rng(8)
    M = 333
    x = _store(3 * rng.standard_normal((M, d)), x_dt)
    g = _store(1 + 0.1 * rng.standard_normal(d), y_dt)
    y = torch.empty((M, d), dtype=tdtype(y_dt), device=cuda())
    S.seer_rmsnorm(to_dev(x, x_dt), x_dt, to_dev(g, y_dt), y, y_dt, M, None, d, 1e-5)
    check_close(host(y), oracle.rmsnorm(x, g, 1e-5), "f32" if y_dt == "f32" else "bf16", "rmsnorm")


def test_convert_bf16_to_f16_is_exact_in_range():
    rng = _rng(9)
    v = _store(rng.standard_normal(4096) * np.exp(rng.uniform(-9, 9, 4096)), "bf16")
    src = to_dev(v, "bf16")
    dst = torch.empty(4096, dtype=torch.float16, device=cuda())
    S.seer_convert(src, "bf16", dst, "f16", 4096)
    got = host(dst)
    normal = (np.abs(v) >= 2.0 ** -14) & (np.abs(v) < 65504)
    np.testing.assert_array_equal(got[normal], v[normal])


# ------------------------------------------------------------------ attention (S7)
def _attention_case(dt, H, dh, lens, kv, scale, seed, structured=False):
    rng = _rng(seed)
    D = H * dh
    cu = np.concatenate([[0], np.cumsum(lens)])
    T = int(cu[-1])
    T_cap = T + 37
    qkv = scale * rng.standard_normal((T_cap, 3 * D))
    if structured:
        for b in range(len(lens)):
            j = np.arange(lens[b])
            for h in range(H):
                qkv[cu[b]:cu[b + 1], h * dh] = 18.0
                qkv[cu[b]:cu[b + 1], h * dh + 1:(h + 1) * dh] *= 0.1
                qkv[cu[b]:cu[b + 1], D + h * dh] = j / 16.0
    qkv = _store(qkv, dt)
    ref = np.full((T, D), np.nan)
    for b in range(len(lens)):
        s0, s1 = cu[b], cu[b + 1]
        ref[s0:s1] = oracle.attention(qkv[s0:s1, :D], qkv[s0:s0 + kv[b], D:2 * D], qkv[s0:s0 + kv[b], 2 * D:], H)
    out = torch.full((T_cap, D), 3.0, dtype=tdtype(dt), device=cuda())
    ws_bytes = (H * ((T_cap + 127) // 128 + len(lens)) * 16) + 4096
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=cuda())
    S.seer_attention(to_dev(qkv, dt), out, dt, i32(cu), i32(kv), len(lens), T_cap, H, dh, ws, ws_bytes)
    got = host(out)
    check_close(got[:T], ref, "f32" if dt == "f32" else "bf16", f"attention lens={lens}")
    assert (got[T:] == 3.0).all()


@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("scale", [1.0, 2.0])
def test_attention_16bit_varlen(dt, scale):
    lens = [1, 127, 128, 129, 300, 517, 64]
    kv = [1, 127, 128, 129, 260, 517, 40]     # two segments with padded (masked) key tails
    _attention_case(dt, 2, 128, lens, kv, scale, 11)


@pytest.mark.parametrize("dt", ["f16", "bf16"])
def test_attention_growing_max_forces_rescale(dt):
    # logits grow by ~0.1 per key, so the running max rises by ~18 (log2 units)
    # from one 128-key tile to the next: every tile takes the O-rescale branch
    lens = [517, 300]
    _attention_case(dt, 2, 128, lens, lens, 1.0, 15, structured=True)


@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("H,lens,kv", [
    (4, [1700], [1700]), (3, [2500, 700], [2401, 700]),                        # keys of a unit over 2 CTAs
    (2, [4200], [4133]), (1, [3000], [3000]), (1, [4000, 300], [3900, 77]),    # over 4, some without keys
    (1, [3700], [129])])
def test_attention_split_keys(dt, H, lens, kv):
    _attention_case(dt, H, 128, lens, kv, 1.0, 17)


@pytest.mark.parametrize("dt", ["f16", "bf16"])
def test_attention_split_keys_with_infinite_scores(dt):
    """Shares (and first tiles of shares) whose every score is -inf add nothing: the
    result is the attention over the finite keys."""
    n, keep = 3000, [*range(0, 700), *range(1000, 1300)]          # 4 shares of 6 tiles; two without a finite score
    g = torch.Generator(device="cuda").manual_seed(3)
    qkv = torch.randn((n, 3 * 128), generator=g, device="cuda").to(tdtype(dt))
    qkv[:, 0] = 1.0
    dead = torch.ones(n, dtype=torch.bool, device="cuda")
    dead[keep] = False
    qkv[dead, 128] = float("-inf")
    out = torch.empty((n, 128), dtype=qkv.dtype, device="cuda")
    ws = torch.empty(1 << 16, dtype=torch.uint8, device="cuda")
    S.seer_attention(qkv, out, dt, i32([0, n]), None, 1, n, 1, 128, ws, 1 << 16)
    q = qkv.double()
    ref = torch.softmax(q[:, :128] @ q[keep, 128:256].T / 128 ** 0.5, dim=-1) @ q[keep, 256:]
    check_close(host(out), host(ref.float()), "bf16", "attention, infinite scores")


@pytest.mark.parametrize("B", [1, 4, 30, 44, 45, 64, 65, 200])
def test_attention_schedule_made_by_either_kernel(B):
    """Calls of up to 64 segments with a unit per SM at most make the schedule in the
    attention kernel: equal lengths and masked tails against the oracle, and empty
    segments between them change nothing."""
    rng = _rng(B)
    lens = rng.choice([1, 40, 130, 300], B)
    lens[0] = 257
    kv = np.where(rng.random(B) < 0.3, np.maximum(lens - 7, 1), lens)
    _attention_case("f16", 2, 128, [int(v) for v in lens], [int(v) for v in kv], 1.0, B)
    T, ws = int(lens.sum()), torch.empty(1 << 20, dtype=torch.uint8, device=cuda())
    qkv = torch.randn((T, 3 * 256), generator=torch.Generator(device="cuda").manual_seed(B), device="cuda").half()
    keep = np.sort(rng.choice(B + 20, B, replace=False))              # B + 20 segments, 20 of them empty
    more, more_kv = np.zeros(B + 20, dtype=np.int64), np.zeros(B + 20, dtype=np.int64)
    more[keep], more_kv[keep] = lens, kv
    out = []
    for n, k in ((lens, kv), (more, more_kv)):
        o = torch.empty((T, 256), dtype=torch.float16, device="cuda")
        S.seer_attention(qkv, o, "f16", i32(np.concatenate([[0], np.cumsum(n)])), i32(k), len(n), T, 2, 128, ws, 1 << 20)
        out.append(o)
    assert torch.equal(*out)


def test_attention_many_heads():
    _attention_case("f16", 4, 128, [200, 90], [200, 90], 1.0, 12)


@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("H", [8, 3])
def test_attention_many_units_per_cta(dt, H):
    # hundreds of work units, more than there are SMs: each persistent CTA
    # takes units in turn, mixing paired and single query tiles (odd tile
    # counts), masked key tails and one-row segments, for an even and an odd
    # head count
    r = _rng(21)
    lens = [int(x) for x in r.integers(1, 400, 48)]
    lens[3], lens[7], lens[11] = 1, 256, 257
    kv = [max(1, L - int(r.integers(0, min(L, 40)))) for L in lens]
    _attention_case(dt, H, 128, lens, kv, 1.0, 22)


def test_attention_workspace_reused_across_schedules():
    # the unit counter lives in the schedule workspace: a second call with
    # another schedule on the same workspace must start from unit 0 again
    H, dh = 4, 128
    D = H * dh
    T_cap = 3000
    ws_bytes = (H * ((T_cap + 127) // 128 + 64) * 16) + 4096
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=cuda())
    for seed, lens in ((31, [900, 40, 700, 1, 300]), (32, [129] * 20), (33, [2999])):
        rng = _rng(seed)
        cu = np.concatenate([[0], np.cumsum(lens)])
        T = int(cu[-1])
        qkv = _store(rng.standard_normal((T_cap, 3 * D)), "f16")
        out = torch.full((T_cap, D), 3.0, dtype=torch.float16, device=cuda())
        S.seer_attention(to_dev(qkv, "f16"), out, "f16", i32(cu), None, len(lens), T_cap, H, dh, ws, ws_bytes)
        ref = np.concatenate([oracle.attention(qkv[a:b, :D], qkv[a:b, D:2 * D], qkv[a:b, 2 * D:3 * D], H)
                              for a, b in zip(cu[:-1], cu[1:])])
        got = host(out)
        check_close(got[:T], ref, "bf16", f"attention reuse lens={lens}")
        assert (got[T:] == 3.0).all()


def test_attention_f32():
    _attention_case("f32", 4, 64, [1, 70, 33, 130], [1, 70, 20, 130], 1.0, 13)


# ------------------------------------------------------------------ SNR scan (S2)
def _golden(name):
    with open(os.path.join(GOLDEN, name)) as f:
        return json.load(f)["cases"]


def test_snr_scan_golden_bit_exact():
    for case in _golden("snr_cases.json"):
        N = len(case["counts"])
        c = i32(case["counts"])
        L = torch.full((1,), -7, dtype=torch.int32, device=cuda())
        I = torch.full((1,), -7, dtype=torch.int32, device=cuda())
        p = S.make_params(0.0, case["tau_jump"], case["gamma"], case["window"])
        S.seer_snr_scan(c, 1, N, case["F"], p, L, I)
        assert (int(I.item()), int(L.item())) == (case["i_star"], case["L_star"]), case["name"]


@pytest.mark.parametrize("B,N", [(256, 1024), (3, 20000)])
def test_snr_scan_large_shapes_match_oracle_exactly(B, N):
    # many sequences (one block each), and a window longer than the shared-memory
    # staging of the counts (the scan then reads them from global memory)
    rng = _rng(50 + N)
    F = 12288
    counts = rng.integers(0, 100, size=(B, N))
    for b in range(B):
        j = int(rng.integers(1, N - 3))
        counts[b, j:] += int(rng.integers(0, 3000))        # a jump below tau_jump * F (369) is no boundary
    counts[0, :] = 0                                       # no jump at all: L* = N
    p = S.make_params(0.0, 0.03, 0.6, 3)
    L = torch.empty(B, dtype=torch.int32, device=cuda())
    I = torch.empty(B, dtype=torch.int32, device=cuda())
    S.seer_snr_scan(i32(counts.ravel()), B, N, F, p, L, I)
    i_ref, L_ref = oracle.snr_boundaries(counts, F, 0.03, 0.6, 3)
    np.testing.assert_array_equal(I.cpu().numpy(), i_ref)
    np.testing.assert_array_equal(L.cpu().numpy(), L_ref)
    assert L_ref[0] == N and (L_ref[1:] < N).any()


def test_snr_scan_random_matches_oracle_exactly():
    rng = _rng(14)
    B, N, F = 37, 300, 768
    counts = rng.integers(0, 40, size=(B, N))
    for b in range(B):
        j = int(rng.integers(1, N - 3))
        counts[b, j:] = counts[b, j:] + int(rng.integers(0, 200))
    p = S.make_params(0.0, 0.03, 0.6, 3)
    L = torch.empty(B, dtype=torch.int32, device=cuda())
    I = torch.empty(B, dtype=torch.int32, device=cuda())
    S.seer_snr_scan(i32(counts.ravel()), B, N, F, p, L, I)
    i_ref, L_ref = oracle.snr_boundaries(counts, F, 0.03, 0.6, 3)
    np.testing.assert_array_equal(I.cpu().numpy(), i_ref)
    np.testing.assert_array_equal(L.cpu().numpy(), L_ref)


@pytest.mark.parametrize("window", [1, 2, 4, 5, 7, 10])
def test_snr_scan_window_variants_match_oracle_exactly(window):
    # look-ahead window variants (Sec. 4.5, Table 12): plateaus of random length around the window
    rng = _rng(40 + window)
    B, N, F = 29, 260, 768
    counts = rng.integers(0, 12, size=(B, N))
    for b in range(B):
        j = int(rng.integers(1, N - window))
        run = int(rng.integers(1, 2 * window + 2))
        counts[b, j:j + run] += int(rng.integers(20, 300))
    p = S.make_params(0.0, 0.03, 0.6, window)
    L = torch.empty(B, dtype=torch.int32, device=cuda())
    I = torch.empty(B, dtype=torch.int32, device=cuda())
    S.seer_snr_scan(i32(counts.ravel()), B, N, F, p, L, I)
    i_ref, L_ref = oracle.snr_boundaries(counts, F, 0.03, 0.6, window)
    np.testing.assert_array_equal(I.cpu().numpy(), i_ref)
    np.testing.assert_array_equal(L.cpu().numpy(), L_ref)


def test_multi_layer_sparsity_tap():
    # counts of three layers' gate/up weights summed (a count out of 3F), then one scan
    from paper_2607_14557_gb300 import driver as D
    wl = synth.tiny_workload(dtype="bf16", seed=240, d=256, n_heads=2, head_dim=128, d_ff=768, batch=4, window=200,
                             boundary=("uniform", 8, 190), n_layers=3)
    lens = synth.lengths(wl)
    x, cu, resp = synth.hidden_full(wl, lens)
    B, N, F = wl.batch, wl.window, wl.d_ff
    ws = [synth.layer_weights(wl, l) for l in range(3)]
    taps = [D.LayerWeights.from_host(w, "bf16") for w in ws]
    path = D.SeerPath(S.make_dims(wl.d, wl.n_heads, wl.head_dim, F), "bf16", B, N, x.shape[0],
                      S.make_params(wl.act_eps))
    path.detect_multi(to_dev(x, "bf16"), i32(resp), taps)
    torch.cuda.synchronize()
    got = path.counts.cpu().numpy().reshape(B, N)
    for b in range(B):
        ref = sum(oracle.sparsity_counts(x[resp[b]:resp[b] + N], w["wg"], w["wu"], wl.act_eps) for w in ws)
        assert np.abs(got[b] - ref).max() <= 0.005 * 3 * F
    i_ref, L_ref = oracle.snr_boundaries(got, 3 * F)
    np.testing.assert_array_equal(path.L_star.cpu().numpy(), L_ref)
    np.testing.assert_array_equal(path.i_star.cpu().numpy(), i_ref)
    np.testing.assert_array_equal(L_ref, lens.boundary + 1)


# ------------------------------------------------------------------ detector end to end (S1 + S2)
@pytest.mark.parametrize("dtype,seed", [("bf16", 1), ("bf16", 2), ("f32", 3)])
def test_detect_boundary_planted(dtype, seed):
    d = 256
    wl = synth.tiny_workload(dtype=dtype, seed=200 + seed, d=d, n_heads=2 if dtype == "bf16" else 4,
                             head_dim=128 if dtype == "bf16" else 64, d_ff=768, batch=5, window=200,
                             boundary=("uniform", 8, 190))
    lens = synth.lengths(wl)
    x, cu, resp = synth.hidden_full(wl, lens)
    w = synth.layer_weights(wl, 0)
    B, N, F = wl.batch, wl.window, wl.d_ff
    counts = torch.empty(B * N, dtype=torch.int32, device=cuda())
    L = torch.empty(B, dtype=torch.int32, device=cuda())
    I = torch.empty(B, dtype=torch.int32, device=cuda())
    S.seer_detect_boundary(to_dev(x, dtype), dtype, x.shape[0], i32(resp), B, N, to_dev(w["wg"], dtype),
                           to_dev(w["wu"], dtype), S.make_dims(d, wl.n_heads, wl.head_dim, F),
                           S.make_params(wl.act_eps), counts, L, I)
    got = counts.cpu().numpy().reshape(B, N)
    for b in range(B):
        ref = oracle.sparsity_counts(x[resp[b]:resp[b] + N], w["wg"], w["wu"], wl.act_eps)
        assert np.abs(got[b] - ref).max() <= 0.005 * F
    np.testing.assert_array_equal(L.cpu().numpy(), lens.boundary + 1)
    np.testing.assert_array_equal(I.cpu().numpy(), lens.boundary)


# ------------------------------------------------------------------ routing + pack (S3 + S4)
def _pack_case(dtype, ctx, L_star, N, d, tau_pad=0.2, seed=0, extra_cap=50, bucket_min=8):
    rng = _rng(seed)
    B = len(ctx)
    full = np.asarray(ctx) + N
    cu_full = np.concatenate([[0], np.cumsum(full)])
    x = synth.round_storage(rng.standard_normal((int(cu_full[-1]), d)), dtype)
    seg, kv, cu = oracle.segment_layout(ctx, L_star, N, tau_pad, bucket_min=bucket_min)
    ref_rows = oracle.pack_rows(x, cu_full, seg)
    T_cap = int(cu[-1]) + extra_cap
    out = torch.full((T_cap, d), 5.0, dtype=tdtype(dtype), device=cuda())
    cu_out = torch.empty(B + 1, dtype=torch.int32, device=cuda())
    kv_out = torch.empty(B, dtype=torch.int32, device=cuda())
    meta = torch.empty(S.CTRL_WORDS, dtype=torch.int32, device=cuda())
    hctrl = torch.zeros(S.CTRL_WORDS, dtype=torch.int32).pin_memory()
    p = S.make_params(0.0, tau_pad=tau_pad, bucket_min=bucket_min)
    S.seer_pack_ragged(to_dev(x, dtype), dtype, i32(cu_full), i32(ctx), i32(L_star), B, d, N, T_cap, p, out, cu_out,
                       kv_out, meta, hctrl, 9)
    ctrl = torch.zeros(S.CTRL_WORDS, dtype=torch.int32)
    S.seer_poll_ctrl(hctrl, 9, 5_000_000, ctrl)
    torch.cuda.synchronize()
    got = host(out)
    np.testing.assert_array_equal(got[:cu[-1]], ref_rows)
    assert (got[cu[-1]:] == 5.0).all()           # zero work past the packed total
    np.testing.assert_array_equal(cu_out.cpu().numpy(), cu)
    np.testing.assert_array_equal(kv_out.cpu().numpy(), kv)
    m = meta.cpu().numpy()
    c = ctrl.numpy()
    np.testing.assert_array_equal(m, c)
    groups = oracle.route(L_star, N, tau_pad, bucket_min=bucket_min)
    assert c[0] == 9 and c[1] == cu[-1] and c[2] == seg.max() and c[4] == len(groups)
    assert c[5] == sum(1 << p_ for p_ in {g["path"] for g in groups})
    pad_ref = sum(g["bucket"] * len(g["members"]) - sum(L_star[i] for i in g["members"])
                  for g in groups if g["path"] == oracle.PATH_STATIC)
    assert c[6] == pad_ref
    for gi, g in enumerate(groups):
        assert list(c[8 + 4 * gi: 12 + 4 * gi]) == [g["bucket"], len(g["members"]), g["path"],
                                                   int(np.floor(g["rho"] * 1e6))]
    # graph capacity: the smallest m * 2^e >= total with m in 8..15
    cands = sorted(m_ * 2 ** e for m_ in range(8, 16) for e in range(0, 24))
    assert c[3] == next(v for v in cands if v >= max(cu[-1], 1))


def test_pack_route_mixed_paths_bf16():
    ctx = [100, 50, 70, 30, 10, 64, 64]
    L = [120, 128, 110, 125, 300, 5, 16]
    _pack_case("bf16", ctx, L, 1024, 256, seed=1)


def test_pack_route_varlen_and_eager_f32():
    ctx = [33, 17, 80]
    L = [65, 70, 128]
    _pack_case("f32", ctx, L, 128, 64, seed=2)


def test_pack_route_untruncated_is_identity_layout():
    ctx = [40, 41, 42]
    N = 96
    _pack_case("bf16", ctx, [N, N, N], N, 256, seed=3)


@pytest.mark.parametrize("B,tau_pad,bucket_min", [(64, 0.2, 8), (256, 0.2, 8), (256, -1.0, 1), (256, 0.9, 64)])
def test_pack_route_large_batches(B, tau_pad, bucket_min):
    # the routing ablation's batch sizes: every block recomputes the route of all
    # B sequences in shared memory; groups, layout, control word and rows exact
    rng = _rng(40 + B)
    N = 1024
    ctx = list(map(int, rng.integers(0, 3000, B)))
    L = list(map(int, rng.integers(1, N + 1, B)))
    _pack_case("bf16", ctx, L, N, 64, tau_pad=tau_pad, seed=41 + B, bucket_min=bucket_min)


@pytest.mark.parametrize("bucket_min", [1, 16, 64, 1024])
def test_pack_route_bucket_set_variants(bucket_min):
    # the smallest micro-bucket moves the group boundaries (routing ablation)
    ctx = [100, 50, 70, 30, 10, 64, 64, 20]
    L = [120, 128, 110, 125, 300, 5, 16, 3]
    _pack_case("bf16", ctx, L, 1024, 256, seed=30 + bucket_min, bucket_min=bucket_min)


@pytest.mark.parametrize("N,w", [(2, 1), (4, 3), (129, 3), (130, 1), (257, 10), (12284, 3), (12285, 3), (12288, 3), (12289, 3)])
@pytest.mark.parametrize("F,tau,gamma", [(12288, 0.03, 0.6), (100, 0.07, 0.5), (3 * 12288, 0.0, 0.0), (7, 3 / 7, 1.0)])
def test_snr_scan_at_the_thresholds(N, w, F, tau, gamma):
    """Counts whose jump and noise land on, just under and just over tau F and gamma
    jump (where the fp32 filter must leave the decision to the fp64 test), hits in
    every round of candidates and none; bit-exact against the oracle."""
    rng = _rng(N + w + F)
    B = 24
    c = np.zeros((B, N), dtype=np.int64)
    for b in range(B):
        i = int(rng.integers(1, N)) if b % 4 else N - w
        jump = int(np.ceil(tau * F)) + int(rng.integers(-1, 2))
        noise = int(gamma * max(jump, 0)) + int(rng.integers(-1, 2))
        base = int(rng.integers(0, 3))
        c[b, :i] = base
        c[b, i:] = base + max(jump, 0)
        tail = c[b, i:]
        tail[rng.random(len(tail)) < 0.3] += max(noise, 0)
    counts = np.clip(c, 0, F).astype(np.int32)
    L, I = torch.empty(B, dtype=torch.int32, device=cuda()), torch.empty(B, dtype=torch.int32, device=cuda())
    S.seer_snr_scan(torch.from_numpy(counts).to(cuda()), B, N, F, S.make_params(0.0, tau_jump=tau, gamma=gamma, window=w), L, I)
    i_ref, L_ref = oracle.snr_boundaries(counts, F, tau, gamma, w)
    np.testing.assert_array_equal(I.cpu().numpy(), i_ref)
    np.testing.assert_array_equal(L.cpu().numpy(), L_ref)


@pytest.mark.parametrize("tau", [0.0, -1.0, 1e300, -1e300])
@pytest.mark.parametrize("gamma", [0.6, 1e38, 1e300, -1e300, float("inf")])
def test_snr_scan_parameters_beyond_the_fp32_range(tau, gamma):
    """Thresholds that the fp32 filter cannot hold: flat, rising, falling and noisy counts."""
    c = np.array([[5] * 20, [5] * 8 + [9] * 12, [9] * 8 + [5] * 12, [3, 7] * 10, list(range(20))], dtype=np.int32)
    B, N = c.shape
    L, I = torch.empty(B, dtype=torch.int32, device=cuda()), torch.empty(B, dtype=torch.int32, device=cuda())
    S.seer_snr_scan(torch.from_numpy(c).to(cuda()), B, N, 768, S.make_params(0.0, tau_jump=tau, gamma=gamma, window=3), L, I)
    i_ref, L_ref = oracle.snr_boundaries(c, 768, tau, gamma, 3)
    np.testing.assert_array_equal(I.cpu().numpy(), i_ref)
    np.testing.assert_array_equal(L.cpu().numpy(), L_ref)


@pytest.mark.parametrize("B,N,bucket_min", [(1, 1, 1), (33, 1000, 8), (64, 64, 1), (300, 4096, 3), (1000, 17, 8),
                                            (4000, 17, 8), (5327, 17, 8), (5328, 17, 8), (19303, 17, 8)])
def test_pack_route_many_segments(B, N, bucket_min):
    """More segments than a warp, every bucket count, rows of 48 bytes .. 8 KB; segments
    whose lengths, offsets and buckets need more than the default shared memory."""
    rng = _rng(B + N)
    ctx, L = rng.integers(0, 20, B), rng.integers(1, N + 1, B)
    _pack_case("bf16", ctx, L, N, 24 if B > 100 else 4096, seed=B, bucket_min=bucket_min)
