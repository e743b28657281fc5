"""GPU parity of decode attention over a (compacted) cache against the CPU oracle, through the C ABI.

Tolerance: element by element, |gpu - oracle| <= 2e-3 x max(|oracle|, 1e-3 x m), where m is the magnitude
of the weighted sum's terms, sum_j p_j |V[j]| (stepkv_testlib.DECODE_FLOOR).  The GPU computes logits in
fp32 from exact bf16 products, exponentials with the MUFU ex2 and fp32 sums over at most a few thousand
weighted rows, so its error is orders of magnitude below that.
"""
import numpy as np
import pytest

from oracle import stepkv_oracle as O
from paper_2609_22158_gb300 import workload as wl
import stepkv_testlib as TL

pytestmark = pytest.mark.gpu
TOL = 2e-3


@pytest.fixture(scope="module")
def B():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2609_22158_gb300 import binding, build
    build.build_library()
    binding.load_library()
    return binding


def _bits(rng, shape, scale=1.0):
    return wl.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32) * np.float32(scale))


DECODE_CASES = [
    # Hkv, G, d, n, rows, layers, key scale
    (2, 4, 128, 1, 1, 1, 1.0),        # a single key: the output is that key's value row
    (2, 4, 128, 1000, 1000, 2, 1.0),  # ragged last split (1000 = 512 + 488)
    (8, 4, 128, 8272, 8272, 1, 1.0),  # the incremental loop's compacted cache (8192 budget + prefix/window)
    (2, 2, 64, 513, 600, 3, 2.0),     # d = 64, capacity stride above n, one key past a split
    (1, 8, 128, 777, 900, 1, 3.0),    # G = 8, peaky softmax
    (2, 5, 128, 300, 300, 1, 1.0),    # G = 5
    (4, 1, 64, 2049, 2100, 1, 1.0),   # no grouping
]


@pytest.mark.parametrize("Hkv,G,d,n,rows,L,ks", DECODE_CASES)
def test_decode_matches_oracle(B, Hkv, G, d, n, rows, L, ks):
    import torch
    rng = np.random.default_rng(100 + n + d + G)
    qs = [_bits(rng, (Hkv * G, d)) for _ in range(L)]
    Ks = [_bits(rng, (Hkv, rows, d), ks) for _ in range(L)]
    Vs = [_bits(rng, (Hkv, rows, d)) for _ in range(L)]
    st = B.new_status()
    out = B.stepkv_decode([TL.bf16_dev(x) for x in qs], [TL.bf16_dev(x) for x in Ks], [TL.bf16_dev(x) for x in Vs],
                          n, status=st)
    torch.cuda.synchronize()
    assert st.item() == 0
    for l in range(L):
        TL.assert_decode_close(out[l].cpu().numpy(), qs[l], Ks[l][:, :n], Vs[l][:, :n], f"layer {l}")


def test_decode_n_on_device_equals_host_n(B):
    import torch
    rng = np.random.default_rng(5)
    Hkv, G, d, rows, n = 2, 4, 128, 1200, 1100
    q = [TL.bf16_dev(_bits(rng, (Hkv * G, d)))]
    K = [TL.bf16_dev(_bits(rng, (Hkv, rows, d)))]
    V = [TL.bf16_dev(_bits(rng, (Hkv, rows, d)))]
    a = B.stepkv_decode(q, K, V, n)[0]
    b = B.stepkv_decode(q, K, V, torch.tensor([n], dtype=torch.int32, device="cuda"))[0]
    c = B.stepkv_decode(q, K, V, n)[0]
    torch.cuda.synchronize()
    assert torch.equal(a, b) and torch.equal(a, c)  # device-side n, and run-to-run determinism


def test_decode_n_above_capacity_sets_enospace(B):
    import torch
    rng = np.random.default_rng(6)
    Hkv, G, d, rows = 1, 4, 64, 300
    q = [TL.bf16_dev(_bits(rng, (Hkv * G, d)))]
    K = [TL.bf16_dev(_bits(rng, (Hkv, rows, d)))]
    V = [TL.bf16_dev(_bits(rng, (Hkv, rows, d)))]
    st = B.new_status()
    over = B.stepkv_decode(q, K, V, torch.tensor([rows + 7], dtype=torch.int32, device="cuda"), status=st)[0]
    full = B.stepkv_decode(q, K, V, rows)[0]
    torch.cuda.synchronize()
    assert st.item() == B.STEPKV_ENOSPACE
    assert torch.equal(over, full)  # clamped to the capacity


def test_decode_over_compacted_cache(B):
    """Compress a trajectory, then decode over K_out/V_out with n = n_kept read on the device."""
    import torch
    tr = wl.custom(51, L=2, Hq=8, Hkv=2, d=128, T=3000, W=32, n_steps=6, budget=wl.Budget.ratio(1, 5))
    g = TL.GpuTraj(tr)
    prob = g.problem()
    st = B.stepkv_compress([prob], B.Params())
    rng = np.random.default_rng(52)
    qs = [_bits(rng, (8, 128)) for _ in range(tr.shape.L)]
    out = B.stepkv_decode([TL.bf16_dev(x) for x in qs], g.K_out, g.V_out, g.out.n_kept, status=st)
    torch.cuda.synchronize()
    assert st.item() == 0
    n = int(g.out.n_kept.item())
    kept = g.out.kept_idx[:n].cpu().numpy()
    for l in range(tr.shape.L):
        TL.assert_decode_close(out[l].cpu().numpy(), qs[l], O.compact_rows(tr.keys(l), kept),
                               O.compact_rows(tr.values(l), kept), f"layer {l}")


@pytest.mark.parametrize("G,d,h2o", [(1, 64, False), (4, 128, False), (5, 128, True), (8, 64, True)])
@pytest.mark.parametrize("n", [1, 16, 17, 4099, 8190])
def test_decode_stream_split(B, G, d, h2o, n):
    """64 (layer, KV head) pairs of 8192-row caches: every warp streams a range of the list of all pairs' 16-key
    blocks, so ranges begin and end inside pairs, in the last block's remainder, or hold no key at all.  Rows past n
    hold NaN and must not be read into the result."""
    import torch
    rng = np.random.default_rng(7 * n + d + G)
    Hkv, rows = 64, 8192
    q, K, V = _bits(rng, (Hkv * G, d), 2.0), _bits(rng, (Hkv, n, d)), _bits(rng, (Hkv, n, d))
    pad = lambda x: torch.cat([TL.bf16_dev(x), torch.full((Hkv, rows - n, d), float("nan"), dtype=torch.bfloat16,
                                                          device="cuda")], 1)
    Kd, Vd, st = [pad(K)], [pad(V)], B.new_status()
    mass = [torch.zeros((Hkv, rows), dtype=torch.float32, device="cuda")]
    out = B.stepkv_decode([TL.bf16_dev(q)], Kd, Vd, n, status=st)[0]
    if h2o:
        same = B.stepkv_decode_h2o([TL.bf16_dev(q)], Kd, Vd, n, mass, status=st)[0]
    torch.cuda.synchronize()
    assert st.item() == 0
    TL.assert_decode_close(out.cpu().numpy(), q, K, V, f"n {n}")
    if h2o:
        assert torch.equal(same, out)
        TL.assert_close(mass[0][:, :n].cpu().numpy(), O.decode_attention_mass(q, K), "mass", floor=1e-30)
        assert not mass[0][:, n:].any()


@pytest.mark.parametrize("L,Hkv", [(5, 32), (16, 32), (40, 32), (64, 40)])
@pytest.mark.parametrize("G,d,n", [(1, 128, 1), (1, 128, 130), (4, 128, 17), (5, 128, 300), (8, 64, 33), (2, 64, 500)])
def test_decode_more_pairs_than_sms(B, L, Hkv, G, d, n):
    """160 to 2560 (layer, KV head) pairs of few rows: one CTA of four, two or one warps per pair, several on an SM, with
    warps that get no key, one block or a remainder.  Rows past n hold NaN."""
    import torch
    rng = np.random.default_rng(L + n + d)
    rows = n + 7
    some = [(_bits(rng, (Hkv * G, d), 2.0), _bits(rng, (Hkv, n, d)), _bits(rng, (Hkv, n, d))) for _ in range(3)]
    pad = lambda x: torch.cat([TL.bf16_dev(x), torch.full((Hkv, rows - n, d), float("nan"), dtype=torch.bfloat16,
                                                          device="cuda")], 1)
    q, K, V = ([f(s[i]) for s in some] for i, f in enumerate((TL.bf16_dev, pad, pad)))
    st = B.new_status()
    args = [[x[l % 3] for l in range(L)] for x in (q, K, V)]
    out = B.stepkv_decode(*args, n, status=st)
    mass = [torch.zeros((Hkv, rows), dtype=torch.float32, device="cuda") for _ in range(L)]
    same = B.stepkv_decode_h2o(*args, n, mass, status=st)
    torch.cuda.synchronize()
    assert st.item() == 0
    for l in range(3):
        TL.assert_decode_close(out[l].cpu().numpy(), *some[l], f"layer {l}")
        TL.assert_close(mass[l][:, :n].cpu().numpy(), O.decode_attention_mass(some[l][0], some[l][1]), "mass", floor=1e-30)
    for l in range(L):
        assert torch.equal(out[l], out[l % 3]) and torch.equal(same[l], out[l]), l
        assert torch.equal(mass[l], mass[l % 3]) and not mass[l][:, n:].any()


@pytest.mark.parametrize("Hkv,d,rows", [(2, 128, 60), (2, 64, 600), (8, 128, 8911)])
def test_decode_chain_with_changing_n(B, Hkv, d, rows):
    """Calls in a row whose number of keys is written on the device just before each: a call that starts fetching while
    its predecessor finishes sees an older count, above, below or out of range, and must not depend on it.  The rows past
    n are NaN."""
    import torch
    rng = np.random.default_rng(rows)
    q = TL.bf16_dev(_bits(rng, (Hkv * 4, d), 2.0))
    ns = [rows, 1, rows // 2, 17, rows, 33, rows - 1, 16]
    K, V = [], []
    for n in ns:
        for x in (K, V):
            t = torch.full((Hkv, rows, d), float("nan"), dtype=torch.bfloat16, device="cuda")
            t[:, :n] = TL.bf16_dev(_bits(rng, (Hkv, n, d)))
            x.append(t)
    st, n_dev = B.new_status(), torch.full((1,), 2**31 - 1, dtype=torch.int32, device="cuda")
    alone = [B.stepkv_decode([q], [k], [v], n, status=st)[0] for k, v, n in zip(K, V, ns)]
    torch.cuda.synchronize()
    chain = []
    for k, v, n in zip(K, V, ns):
        n_dev.fill_(n)
        chain.append([B.stepkv_decode([q], [k], [v], n_dev, status=st)[0] for _ in range(3)])
        n_dev.fill_(2**31 - 1)
    torch.cuda.synchronize()
    assert st.item() == 0
    for want, got, n in zip(alone, chain, ns):
        assert torch.isfinite(want).all() and all(torch.equal(g, want) for g in got), n


@pytest.mark.parametrize("G", [4, 5])
@pytest.mark.parametrize("Hkv,n", [(2, 60), (2, 3000), (64, 8190)])
def test_decode_infinities(B, Hkv, n, G):
    """Infinite values reach the output as infinities (both signs or a NaN among them: NaN), and keys whose logit is -inf,
    48 in a row, weigh nothing: one CTA per pair, split pairs, and streamed ranges."""
    import torch
    d = 128
    rng = np.random.default_rng(n + G)
    q, K, V = _bits(rng, (Hkv * G, d), 2.0), _bits(rng, (Hkv, n, d)), _bits(rng, (Hkv, n, d))
    q[:, 7] &= 0x7FFF                                   # positive
    K[:, :48, 7] = 0xFF80                               # -inf
    mask = np.ones(n, bool)
    mask[:48] = False
    want = O.decode_attention(q, K[:, mask], V[:, mask])
    V[:, 50, 3], V[:, 52, 4], V[:, 54, 5], V[:, 55, 6] = 0x7F80, 0xFF80, 0x7F80, 0x7FC0
    V[:, 53, 5] = 0xFF80
    want[:, 3], want[:, 4], want[:, 5], want[:, 6] = np.inf, -np.inf, np.nan, np.nan
    st = B.new_status()
    out = B.stepkv_decode([TL.bf16_dev(q)], [TL.bf16_dev(K)], [TL.bf16_dev(V)], n, status=st)[0].cpu().numpy()
    assert st.item() == 0
    np.testing.assert_array_equal(out[:, 3:7], want[:, 3:7].astype(np.float32))
    keep = [e for e in range(d) if not 3 <= e < 7]
    assert np.abs(out[:, keep] - want[:, keep]).max() < 1e-5


@pytest.mark.parametrize("kind", ["nan key", "inf logit", "only nan keys"])
@pytest.mark.parametrize("G", [4, 5])
@pytest.mark.parametrize("Hkv,n", [(2, 60), (2, 3000), (64, 8190)])
def test_decode_nan_logits_reach_the_output(B, Hkv, n, G, kind):
    """A key that is NaN, or a logit of +inf, makes every output of its KV head's query heads NaN: one CTA per pair, split
    pairs, and streamed ranges, with and without accumulated attention.  The other heads are untouched."""
    import torch
    d = 128
    rng = np.random.default_rng(n + G)
    q, K, V = _bits(rng, (Hkv * G, d), 2.0), _bits(rng, (Hkv, n, d)), _bits(rng, (Hkv, n, d))
    h = Hkv - 1
    if kind == "nan key":
        K[h, n // 2, 9] = 0x7FC0
    elif kind == "inf logit":
        q[h * G:, 9] &= 0x7FFF
        K[h, n // 2, 9] = 0x7F80
    else:
        K[h, :, 9] = 0x7FC0
    want = O.decode_attention(q[:h * G], K[:h], V[:h])
    st = B.new_status()
    args = [TL.bf16_dev(q)], [TL.bf16_dev(K)], [TL.bf16_dev(V)], n
    mass = [torch.zeros((Hkv, n), dtype=torch.float32, device="cuda")]
    for out in (B.stepkv_decode(*args, status=st)[0], B.stepkv_decode_h2o(*args, mass, status=st)[0]):
        out = out.cpu().numpy()
        assert st.item() == 0
        assert np.isnan(out[h * G:]).all()
        assert np.abs(out[:h * G] - want).max() < 1e-5
    assert torch.isfinite(mass[0][:h]).all()


def test_decode_rejects_one_bad_layer_among_many(B):
    """Layers laid out alike are checked once: one that differs, wherever it stands, is still found."""
    import torch
    L, Hkv, G, d, rows = 4, 2, 4, 64, 96
    z = lambda *s, **k: torch.zeros(s, device="cuda", **k)
    bf = torch.bfloat16
    good = dict(q=lambda: [z(Hkv * G, d, dtype=bf) for _ in range(L)], K=lambda: [z(Hkv, rows, d, dtype=bf) for _ in range(L)],
                V=lambda: [z(Hkv, rows, d, dtype=bf) for _ in range(L)], mass=lambda: [z(Hkv, rows) for _ in range(L)],
                out=lambda: [z(Hkv * G, d) for _ in range(L)])
    bad = [("q", z(d, Hkv * G, dtype=bf).T, ValueError), ("q", z(Hkv * G, d), TypeError), ("q", z(Hkv * G, d, dtype=bf).cpu(), ValueError),
           ("K", z(Hkv, 2 * rows, d, dtype=bf)[:, :rows], ValueError), ("V", z(Hkv, rows, 2 * d, dtype=bf)[:, :, ::2], ValueError),
           ("K", z(Hkv, rows, d), TypeError), ("V", z(Hkv, rows, d, dtype=bf).cpu(), ValueError),
           ("mass", z(Hkv, rows, dtype=torch.float64), TypeError), ("mass", z(Hkv, rows - 1), ValueError),
           ("mass", z(Hkv, 2 * rows)[:, :rows], ValueError), ("out", z(Hkv * G, d, dtype=bf), TypeError), ("out", z(Hkv * G * d), ValueError)]
    for name, tensor, err in bad:
        for at in (1, L - 1):
            a = {k: f() for k, f in good.items()}
            a[name][at] = tensor
            with pytest.raises(err):
                B.stepkv_decode_h2o(a["q"], a["K"], a["V"], rows, a["mass"], out=a["out"])
    a = {k: f() for k, f in good.items()}
    B.stepkv_decode_h2o(a["q"], a["K"], a["V"], rows, a["mass"], out=a["out"])
    torch.cuda.synchronize()
