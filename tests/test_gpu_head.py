"""LM head + entropy + Gumbel-max kernels against the fp64 oracle
(Eqs. 6-7): entropies within 1e-3 nats; tokens bit-exact except rows whose
oracle top-2 score gap is below the kernel's accumulation error bound."""
import numpy as np
import pytest

import gen
import oracle
from tests.helpers import ENTROPY_TOL, cached_weight, step_inputs, to_dev, token_tolerance, top2_gap

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbd():
    import paper_2509_04185_gb300 as m
    return m


def run_head(sbd, d, dt, tau, with_noise=True):
    import torch
    hid = to_dev(d["hidden"], dt)
    W = to_dev(d["w"], dt)
    m = torch.from_numpy(d["masked"]).cuda()
    g = torch.from_numpy(d["gumbel"]).cuda() if with_noise else None
    ent, tok = sbd.sbd_head_entropy_sample(hid, W, m, g, tau)
    return ent.cpu().numpy(), tok.cpu().numpy()


def compare_head(d, dt, tau, ent, tok, with_noise=True, rows=None):
    """Returns the number of token exemptions (near ties)."""
    g = d["gumbel"] if with_noise else None
    rent, rtok, zs = oracle.head_entropy_sample(oracle.widen(d["hidden"], dt), d["w"], dt,
                                                d["masked"], g, tau, rows=rows)
    m = d["masked"].astype(bool)
    sel = np.zeros_like(m)
    for (b, i) in zs:
        sel[b, i] = True
    assert np.all(np.isinf(ent[~m]) & (ent[~m] > 0)), "unmasked rows must get +inf"
    assert np.all(tok[~m] == -1), "unmasked rows must get token -1"
    err = np.abs(ent[sel] - rent[sel])
    assert err.size == 0 or err.max() <= ENTROPY_TOL, err.max()
    acc = d["hidden"].shape[-1] // (16 if dt == "bf16" else 1)
    exempt = 0
    for (b, i), z in zs.items():
        if tok[b, i] == rtok[b, i]:
            continue
        gb = None if g is None else g[b, i]
        gap = top2_gap(z, gb, tau)
        assert gap < token_tolerance(z, acc), (b, i, tok[b, i], rtok[b, i], gap)
        exempt += 1
    return exempt


def test_tiny_f32_config(sbd):
    w = gen.get_workload("tiny_f32")
    for seed in range(3):
        d = step_inputs(w, seed)
        for tau in (0.0, 1.0):
            ent, tok = run_head(sbd, d, w.dtype, tau, with_noise=tau != 0.0)
            assert compare_head(d, w.dtype, tau, ent, tok, with_noise=tau != 0.0) == 0


@pytest.mark.parametrize("case", range(12))
def test_f32_random_shapes(sbd, case):
    """Seeded random fp32 shapes through head_f32_kernel: hidden widths that
    end in a partial 32-column chunk, partial vocabulary tiles, several
    groups of 32 live rows, tau 0 and 1."""
    rng = np.random.default_rng(3000 + case)
    B = int(rng.integers(1, 5))
    k = int(rng.integers(1, 33))
    V = int(rng.integers(100, 2500))
    H = int(rng.choice([4, 36, 64, 100, 260, 320]))
    tau = float(rng.choice([0.0, 1.0]))
    w = gen.shrink(gen.get_workload("tiny_f32"), batch=B, block_k=k, vocab=V, hidden=H,
                   decoded=("uniform", 0, k))
    d = step_inputs(w, seed=case)
    ent, tok = run_head(sbd, d, "f32", tau, with_noise=tau != 0.0)
    assert compare_head(d, "f32", tau, ent, tok, with_noise=tau != 0.0) <= 1


@pytest.mark.parametrize("philox", [False, True])
@pytest.mark.parametrize("V,H", [(1, 4), (127, 28), (129, 32), (261, 100)])
@pytest.mark.parametrize("R", [1, 8, 9, 16, 17, 24, 25, 32, 33, 41, 64])
def test_f32_row_groups(sbd, R, V, H, philox):
    """Exactly R masked rows of 64 through head_f32_kernel: the edges of its
    row counts per group (8, 16, 24, 32), one id, one id past a tile, column
    counts around the 32-column stage; noise from the buffer and the kernel's
    own, which must agree bit for bit."""
    import torch
    w = gen.shrink(gen.get_workload("tiny_f32"), batch=4, block_k=16, vocab=V, hidden=H)
    d = dict(step_inputs(w, seed=R))
    m = np.zeros(64, dtype=np.uint8)
    m[np.random.default_rng(R).choice(64, size=R, replace=False)] = 1
    d["masked"] = m.reshape(4, 16)
    if philox:
        ids = torch.arange(64, dtype=torch.int32, device="cuda")
        d["gumbel"] = sbd.sbd_gumbel_philox(ids, V, 9, 3).cpu().numpy().reshape(4, 16, V)
    ent, tok = run_head(sbd, d, "f32", 1.0)
    assert compare_head(d, "f32", 1.0, ent, tok) <= 1
    if philox:
        e2, t2 = sbd.sbd_head_entropy_sample_philox(
            to_dev(d["hidden"], "f32"), to_dev(d["w"], "f32"), torch.from_numpy(d["masked"]).cuda(), 9, 3, 1.0)
        assert np.array_equal(t2.cpu().numpy(), tok) and np.array_equal(e2.cpu().numpy(), ent)
    assert sbd.sbd_device_error() == 0


@pytest.mark.parametrize("which", ["none", "all", "first", "last", "odd", "run"])
@pytest.mark.parametrize("B,k", [(1, 1), (1, 31), (4, 8), (3, 11), (15, 17), (8, 32), (257, 1), (16, 32)])
def test_f32_finds_the_masked_rows(sbd, B, k, which):
    """The fp32 kernel's own list of masked rows: counts around its words of 32
    flags and its 256 threads, up to 512; nothing, everything, one row at either
    end, every other row and a run that crosses the words' edges masked."""
    N = B * k
    m = np.zeros(N, dtype=np.uint8)
    m[{"none": slice(0, 0), "all": slice(0, N), "first": slice(0, 1), "last": slice(N - 1, N),
       "odd": slice(1, N, 2), "run": slice(N // 3, 2 * N // 3 + 1)}[which]] = 1
    w = gen.shrink(gen.get_workload("tiny_f32"), batch=B, block_k=k, vocab=37, hidden=12)
    d = dict(step_inputs(w, seed=N))
    d["masked"] = m.reshape(B, k)
    ent, tok = run_head(sbd, d, "f32", 1.0)
    assert compare_head(d, "f32", 1.0, ent, tok) <= 1
    assert sbd.sbd_device_error() == 0


@pytest.mark.parametrize("B,k,V,H", [(1, 1, 1000, 256), (1, 16, 4096 + 5, 512), (2, 16, 3000, 128),
                                     (3, 7, 777, 64), (16, 16, 2100, 256), (1, 17, 500, 128),
                                     (10, 30, 999, 64), (16, 32, 1500, 128),
                                     (2, 16, 40000, 1024), (1, 8, 60013, 512)])
@pytest.mark.parametrize("tau", [0.0, 1.0])
def test_bf16_shapes(sbd, B, k, V, H, tau):
    w = gen.shrink(gen.get_workload("llama8b_k16"), batch=B, block_k=k, vocab=V, hidden=H,
                   decoded=("uniform", 0, k))
    d = step_inputs(w, seed=B + k)
    ent, tok = run_head(sbd, d, "bf16", tau, with_noise=tau != 0.0)
    assert compare_head(d, "bf16", tau, ent, tok, with_noise=tau != 0.0) <= 1


@pytest.mark.parametrize("R", [1, 17, 64, 80, 128, 129, 144, 160, 161, 192, 208, 255, 256, 257, 320, 400, 511,
                               512])
def test_bf16_hidden_box_decomposition(sbd, R):
    """Exactly R masked rows out of 512 (the CTA-pair kernel): the live rows
    are loaded in boxes of 128, 64 and 16 rows (144 = 128 + 16,
    208 = 128 + 64 + 16); up to 160 rows the vocabulary-lane layout (above
    128 rows with N = 160), from 161 the row-lane layout, from 257 with two
    row groups; every row must
    come out right."""
    w = gen.shrink(gen.get_workload("llama8b_k16"), batch=16, block_k=32, vocab=1100, hidden=192,
                   cache_len=16)
    d = step_inputs(w, seed=R)
    rng = np.random.default_rng(R)
    m = np.zeros(16 * 32, dtype=np.uint8)
    m[rng.choice(16 * 32, size=R, replace=False)] = 1
    d["masked"] = m.reshape(16, 32)
    ent, tok = run_head(sbd, d, "bf16", 1.0)
    assert compare_head(d, "bf16", 1.0, ent, tok) <= max(1, R // 50)


def test_bf16_all_masked_and_none_masked(sbd):
    w = gen.shrink(gen.get_workload("llama8b_k16"), batch=4, block_k=8, vocab=1500, hidden=256)
    d = step_inputs(w, seed=5)
    d["masked"] = np.ones_like(d["masked"])
    ent, tok = run_head(sbd, d, "bf16", 1.0)
    assert compare_head(d, "bf16", 1.0, ent, tok) <= 1
    d["masked"] = np.zeros_like(d["masked"])
    ent, tok = run_head(sbd, d, "bf16", 1.0)
    assert np.isinf(ent).all() and (tok == -1).all()


@pytest.mark.parametrize("V", [1, 100, 128])
def test_single_cta_kernel_for_one_vocabulary_tile(sbd, V):
    """A vocabulary of one 128-row tile leaves no CTA pair: the single-CTA
    kernel serves it."""
    w = gen.shrink(gen.get_workload("llama8b_k16"), batch=3, block_k=8, vocab=V, hidden=256,
                   decoded=("uniform", 0, 8))
    d = step_inputs(w, seed=V)
    for tau in (0.0, 1.0):
        ent, tok = run_head(sbd, d, "bf16", tau, with_noise=tau != 0.0)
        assert compare_head(d, "bf16", tau, ent, tok, with_noise=tau != 0.0) <= 1


@pytest.mark.parametrize("philox", [False, True])
def test_pair_kernel_without_masked_rows(sbd, philox):
    """256 allocated rows (the CTA-pair kernel) and none masked: every CTA
    pair allocates, meets and releases with no work, and every output is
    +inf / -1."""
    import torch
    w = gen.shrink(gen.get_workload("llama8b_k16"), batch=16, block_k=16, vocab=3000, hidden=256)
    d = step_inputs(w, seed=2)
    hid, W = to_dev(d["hidden"], "bf16"), to_dev(d["w"], "bf16")
    m = torch.zeros(16, 16, dtype=torch.uint8, device="cuda")
    if philox:
        ent, tok = sbd.sbd_head_entropy_sample_philox(hid, W, m, 5, 6, 1.0)
    else:
        ent, tok = sbd.sbd_head_entropy_sample(hid, W, m, torch.from_numpy(d["gumbel"]).cuda(), 1.0)
    assert torch.isinf(ent).all() and (ent > 0).all() and (tok == -1).all()
    assert sbd.sbd_device_error() == 0


@pytest.mark.parametrize("which", ["none", "all", "first", "last", "odd"])
@pytest.mark.parametrize("B,k", [(1, 1), (1, 15), (2, 8), (1, 17), (31, 1), (4, 8), (3, 11),
                                 (4, 24), (8, 16), (3, 43)])
def test_bf16_rows_in_place(sbd, B, k, which):
    """Up to 32 rows the pair kernel reads every hidden row where it is: rows
    that are not masked may hold anything (NaN here) without touching the
    others, and none masked means no work; 33 rows are compacted, and above 128
    the kernel has both layouts.  Noise from the buffer and the kernel's own, which must agree bit for bit."""
    import torch
    N = B * k
    m = np.zeros(N, dtype=np.uint8)
    m[{"none": slice(0, 0), "all": slice(0, N), "first": slice(0, 1), "last": slice(N - 1, N),
       "odd": slice(1, N, 2)}[which]] = 1
    w = gen.shrink(gen.get_workload("llama8b_k16"), batch=B, block_k=k, vocab=801, hidden=192,
                   cache_len=64)
    d = dict(step_inputs(w, seed=N))
    d["masked"] = m.reshape(B, k)
    ids = torch.arange(N, dtype=torch.int32, device="cuda")
    d["gumbel"] = sbd.sbd_gumbel_philox(ids, 801, 5, 2).cpu().numpy().reshape(B, k, 801)
    hid, W, mk = to_dev(d["hidden"], "bf16"), to_dev(d["w"], "bf16"), torch.from_numpy(d["masked"]).cuda()
    hid[mk == 0] = float("nan")
    ent, tok = sbd.sbd_head_entropy_sample(hid, W, mk, torch.from_numpy(d["gumbel"]).cuda(), 1.0)
    assert compare_head(d, "bf16", 1.0, ent.cpu().numpy(), tok.cpu().numpy()) <= 1
    e2, t2 = sbd.sbd_head_entropy_sample_philox(hid, W, mk, 5, 2, 1.0)
    assert torch.equal(e2, ent) and torch.equal(t2, tok)
    assert sbd.sbd_device_error() == 0


def test_bf16_uniform_and_one_hot_rows(sbd):
    """Closed forms through the kernel: zero hidden -> uniform -> log V;
    a huge logit -> entropy 0 and that token."""
    V, H = 2048, 128
    w = gen.shrink(gen.get_workload("llama8b_k16"), batch=1, block_k=2, vocab=V, hidden=H)
    d = step_inputs(w, seed=1)
    d["hidden"] = d["hidden"].copy()
    d["w"] = d["w"].copy()
    d["masked"] = np.ones((1, 2), dtype=np.uint8)
    d["hidden"][0, 0] = 0                                     # bf16 +0.0
    d["hidden"][0, 1] = gen.f32_to_bf16_bits(np.full(H, 1.0, np.float32))
    d["w"][77] = gen.f32_to_bf16_bits(np.full(H, 2.0, np.float32))   # z_77 = 256
    ent, tok = run_head(sbd, d, "bf16", 0.0, with_noise=False)
    assert abs(ent[0, 0] - np.log(V)) < 1e-4
    assert tok[0, 0] == 0                                      # all equal -> lowest id
    assert ent[0, 1] < 1e-4 and tok[0, 1] == 77


@pytest.mark.parametrize("name", ["llama8b_k16", "ragged_b32_k8", "qwen8b_long_k16"])
def test_full_size_configs(sbd, name):
    w = gen.get_workload(name)
    d = step_inputs(w, seed=0)
    ent, tok = run_head(sbd, d, w.dtype, 1.0)
    assert compare_head(d, w.dtype, 1.0, ent, tok) <= 1
    ent0, tok0 = run_head(sbd, d, w.dtype, 0.0, with_noise=False)
    assert compare_head(d, w.dtype, 0.0, ent0, tok0, with_noise=False) <= 1
    np.testing.assert_array_equal(ent, ent0)                  # entropy independent of tau


@pytest.mark.parametrize("k", [16, 32])
def test_sweep_first_step(sbd, k):
    """The first step of a k = 16 or k = 32 block of the 32-layer sweep:
    batch 16, all 256 or 512 block positions masked, hidden 4096, vocab
    128256 (the compute-bound row-lane layout of the CTA-pair kernel, with
    one or two row groups), at tau = 1 and tau = 0, against one evaluation
    of the oracle's logits."""
    w = gen.sweep_workload(k)
    B, k, V, H = w.batch, w.block_k, w.vocab, w.hidden
    d = {"w": cached_weight(V, H, "bf16", 0), "hidden": gen.hidden_states(w, 0, 0),
         "gumbel": gen.gumbel_noise(w, 0, 0), "masked": np.ones((B, k), dtype=np.uint8)}
    ent1, tok1 = run_head(sbd, d, "bf16", 1.0)
    ent0, tok0 = run_head(sbd, d, "bf16", 0.0, with_noise=False)
    np.testing.assert_array_equal(ent1, ent0)
    rent, rtok1, zs = oracle.head_entropy_sample(oracle.widen(d["hidden"], "bf16"), d["w"], "bf16",
                                                 d["masked"], d["gumbel"], 1.0)
    assert len(zs) == B * k
    assert np.abs(ent1 - rent).max() <= ENTROPY_TOL
    acc = H // 16
    exempt = 0
    for (b, i), z in zs.items():
        for tau, tok, g in ((1.0, tok1, d["gumbel"][b, i]), (0.0, tok0, None)):
            want = rtok1[b, i] if tau == 1.0 else oracle.sample_token(z, None, 0.0)
            if tok[b, i] != want:
                gap = top2_gap(z, g, tau)
                assert gap < token_tolerance(z, acc), (b, i, tau, tok[b, i], want, gap)
                exempt += 1
    print(f"token exemptions: {exempt} of {2 * B * k}")
    assert exempt <= 2


@pytest.mark.parametrize("case", range(40))
def test_pair_kernel_random_shapes(sbd, case):
    """Seeded random shapes through the CTA-pair LM head: vocabularies that
    leave a partial pair tile (or a pair tile past the end), hidden sizes of
    any number of 64-column boxes, live-row counts across both layouts and
    both row-group counts, noise from the buffer or in-kernel, tau 0 or 1."""
    import torch
    rng = np.random.default_rng(1000 + case)
    B = int(rng.integers(1, 17))
    k = int(rng.integers(1, 33))
    while B * k > 512:
        k //= 2
    V = int(rng.integers(257, 6000))
    H = 64 * int(rng.integers(1, 17))
    R = int(rng.integers(0, B * k + 1))
    tau = float(rng.choice([0.0, 1.0]))
    philox = bool(rng.integers(0, 2)) and tau != 0.0
    w = gen.shrink(gen.get_workload("llama8b_k16"), batch=B, block_k=k, vocab=V, hidden=H,
                   cache_len=16)
    d = step_inputs(w, seed=case)
    m = np.zeros(B * k, dtype=np.uint8)
    m[rng.choice(B * k, size=R, replace=False)] = 1
    d["masked"] = m.reshape(B, k)
    hid, W = to_dev(d["hidden"], "bf16"), to_dev(d["w"], "bf16")
    mt = torch.from_numpy(d["masked"]).cuda()
    if philox:
        seed, offset = 77 + case, 5 * case
        ent, tok = sbd.sbd_head_entropy_sample_philox(hid, W, mt, seed, offset, tau)
        g, _ = oracle.philox_gumbel(np.arange(B * k), V, seed, offset)
        d["gumbel"] = g.reshape(B, k, V)
        slack = 2e-5 * tau
    else:
        g = torch.from_numpy(d["gumbel"]).cuda() if tau != 0.0 else None
        ent, tok = sbd.sbd_head_entropy_sample(hid, W, mt, g, tau)
        slack = 0.0
    ent, tok = ent.cpu().numpy(), tok.cpu().numpy()
    noise = d["gumbel"] if tau != 0.0 else None
    rent, rtok, zs = oracle.head_entropy_sample(oracle.widen(d["hidden"], "bf16"), d["w"], "bf16",
                                                d["masked"], noise, tau)
    sel = d["masked"].astype(bool)
    assert np.all(np.isinf(ent[~sel])) and np.all(tok[~sel] == -1)
    if R:
        assert np.abs(ent[sel] - rent[sel]).max() <= ENTROPY_TOL, (B, k, V, H, R)
    exempt = 0
    for (b, i), z in zs.items():
        if tok[b, i] != rtok[b, i]:
            gap = top2_gap(z, None if noise is None else noise[b, i], tau)
            assert gap < token_tolerance(z, H // 16) + slack, (B, k, V, H, R, b, i, gap)
            exempt += 1
    assert exempt <= max(1, R // 50)
    assert sbd.sbd_device_error() == 0


@pytest.mark.parametrize("R", [3, 12, 20, 32])
@pytest.mark.parametrize("ids", [(128, 256), (4224, 4352), (4480, 4600)])
def test_f32_tile_of_minus_infinity_logits(sbd, R, ids):
    """A vocabulary tile whose logits are all -inf adds nothing: entropy, token
    and confidence are those of the other ids.  Tiles 33 and 35 of 36 are merged
    into statistics that their lane already holds."""
    import torch
    V, H = 4600, 64
    g = torch.Generator(device="cuda").manual_seed(R)
    hid = torch.rand(1, R, H, generator=g, device="cuda") + 0.5
    w = torch.randn(V, H, generator=g, device="cuda") * 0.3
    gum = torch.randn(1, R, V, generator=g, device="cuda")
    m = torch.ones(1, R, dtype=torch.uint8, device="cuda")
    keep = torch.ones(V, dtype=torch.bool, device="cuda")
    keep[ids[0]:ids[1]] = False
    w[~keep] = -float("inf")
    ent, conf, tok = sbd.sbd_head_entropy_confidence_sample(hid, w, m, gum, 1.0)
    z = hid[0].double() @ w[keep].double().T
    p = torch.log_softmax(z, 1)
    assert float((ent[0] + (p.exp() * p).sum(1)).abs().max()) <= ENTROPY_TOL
    assert float((conf[0] / p.max(1).values.exp() - 1).abs().max()) <= 1e-4
    ref = keep.nonzero()[:, 0][(z + gum[0][:, keep].double()).argmax(1)]
    assert torch.equal(tok[0].long(), ref)
    assert sbd.sbd_device_error() == 0


@pytest.mark.parametrize("B,k", [(1, 1), (1, 16), (4, 8)])
def test_bf16_early_reads_of_a_large_weight(sbd, B, k):
    """A weight large enough that its first part is brought into L2 before the
    kernel's wait, most of it only when a row is seen masked: nothing masked, all,
    one, and flags that a kernel just before the call sets or clears."""
    import torch
    V, H = 25003, 2048
    g = torch.Generator(device="cuda").manual_seed(B * k)
    hid = torch.randn(B, k, H, generator=g, device="cuda").to(torch.bfloat16)
    w = (torch.randn(V, H, generator=g, device="cuda") * 0.02).to(torch.bfloat16)
    z = hid.view(-1, H).double() @ w.double().T
    p = torch.log_softmax(z, 1)
    ref_e, ref_t = -(p.exp() * p).sum(1), z.argmax(1)
    m = torch.zeros(B, k, dtype=torch.uint8, device="cuda")
    ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    one = torch.zeros(B * k, dtype=torch.uint8, device="cuda")
    one[-1] = 1
    for flags in (torch.zeros_like(one), torch.ones_like(one), torch.zeros_like(one), one, 1 - one, torch.ones_like(one)):
        m.view(-1).copy_(flags)
        ent, tok = sbd.sbd_head_entropy_sample(hid, w, m, None, 0.0, workspace=ws)
        on = flags.bool()
        e, t = ent.view(-1), tok.view(-1)
        assert bool(torch.isinf(e[~on]).all()) and bool((t[~on] == -1).all())
        assert not on.any() or float((e - ref_e)[on].abs().max()) <= ENTROPY_TOL
        assert torch.equal(t[on].long(), ref_t[on])
    assert sbd.sbd_device_error() == 0
