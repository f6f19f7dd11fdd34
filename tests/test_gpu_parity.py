"""GPU parity: every CUDA kernel against the CPU oracle, element by element.

All quantities are integers, so the bar is bit-exact equality.  Inputs are
seeded synthetic traces (tracegen) or seeded random arrays; nothing the oracle
sees comes from the CUDA path.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="needs a CUDA GPU")]
else:
    pytestmark = pytest.mark.gpu

import oracle as O
import oracle.pipeline as OP
import tracegen as tg

DEV = torch.device("cuda", 0)


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2608_19677_gb300 as P
    return P


@pytest.fixture(scope="module")
def ctx(P):
    c = P.Context(0)
    yield c
    c.close()


def d_u64(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.uint64).view(np.int64)).to(DEV)


def d_u32(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.uint32).view(np.int32)).to(DEV)


def d_u16(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.uint16).view(np.int16)).to(DEV)


def h_u64(t):
    return t.cpu().numpy().view(np.uint64)


def h_u16(t):
    return t.cpu().numpy().view(np.uint16)


# ------------------------------------------------------------------ a1 hash ---
@pytest.mark.parametrize("align", [1, 2, 4])
def test_hash_trace(P, ctx, align):
    cfg = tg.CONFIGS["70b"].scaled(3000, 1)
    tr = tg.Trace(cfg)
    iv = tr.interval(0)
    tok, off = tg.arena_host(tr, iv, align)
    ref = O.hash_prefixes(tok, off, iv.plen, salt=12345)
    got = P.hash_prefixes(ctx, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen), salt=12345)
    ctx.sync()
    assert (h_u64(got) == ref).all()


def test_hash_edge_lengths_and_offsets(P, ctx):
    rng = np.random.default_rng(5)
    lens = [0, 1, 2, 3, 4, 5, 7, 8, 9, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023,
            1024, 1025, 4095, 4096, 4097, 16383, 16384, 32768]
    tok = rng.integers(-2**31, 2**31, size=200_000, dtype=np.int64).astype(np.int32)
    offs, plens = [], []
    for o0 in range(8):               # every alignment of the span start
        for L in lens:
            o = int(rng.integers(0, tok.size - L - 8)) // 8 * 8 + o0
            offs.append(o)
            plens.append(L)
    offs = np.array(offs, np.uint64)
    plens = np.array(plens, np.uint32)
    ref = O.hash_prefixes(tok, offs, plens, salt=(1 << 64) - 3)
    got = P.hash_prefixes(ctx, torch.from_numpy(tok).to(DEV), d_u64(offs), d_u32(plens), salt=(1 << 64) - 3)
    ctx.sync()
    assert (h_u64(got) == ref).all()


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_hash_every_start_and_remainder(P, ctx, shift):
    # every start within a 16-byte vector (the arena itself starting `shift` tokens into one) with
    # lengths around none, one and several groups of 128 vectors, and every remainder
    plens = np.concatenate([np.arange(0, 24), np.arange(508, 528), np.arange(1020, 1040), np.arange(4090, 4104)])
    plens = np.repeat(plens, 4).astype(np.uint32)
    starts = np.tile(np.arange(4), plens.size // 4)
    pos, offs = 0, []
    for s, p in zip(starts, plens):  # each span at its start within a vector, right after the last
        pos = (pos + 3) // 4 * 4 + int(s)
        offs.append(pos)
        pos += int(p)
    offs = np.array(offs, np.uint64)
    tok = np.random.default_rng(shift).integers(-2**31, 2**31, pos + 1, dtype=np.int64).astype(np.int32)
    ref = O.hash_prefixes(tok, offs, plens, salt=99)
    dev = torch.zeros(tok.size + 3, dtype=torch.int32, device=DEV)[shift:shift + tok.size]
    dev.copy_(torch.from_numpy(tok))
    got = P.hash_prefixes(ctx, dev, d_u64(offs), d_u32(plens), salt=99)
    ctx.sync()
    assert (h_u64(got) == ref).all()


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_hash_short_spans(P, ctx, shift):
    # the lengths that are read word by word (8 to 192 tokens, unless they are whole vectors) and
    # their neighbours, at every start within a vector, the arena itself `shift` tokens into one
    plens = np.repeat(np.concatenate([np.arange(0, 12), np.arange(60, 70), np.arange(124, 132), np.arange(186, 204)]), 4)
    offs = np.cumsum(np.concatenate([[0], plens[:-1] + 5])) // 4 * 4 + np.tile(np.arange(4), plens.size // 4)
    tok = np.random.default_rng(shift).integers(-2**31, 2**31, int(offs[-1] + 300), dtype=np.int64).astype(np.int32)
    ref = O.hash_prefixes(tok, offs.astype(np.uint64), plens.astype(np.uint32), salt=7)
    dev = torch.zeros(tok.size + 3, dtype=torch.int32, device=DEV)[shift:shift + tok.size]
    dev.copy_(torch.from_numpy(tok))
    got = P.hash_prefixes(ctx, dev, d_u64(offs), d_u32(plens), salt=7)
    ctx.sync()
    assert (h_u64(got) == ref).all()


def test_hash_empty(P, ctx):
    t = torch.zeros(4, dtype=torch.int32, device=DEV)
    out = P.hash_prefixes(ctx, t, torch.zeros(0, dtype=torch.int64, device=DEV),
                          torch.zeros(0, dtype=torch.int32, device=DEV))
    ctx.sync()
    assert out.numel() == 0


# ------------------------------------------------------------------ a2..a6 ---
def _rates_keys(rng, nkeys, total, skew=1.2):
    w = rng.pareto(skew, size=nkeys) + 1e-3
    c = np.maximum(1, np.round(w / w.sum() * total)).astype(np.int64)
    ks = rng.integers(0, 2**64, size=nkeys, dtype=np.uint64)
    keys = np.repeat(ks, c)
    rng.shuffle(keys)
    return keys


def _cmp_plan(got, ref):
    assert got["U"] == ref.U
    assert got["n_adm"] == ref.n_adm and got["sum_k"] == ref.sum_k and got["cold"] == ref.cold
    assert (got["adm_key"] == ref.adm_key).all()
    assert (got["adm_cnt"] == ref.adm_cnt).all()
    assert (got["adm_k"] == ref.adm_k).all()
    assert (got["koff"] == ref.koff).all()
    assert (got["members"] == ref.members).all()
    assert (got["jobs"] == ref.jobs).all()
    assert (got["load"] == ref.load).all()


@pytest.mark.parametrize("seed", range(8))
def test_plan_parity(P, ctx, seed):
    rng = np.random.default_rng(200 + seed)
    R = int(rng.choice([1, 2, 3, 7, 30, 64, 100, 1024]))
    W = int(rng.integers(1, 20))
    nkeys = int(rng.integers(1, 5000))
    keys = _rates_keys(rng, nkeys, int(rng.integers(nkeys, 60000)))
    n = keys.size
    num, den = (5 * n, 4 * R) if seed % 2 == 0 else (n, 9 * R)
    variants = ("LPT", "RANDOM", "NOREPL", "SLOTCAP")
    plans = [P.Plan(ctx) for _ in variants]
    params = [P.plan_params(R, W, num, den, v, seed=seed, epoch=3) for v in variants]
    P.build_plans(ctx, d_u64(keys), params, plans)
    uk, uc = O.histogram(keys)
    for pl, v in zip(plans, variants):
        got = pl.export()
        assert (got["ukey"] == uk).all() and (got["ucnt"] == uc).all()
        _cmp_plan(got, O.build_plan(keys, R, W, num, den, variant=v, seed=seed, epoch=3))


def _keys_with_counts(rng, counts):
    ks = np.unique(rng.integers(0, 2**64 - 1, size=len(counts) + 64, dtype=np.uint64))[:len(counts)]
    rng.shuffle(ks)
    keys = np.repeat(ks, np.asarray(counts, np.int64))
    rng.shuffle(keys)
    return keys


@pytest.mark.parametrize("case", ["ties_at_threshold", "U_eq_C", "U_eq_C_minus_1", "U_eq_C_plus_1",
                                  "wide_counts", "single_key", "all_equal"])
def test_plan_admission_candidates(P, ctx, case):
    # the planner sorts only keys whose count reaches the C-th largest (C = R*W);
    # these traces put that threshold on its edge cases
    rng = np.random.default_rng(len(case))
    R, W = 8, 5                      # C = 40
    if case == "ties_at_threshold":  # 30 distinct counts above, 500 keys tied at the 40th count
        counts = list(range(100, 130)) + [7] * 500 + [3] * 200
    elif case == "U_eq_C":
        counts = list(rng.integers(1, 50, size=40))
    elif case == "U_eq_C_minus_1":
        counts = list(rng.integers(1, 50, size=39))
    elif case == "U_eq_C_plus_1":
        counts = list(rng.integers(1, 50, size=41))
    elif case == "wide_counts":      # counts over 17 bits: both select levels matter
        counts = list(rng.integers(1, 120000, size=60)) + list(rng.integers(1, 40, size=3000))
    elif case == "single_key":
        R, W = 1, 1
        counts = [12345]
    else:                            # every key ties
        counts = [5] * 2000
    keys = _keys_with_counts(rng, counts)
    n = keys.size
    params = [P.plan_params(R, W, 5 * n, 4 * R, v, seed=2, epoch=4) for v in ("LPT", "RANDOM", "NOREPL")]
    plans = [P.Plan(ctx) for _ in params]
    P.build_plans(ctx, d_u64(keys), params, plans)
    uk, uc = O.histogram(keys)
    for pl, v in zip(plans, ("LPT", "RANDOM", "NOREPL")):
        got = pl.export()
        assert (got["ukey"] == uk).all() and (got["ucnt"] == uc).all()
        _cmp_plan(got, O.build_plan(keys, R, W, 5 * n, 4 * R, variant=v, seed=2, epoch=4))


@pytest.mark.parametrize("R,nkeys,total", [(30, 150000, 400000), (1024, 300000, 1200000)])
def test_plan_parity_large_histogram(P, ctx, R, nkeys, total):
    # histograms far above the one-CTA sort size (device-wide radix passes)
    rng = np.random.default_rng(nkeys)
    keys = _rates_keys(rng, nkeys, total, skew=0.9)
    n = keys.size
    params = [P.plan_params(R, 64, 5 * n, 4 * R, v, seed=3, epoch=1) for v in ("LPT", "RANDOM", "NOREPL")]
    plans = [P.Plan(ctx) for _ in params]
    P.build_plans(ctx, d_u64(keys), params, plans)
    uk, uc = O.histogram(keys)
    for pl, v in zip(plans, ("LPT", "RANDOM", "NOREPL")):
        got = pl.export()
        assert (got["ukey"] == uk).all() and (got["ucnt"] == uc).all()
        _cmp_plan(got, O.build_plan(keys, R, 64, 5 * n, 4 * R, variant=v, seed=3, epoch=1))


@pytest.mark.parametrize("R,spread", [(33, 0), (64, 50), (257, 3), (1024, 0), (1024, 400)])
def test_plan_equal_rate_runs(P, ctx, R, spread):
    # long runs of keys with the same count and k = 1 (placed a run at a time on
    # the device), hot replicated keys before them, short runs, runs with
    # counts above 1024, and uneven starting loads
    rng = np.random.default_rng(R + spread)
    counts = [3000] * 2 + [1500] * 3 + [1100] * 40 + [37] * 70 + [5] * 300 + [2] * 900 + [1] * 5000
    counts += list(rng.integers(1, 60, size=200))
    ks = np.unique(rng.integers(0, 2**64 - 1, size=len(counts) + 64, dtype=np.uint64))[:len(counts)]
    rng.shuffle(ks)
    keys = np.repeat(ks, counts)
    rng.shuffle(keys)
    init = None
    if spread:
        init = rng.integers(0, spread + 1, size=R).astype(np.uint64)
    W = 2 + 6500 // R
    params = [P.plan_params(R, W, 2000, 1, v, init_load=None if init is None else d_u64(init))
              for v in ("LPT", "NOREPL")]
    plans = [P.Plan(ctx) for _ in params]
    P.build_plans(ctx, d_u64(keys), params, plans)
    for pl, v in zip(plans, ("LPT", "NOREPL")):
        _cmp_plan(pl.export(), O.build_plan(keys, R, W, 2000, 1, variant=v, init_load=init))


def test_plan_hand_example_and_init_load(P, ctx):
    keys = np.array([1] * 21 + [2] * 6 + [3] * 3 + [4], np.uint64)
    pl = P.build_plan(ctx, d_u64(keys), P.plan_params(3, 1, 155, 12))
    _cmp_plan(pl.export(), O.build_plan(keys, 3, 1, 155, 12))
    init = np.array([9, 0, 4], np.uint64)
    pl2 = P.build_plan(ctx, d_u64(keys), P.plan_params(3, 2, 1000, 1, init_load=d_u64(init)))
    _cmp_plan(pl2.export(), O.build_plan(keys, 3, 2, 1000, 1, init_load=init))


@pytest.mark.parametrize("R", [1, 33, 1023, 1024])
@pytest.mark.parametrize("spread", [0, 3000, 2**23, 2**33])
def test_plan_lpt_runs_at_digit_edges(P, ctx, R, spread):
    # runs of equal counts on both sides of the run sort's digit (64, 4096) and of the shortest
    # run (31, 32, 33 keys), from even, uneven (32-bit packed loads) and wide starting loads
    # (64-bit packed loads; above 2^31 no run is placed at once)
    rng = np.random.default_rng(R + spread % 97)
    runs = [(4097, 33), (4096, 32), (4095, 31), (65, 40), (64, 700), (63, 33), (2, 1500), (1, 3000)]
    ids = rng.integers(1, 2**63, sum(m for _, m in runs), dtype=np.int64).astype(np.uint64)
    keys = np.repeat(ids, np.repeat([q for q, _ in runs], [m for _, m in runs]))
    rng.shuffle(keys)
    init = rng.integers(0, spread + 1, R).astype(np.uint64)
    W = max(1, 5000 // R)
    pl = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, keys.size, 1, init_load=d_u64(init)))
    _cmp_plan(pl.export(), O.build_plan(keys, R, W, keys.size, 1, init_load=init))


@pytest.mark.parametrize("variants", [["RANDOM"] * 17, ["LPT", "RANDOM", "NOREPL", "SLOTCAP"] * 5])
def test_plan_placements_in_one_launch(P, ctx, variants):
    # more plans than one placement launch takes, of mixed kinds and fleet sizes (the LPT of
    # R > 1024 and short LPT lists have launches of their own), replicated keys dealt to warps
    rng = np.random.default_rng(len(variants))
    keys = _rates_keys(rng, 3000, 60000)
    Rs = [(1 + 37 * j) % 300 + 2 if j != 4 else 1500 for j in range(len(variants))]
    params = [P.plan_params(R, 8, 300, 1, v, seed=j, epoch=3) for j, (R, v) in enumerate(zip(Rs, variants))]
    plans = [P.Plan(ctx) for _ in variants]
    P.build_plans(ctx, d_u64(keys), params, plans)
    for j, (R, v) in enumerate(zip(Rs, variants)):
        _cmp_plan(plans[j].export(), O.build_plan(keys, R, 8, 300, 1, variant=v, seed=j, epoch=3))


@pytest.mark.parametrize("U,C", [(63, 1000), (65, 3), (4095, 10**5), (4096, 50), (4097, 4000), (4097, 10**5),
                                 (9000, 4096), (9000, 4097), (9000, 6000)])
def test_plan_order_at_sort_edges(P, ctx, U, C):
    # distinct keys and admission candidates on both sides of the shared-memory sort's size, with
    # many equal counts (ties broken by key) and keys that differ only in their low or high bits
    rng = np.random.default_rng(U + C)
    ids = np.unique(np.concatenate([np.arange(U // 3, dtype=np.uint64), np.arange(U // 3, dtype=np.uint64) << np.uint64(50),
                                    rng.integers(1, 2**63, U, dtype=np.int64).astype(np.uint64)]))
    ids = rng.permutation(ids)[:U]
    keys = np.repeat(ids, rng.integers(1, 6, U))
    rng.shuffle(keys)
    pl = P.build_plan(ctx, d_u64(keys), P.plan_params(1, C, keys.size, 1))
    got = pl.export()
    uk, uc = O.histogram(keys)
    assert (got["ukey"] == uk).all() and (got["ucnt"] == uc).all()
    _cmp_plan(got, O.build_plan(keys, 1, C, keys.size, 1))


@pytest.mark.parametrize("extra", [[2**64 - 1], [0], [2**64 - 1, 0, 2**64 - 1, 2**64 - 2]])
def test_plan_extreme_keys(P, ctx, extra):
    # the all-ones key doubles as the device table's empty marker and is counted apart
    rng = np.random.default_rng(len(extra))
    keys = np.concatenate([_rates_keys(rng, 500, 5000), np.array(extra * 7, np.uint64)])
    rng.shuffle(keys)
    R, W = 8, 4
    pl = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, keys.size, 3 * R))
    got = pl.export()
    uk, uc = O.histogram(keys)
    assert (got["ukey"] == uk).all() and (got["ucnt"] == uc).all()
    _cmp_plan(got, O.build_plan(keys, R, W, keys.size, 3 * R))


def test_plan_empty_and_single(P, ctx):
    pl = P.build_plan(ctx, torch.zeros(0, dtype=torch.int64, device=DEV), P.plan_params(4, 2, 1, 1))
    got = pl.export()
    assert got["U"] == 0 and got["n_adm"] == 0 and (got["load"] == 0).all()
    keys = np.array([7, 7, 7], np.uint64)
    pl = P.build_plan(ctx, d_u64(keys), P.plan_params(5, 1, 1, 1))   # q_cap = 1: k = min(R, 3)
    _cmp_plan(pl.export(), O.build_plan(keys, 5, 1, 1, 1))


def test_plan_bad_params(P, ctx):
    keys = d_u64(np.array([1, 2], np.uint64))
    with pytest.raises(P.CacheRouteError):
        P.build_plan(ctx, keys, P.plan_params(0, 1, 1, 1))
    with pytest.raises(P.CacheRouteError):
        P.build_plan(ctx, keys, P.plan_params(4, 1, 1, 0))
    with pytest.raises(P.CacheRouteError):
        P.build_plan(ctx, keys, P.plan_params(P.MAX_R + 1, 1, 1, 1))


# ------------------------------------------------------------------ a7 route ---
@pytest.mark.parametrize("R,B", [(1, 1), (3, 1), (7, 33), (30, 1024), (64, 5000), (1024, 256), (30, 20000),
                                 (5, 16384), (9, 16385), (1024, 1), (64, 2), (30, 3), (7, 31), (1024, 32),
                                 (257, 5), (8192, 1), (8192, 7), (8192, 64)])
def test_route_parity(P, ctx, R, B):
    # batches of <= 32 requests take the one-warp-per-replica kernel, longer ones the CTA kernel
    rng = np.random.default_rng(R * 7 + B)
    keys = _rates_keys(rng, 3000, 40000)
    n = keys.size
    pols = ["CR", "CR_NOLPT", "CR_NOREPL", "P2C", "RR", "HASH", "CR", "P2C", "CHWBL", "CHWBL"]
    seeds = [0, 1, 0, 2, 3, 4, 9, 2**63 + 5, 11, 2**64 - 1]
    ring_args = {8: (64, 5), 9: (1, 2**63 + 1)}  # replica -> (vnodes, ring seed)
    orings = [O.Ring(R, *ring_args[i]) if i in ring_args else None for i in range(len(pols))]
    drings = [P.Ring(ctx, R, *ring_args[i]) if i in ring_args else None for i in range(len(pols))]
    num, den = n, 6 * R            # tight: replicated keys
    W = 4
    oplans = {v: O.build_plan(keys, R, W, num, den, variant=v, seed=s, epoch=1)
              for v, s in (("LPT", 0), ("RANDOM", 1), ("NOREPL", 0))}
    dplans = {}
    for v, s in (("LPT", 0), ("RANDOM", 1), ("NOREPL", 0)):
        dplans[v] = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, num, den, v, seed=s, epoch=1))
    vmap = {"CR": "LPT", "CR_NOLPT": "RANDOM", "CR_NOREPL": "NOREPL"}
    init = rng.integers(0, 50, size=(len(pols), R)).astype(np.uint64)
    ref_dest, ref_load = O.route([oplans.get(vmap.get(p)) for p in pols], pols, seeds, R, keys, 777, B,
                                 load=init, rings=orings)
    load = d_u64(init.reshape(-1)).view(len(pols), R).contiguous()
    dest = P.route_batch(ctx, [dplans.get(vmap.get(p)) for p in pols], pols, seeds, R, d_u64(keys), 777, B, load,
                         rings=drings)
    ctx.sync()
    for i, p in enumerate(pols):
        assert (h_u16(dest[i]) == ref_dest[i]).all(), (i, p)
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("R", [1, 30, 1024, 8191])
@pytest.mark.parametrize("g0,seed", [(0, 2**64 - 1000), (2**40 + 3, 2**64 - 2**40 - 2500), (2**33, 7), (0, 0)])
def test_route_rr_hash_index_edges(P, ctx, R, g0, seed):
    # round robin is (g0 + i + seed) mod 2^64 mod R: the sum wraps inside the call for the
    # first two seeds, and request indices start above 2^32 for the second and third
    rng = np.random.default_rng(R)
    keys = rng.integers(0, 2**63, 5000, dtype=np.int64).astype(np.uint64)
    pols, seeds = ["RR", "HASH", "P2C"], [seed, seed ^ 5, seed]
    ref_dest, ref_load = O.route([None] * 3, pols, seeds, R, keys, g0, 1024)
    load = torch.zeros((3, R), dtype=torch.int64, device=DEV)
    dest = P.route_batch(ctx, [None] * 3, pols, seeds, R, d_u64(keys), g0, 1024, load)
    ctx.sync()
    for i, p in enumerate(pols):
        assert (h_u16(dest[i]) == ref_dest[i]).all(), p
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("R,V,seed", [(1, 1, 0), (3, 1, 0), (7, 5, 123), (1024, 64, 9), (8192, 16, 2**64 - 1),
                                      (5, 1024, 77)])
def test_ring_parity(P, ctx, R, V, seed):
    pt, ow = P.Ring(ctx, R, V, seed).export()
    opt, oow = O.Ring(R, V, seed).export()
    assert (pt == opt).all() and (ow == oow).all()


def _inv_mix(z):
    m64 = (1 << 64) - 1

    def unxs(y, s):
        x = y
        for _ in range(64 // s + 1):
            x = y ^ (x >> s)
        return x & m64
    z = unxs(z, 31)
    z = (z * pow(0x94D049BB133111EB, -1, 1 << 64)) & m64
    z = unxs(z, 27)
    z = (z * pow(0xBF58476D1CE4E5B9, -1, 1 << 64)) & m64
    return unxs(z, 30)


@pytest.mark.parametrize("R,V,B", [(2, 1, 1), (13, 3, 1), (13, 3, 4), (600, 8, 1), (600, 8, 1000)])
def test_route_chwbl_ring_edges(P, ctx, R, V, B):
    # keys exactly on ring points, one past a point, past the last point (wrap), on a
    # half-saturated fleet, so walks run past destinations at their bound
    rng = np.random.default_rng(R + B)
    rs, ks = 2**62 + R, 12345
    opt, _ = O.Ring(R, V, rs).export()
    edge = []
    for p in [int(x) for x in opt[:4]] + [int(x) for x in opt[-4:]]:
        edge += [_inv_mix(p) ^ ks, _inv_mix((p + 1) % 2**64) ^ ks]
    edge += [_inv_mix(2**64 - 1) ^ ks, _inv_mix(0) ^ ks]
    hot = rng.integers(0, 2**63, 8, dtype=np.int64).astype(np.uint64)
    keys = np.concatenate([np.array(edge, np.uint64), hot[rng.integers(0, 8, 5000)],
                           rng.integers(0, 2**63, 3000, dtype=np.int64).astype(np.uint64)])
    rng.shuffle(keys)
    init = np.zeros((1, R), np.uint64)
    init[0, : R // 2] = rng.integers(0, 30, R // 2).astype(np.uint64) + np.uint64(keys.size // R)
    ref_dest, ref_load = O.route([None], ["CHWBL"], [ks], R, keys, 5, B, load=init, rings=[O.Ring(R, V, rs)])
    load = d_u64(init.reshape(-1)).view(1, R).contiguous()
    dest = P.route_batch(ctx, [None], ["CHWBL"], [ks], R, d_u64(keys), 5, B, load, rings=[P.Ring(ctx, R, V, rs)])
    ctx.sync()
    assert (h_u16(dest) == ref_dest).all()
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("B", [1, 2, 3, 16, 32])
def test_route_small_batches_one_hot_key(P, ctx, B):
    # every request carries the same replicated key: every lane of a warp step competes
    # for the same members, the slowest case of the fixed-point resolution
    R, W = 64, 2
    keys = np.concatenate([np.full(20000, 0xDEADBEEF, np.uint64), np.arange(1, 2001, dtype=np.uint64)])
    num, den = 1, 1  # q_cap = 1: k_b = min(R, lambda) -> all R destinations
    opl = O.build_plan(keys, R, W, num, den)
    dpl = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, num, den))
    pols, seeds = ["CR", "P2C", "CHWBL"], [0, 1, 2]
    ref_dest, ref_load = O.route([opl, None, None], pols, seeds, R, keys, 0, B,
                                 rings=[None, None, O.Ring(R, 4, 3)])
    load = torch.zeros((3, R), dtype=torch.int64, device=DEV)
    dest = P.route_batch(ctx, [dpl, None, None], pols, seeds, R, d_u64(keys), 0, B, load,
                         rings=[None, None, P.Ring(ctx, R, 4, 3)])
    ctx.sync()
    assert (h_u16(dest) == ref_dest).all()
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("R,B,n", [(1, 1, 257), (2, 31, 1), (31, 1, 255), (32, 5, 4099), (33, 1, 4099), (257, 16, 2049)])
@pytest.mark.parametrize("loads", ["zero", "high", "spread", "huge"])
def test_route_small_batches_load_ranges(P, ctx, R, B, n, loads):
    # the 32-bit loops (loads within 2^30 of the least, also far from zero) and the 64-bit one, on
    # both sides of the 32-destination ring path, with chunks and steps cut short
    rng = np.random.default_rng(R * 31 + n)
    hot = rng.integers(1, 2**63, 12, dtype=np.int64).astype(np.uint64)
    keys = np.where(rng.random(n) < 0.5, hot[rng.integers(0, 12, n)],
                    rng.integers(1, 2**63, n, dtype=np.int64).astype(np.uint64))
    pols, seeds = ["CR", "P2C", "CHWBL", "CHWBL"], [3, 1, 2, 7]
    opl = O.build_plan(keys, R, 4, max(1, n // 40), 1)   # the hot keys take several destinations
    dpl = P.build_plan(ctx, d_u64(keys), P.plan_params(R, 4, max(1, n // 40), 1))
    orings = [None, None, O.Ring(R, 64, 5), O.Ring(R, 1, 6)]
    drings = [None, None, P.Ring(ctx, R, 64, 5), P.Ring(ctx, R, 1, 6)]
    init = rng.integers(0, 9, (4, R)).astype(np.uint64)
    if loads == "high":
        init += np.uint64(2**46)
    elif loads == "spread":
        init[:, : (R + 1) // 2] += np.uint64(2**30)
    elif loads == "huge":
        init += np.uint64(2**48)
    ref_dest, ref_load = O.route([opl, None, None, None], pols, seeds, R, keys, 99, B, load=init, rings=orings)
    load = d_u64(init.reshape(-1)).view(4, R).contiguous()
    dest = P.route_batch(ctx, [dpl, None, None, None], pols, seeds, R, d_u64(keys), 99, B, load, rings=drings)
    ctx.sync()
    assert (h_u16(dest) == ref_dest).all()
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("R", [31, 700])
@pytest.mark.parametrize("B", [33, 700, 1024, 1025, 4096, 4097])
@pytest.mark.parametrize("loads", ["zero", "high", "limit", "spread"])
def test_route_batches_load_ranges(P, ctx, R, B, loads):
    # batches of more than 32: the loop on 32-bit relative loads (one request per thread and
    # batch up to 1024, up to four above) and the 64-bit one that larger batches and loads
    # 2^32 - n or more apart take; keys with short and long member lists, some of them met
    # only in a later staging chunk
    rng = np.random.default_rng(R + B)
    n = 37000
    hot = rng.integers(1, 2**63, 14, dtype=np.int64).astype(np.uint64)
    planned = np.concatenate([np.repeat(hot, 40 * (1 + np.arange(14) * 2)),
                              rng.integers(1, 2**63, 900, dtype=np.int64).astype(np.uint64)])
    opl = O.build_plan(planned, R, 4, 12, 1)   # k_b = ceil(lambda / 12): 4 .. 90, at most R
    dpl = P.build_plan(ctx, d_u64(planned), P.plan_params(R, 4, 12, 1))
    assert 1 < np.asarray(opl.adm_k).max() <= R
    keys = planned[rng.integers(0, planned.size, n)]
    keys[:20000] = np.where(np.isin(keys[:20000], hot[8:]), hot[0], keys[:20000])
    fresh = rng.random(n) < 0.3
    keys[fresh] = rng.integers(1, 2**63, int(fresh.sum()), dtype=np.int64).astype(np.uint64)
    pols, seeds = ["CR", "P2C", "CHWBL", "CR"], [3, 1, 2, 7]
    init = rng.integers(0, 9, (4, R)).astype(np.uint64)
    if loads == "high":
        init += np.uint64(2**47)
    elif loads == "limit":
        init[:, 0] = np.uint64(2**32 - 2 - n)  # the largest difference of the 32-bit loop
        init[:, 1] = 0
    elif loads == "spread":
        init[:, : (R + 1) // 2] += np.uint64(2**32)
    orings = [None, None, O.Ring(R, 16, 5), None]
    drings = [None, None, P.Ring(ctx, R, 16, 5), None]
    ref_dest, ref_load = O.route([opl, None, None, opl], pols, seeds, R, keys, 99, B, load=init, rings=orings)
    load = d_u64(init.reshape(-1)).view(4, R).contiguous()
    dest = P.route_batch(ctx, [dpl, None, None, dpl], pols, seeds, R, d_u64(keys), 99, B, load, rings=drings)
    ctx.sync()
    assert (h_u16(dest) == ref_dest).all()
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("B", [32, 33, 1024, 4097])
@pytest.mark.parametrize("room", [9000, 8999, 150])
def test_route_loads_that_wrap(P, ctx, B, room):
    # loads at most `room` requests below 2^64 - 1: all 9,000 just fit at one destination, one
    # more than fits, or most destinations wrap to 0 on the way and are the least loaded after
    rng = np.random.default_rng(B + room)
    n, R = 9000, 30
    hot = rng.choice(2**62, 40, replace=False).astype(np.uint64)
    keys = np.where(rng.random(n) < 0.6, hot[rng.integers(0, 40, n)], rng.integers(1, 2**63, n).astype(np.uint64))
    opl = O.build_plan(keys, R, 4, n, 200)
    dpl = P.build_plan(ctx, d_u64(keys), P.plan_params(R, 4, n, 200))
    assert opl.adm_k.max() > 1
    init = np.uint64(2**64 - 1 - room) - rng.integers(0, 50, (2, R)).astype(np.uint64)
    init[:, 3] = 2**64 - 1 - room
    if room < 1000:
        init += rng.integers(0, room, (2, R)).astype(np.uint64)
    ref_dest, ref_load = O.route([opl, None], ["CR", "P2C"], [3, 1], R, keys, 99, B, load=init)
    assert (ref_load < np.uint64(2**32)).any() == (room < 1000)
    load = d_u64(init.reshape(-1)).view(2, R).contiguous()
    dest = P.route_batch(ctx, [dpl, None], ["CR", "P2C"], [3, 1], R, d_u64(keys), 99, B, load)
    ctx.sync()
    assert (h_u16(dest) == ref_dest).all()
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("case", ["few", "many", "pool", "wide"])
@pytest.mark.parametrize("B", [100, 1024])
def test_route_replicated_keys_per_batch(P, ctx, case, B):
    # keys with k_b > 1 decided once per batch from a shared-memory cache of their member
    # lists: a few such keys; more keys than the cache holds (300); member lists larger than
    # its pool (two keys on every one of 4096 destinations); and R = 8192, where the cache
    # does not fit beside the loads.  q_cap = 1, so a key seen c times gets k_b = min(c, R).
    rng = np.random.default_rng(B + len(case))
    R, W = {"few": (64, 64), "many": (64, 64), "pool": (4096, 2), "wide": (8192, 1)}[case]
    counts = {"few": [2, 3, 5, 8, 13, 21, 34, 55, 64, 64], "many": [2] * 300 + [3] * 20,
              "pool": [4096, 4096], "wide": [7, 300, 2]}[case]
    ks = rng.integers(1, 2**63, len(counts) + 30000, dtype=np.int64).astype(np.uint64)
    keys = np.concatenate([np.repeat(ks[: len(counts)], counts), ks[len(counts):]])
    rng.shuffle(keys)
    pols, seeds = ["CR", "CR_NOLPT", "CR_NOREPL", "P2C", "CR"], [0, 1, 0, 2, 3]
    vmap = {"CR": ("LPT", 0), "CR_NOLPT": ("RANDOM", 1), "CR_NOREPL": ("NOREPL", 0)}
    opl = {p: O.build_plan(keys, R, W, 1, 1, variant=v, seed=s, epoch=0) for p, (v, s) in vmap.items()}
    dpl = {p: P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, 1, 1, v, seed=s, epoch=0))
           for p, (v, s) in vmap.items()}
    assert (np.asarray(opl["CR"].adm_k) > 1).sum() >= min(len(counts), 2)
    init = rng.integers(0, 9, size=(len(pols), R)).astype(np.uint64)
    ref_dest, ref_load = O.route([opl.get(p) for p in pols], pols, seeds, R, keys, 11, B, load=init)
    load = d_u64(init.reshape(-1)).view(len(pols), R).contiguous()
    dest = P.route_batch(ctx, [dpl.get(p) for p in pols], pols, seeds, R, d_u64(keys), 11, B, load)
    ctx.sync()
    for i, p in enumerate(pols):
        assert (h_u16(dest[i]) == ref_dest[i]).all(), (i, p)
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("R,W,counts", [(64, 64, [2] * 256), (64, 64, [2] * 257), (64, 64, [15] * 100 + [16] * 100 + [2] * 57),
                                        (512, 64, [40] * 300 + [17] * 40 + [16] * 40 + [15] * 40 + [2] * 400),
                                        (8192, 2, [40] * 200 + [16] * 100 + [3] * 700)])
@pytest.mark.parametrize("B", [33, 1024, 1030])
def test_route_more_replicated_keys_than_tracked(P, ctx, R, W, counts, B):
    # at most 256 keys with k_b > 1: all may be tracked; more: only those with 16 members or more,
    # as many of them as there is room for.  q_cap = 1, so a key seen c times gets k_b = min(c, R).
    rng = np.random.default_rng(B + len(counts))
    ks = rng.choice(2**62, len(counts) + 5000, replace=False).astype(np.uint64)
    keys = np.concatenate([np.repeat(ks[: len(counts)], counts), ks[len(counts):]])
    rng.shuffle(keys)
    opl = O.build_plan(keys, R, W, 1, 1)
    dpl = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, 1, 1))
    assert (np.asarray(opl.adm_k) > 1).sum() == len(counts)
    init = rng.integers(0, 9, (2, R)).astype(np.uint64)
    ref_dest, ref_load = O.route([opl, opl], ["CR", "CR"], [0, 3], R, keys, 11, B, load=init)
    load = d_u64(init.reshape(-1)).view(2, R).contiguous()
    dest = P.route_batch(ctx, [dpl, dpl], ["CR", "CR"], [0, 3], R, d_u64(keys), 11, B, load)
    ctx.sync()
    assert (h_u16(dest) == ref_dest).all()
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("B", [1025, 2047, 2048, 2049, 3073, 4098, 5001, 8200, 16381])
def test_route_batch_remainders(P, ctx, B):
    # batches of one to many requests per thread: four, two or one at a time, and staging chunks
    # of whole quadruples (16-byte copies) or not
    rng = np.random.default_rng(B)
    n, R = 20011, 31
    hot = rng.choice(2**62, 60, replace=False).astype(np.uint64)
    keys = np.where(rng.random(n) < 0.7, hot[rng.integers(0, 60, n)], rng.integers(1, 2**63, n).astype(np.uint64))
    opl = O.build_plan(keys, R, 6, n, 100)
    dpl = P.build_plan(ctx, d_u64(keys), P.plan_params(R, 6, n, 100))
    init = rng.integers(0, 9, (2, R)).astype(np.uint64)
    ref_dest, ref_load = O.route([opl, None], ["CR", "P2C"], [0, 3], R, keys, 11, B, load=init)
    load = d_u64(init.reshape(-1)).view(2, R).contiguous()
    dest = P.route_batch(ctx, [dpl, None], ["CR", "P2C"], [0, 3], R, d_u64(keys), 11, B, load)
    ctx.sync()
    assert (h_u16(dest) == ref_dest).all()
    assert (h_u64(load) == ref_load).all()


@pytest.mark.parametrize("R", [1, 2, 3, 5, 6, 8, 9, 17, 32])
@pytest.mark.parametrize("B", [1, 5, 32])
def test_route_bounded_loads_few_destinations(P, ctx, R, B):
    # steps of at most 32 requests: the list of a walk's owners ends before all are met (rings of
    # one point per destination or of many), and a few hot keys fill the first ones
    rng = np.random.default_rng(40 * R + B)
    keys = rng.choice(2**62, 4, replace=False).astype(np.uint64)[rng.integers(0, 4, 3001)]
    keys[rng.random(3001) < 0.2] = rng.integers(1, 2**63)
    V = [1, 3, 100]
    pols, seeds = ["CHWBL"] * 3, [0, 1, 2]
    init = np.zeros((3, R), np.uint64)
    init[:, : R // 2] = 40
    ref_dest, ref_load = O.route([None] * 3, pols, seeds, R, keys, 11, B, load=init, rings=[O.Ring(R, v, 7) for v in V])
    load = d_u64(init.reshape(-1)).view(3, R).contiguous()
    dest = P.route_batch(ctx, [None] * 3, pols, seeds, R, d_u64(keys), 11, B, load, rings=[P.Ring(ctx, R, v, 7) for v in V])
    ctx.sync()
    assert (h_u16(dest) == ref_dest).all()
    assert (h_u64(load) == ref_load).all()


def test_route_rejects_bad_args(P, ctx):
    keys = d_u64(np.array([1, 2, 3], np.uint64))
    load = torch.zeros((1, 4), dtype=torch.int64, device=DEV)
    with pytest.raises(P.CacheRouteError):
        P.route_batch(ctx, [None], ["CR"], [0], 4, keys, 0, 16, load)       # plan missing
    with pytest.raises(P.CacheRouteError):
        P.route_batch(ctx, [None], ["P2C"], [0], 4, keys, 0, 0, load)       # B = 0
    with pytest.raises(P.CacheRouteError):
        P.route_batch(ctx, [None], ["P2C"], [0], 0, keys, 0, 4, load)       # R = 0
    with pytest.raises(P.CacheRouteError):
        P.route_batch(ctx, [None], ["CHWBL"], [0], 4, keys, 0, 1, load)     # ring missing
    with pytest.raises(P.CacheRouteError):
        P.route_batch(ctx, [None], ["CHWBL"], [0], 4, keys, 0, 1, load, rings=[P.Ring(ctx, 5, 2, 0)])  # R differs
    with pytest.raises(P.CacheRouteError):
        P.Ring(ctx, 4, 0, 0)                                                # no points
    with pytest.raises(P.CacheRouteError):
        P.Ring(ctx, 4, P.MAX_VNODES + 1, 0)


# ------------------------------------------------------------------ a8, a9 ---
@pytest.mark.parametrize("caps", [[1], [2, 16], [12], [32], [33], [64, 256, 1024], [5, 33, 100], [1024],
                                  [1, 40, 64], [2, 2, 50], [256, 64], [1, 2, 3, 4, 5, 6, 7, 40]])
def test_replay_parity(P, ctx, caps):
    rng = np.random.default_rng(sum(caps))
    n_rep, R = 3, 5
    n = 20000
    keys = _rates_keys(rng, int(rng.integers(20, 3000)), n)[:n]
    n = keys.size
    plen = rng.integers(16, 5000, size=n).astype(np.uint32)
    slen = np.full(n, 64, np.uint32)
    dest = tg.random_dest(n_rep, n, R, 3)
    orp = O.Replay(n_rep, R, caps)
    rp = P.Replay(ctx, n_rep, R, caps)
    ctr = torch.zeros((n_rep, len(caps), R, 5), dtype=torch.int64, device=DEV)
    dk, dp, ds, dd = d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest)
    # two calls: state persists across them
    cut = n // 3
    for a, b in ((0, cut), (cut, n)):
        orp.step(keys[a:b], plen[a:b], slen[a:b], dest[:, a:b])
        P.shadow_replay(ctx, rp, dk[a:b].contiguous(), dp[a:b].contiguous(), ds[a:b].contiguous(),
                        dd[:, a:b].contiguous(), ctr)
        ctx.sync()
        assert (h_u64(ctr) == orp.ctr).all()
    cmax = max(caps)
    for rep in range(n_rep):
        for r in range(R):
            st = rp.state(rep, r)
            ci = caps.index(cmax)
            assert (st == orp.state(rep, ci, r)).all()
            for c_i, c in enumerate(caps):
                assert (st[:c] == orp.state(rep, c_i, r)).all()


@pytest.mark.parametrize("nkeys", [1500, 6000])
def test_replay_parity_long_streams(P, ctx, nkeys):
    # streams far longer than any chunk the replay splits work into (> 16,384 requests per
    # stream per call), at the Large configuration's capacities: the state each chunk starts
    # from must be rebuilt exactly, in both calls (the second starts from persisted state)
    rng = np.random.default_rng(nkeys)
    caps = [64, 256, 1024]
    n_rep, R = 2, 2
    keys = _rates_keys(rng, nkeys, 130000, skew=0.9)
    n = keys.size
    plen = rng.integers(16, 5000, size=n).astype(np.uint32)
    slen = np.full(n, 64, np.uint32)
    dest = tg.random_dest(n_rep, n, R, 11)
    orp = O.Replay(n_rep, R, caps)
    rp = P.Replay(ctx, n_rep, R, caps)
    ctr = torch.zeros((n_rep, len(caps), R, 5), dtype=torch.int64, device=DEV)
    dk, dp, ds, dd = d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest)
    cut = n // 3
    for a, b in ((0, cut), (cut, n)):
        per_stream = np.bincount(dest[0, a:b], minlength=R)
        assert per_stream.min() > 16384
        orp.step(keys[a:b], plen[a:b], slen[a:b], dest[:, a:b])
        P.shadow_replay(ctx, rp, dk[a:b].contiguous(), dp[a:b].contiguous(), ds[a:b].contiguous(),
                        dd[:, a:b].contiguous(), ctr)
        ctx.sync()
        got = h_u64(ctr)
        assert (got == orp.ctr).all()
        assert 0 < got[:, 0, :, 1].sum() < got[:, 2, :, 1].sum() < got[:, 2, :, 0].sum()  # hits differ by cap
    for rep in range(n_rep):
        for r in range(R):
            st = rp.state(rep, r)
            for c_i, c in enumerate(caps):
                assert (st[:c] == orp.state(rep, c_i, r)).all()


def test_replay_reset_and_bad_dest(P, ctx):
    rp = P.Replay(ctx, 1, 4, [8])
    keys = d_u64(np.arange(10, dtype=np.uint64))
    plen = d_u32(np.full(10, 5, np.uint32))
    dest = d_u16(np.array([[0, 1, 2, 3, 0, 1, 2, 3, 0, 9]], np.uint16))   # 9 >= R
    ctr = torch.zeros((1, 1, 4, 5), dtype=torch.int64, device=DEV)
    P.shadow_replay(ctx, rp, keys, plen, plen, dest, ctr)
    with pytest.raises(P.CacheRouteError):
        ctx.sync()
    assert int(ctr[..., 0].sum()) == 9
    rp.reset()
    ctx.sync()
    assert rp.state(0, 0).size == 0


# ------------------------------------------------------------------ pipeline ---
@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("name,n,nint", [("tiny", 20000, 1), ("70b", 30000, 3), ("8b", 6000, 4),
                                          ("burst", 30000, 2), ("70b-gamma", 30000, 3)])
def test_pipeline_parity(P, ctx, name, n, nint, overlap):
    from paper_2608_19677_gb300.pipeline import Pipeline
    cfg = tg.CONFIGS[name]
    if name != "tiny":
        cfg = cfg.scaled(n, nint)
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=1024, keep=True)
    pipe = Pipeline(ctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, batch_B=1024, overlap=overlap)
    for rep in range(2):          # twice: reset() must restore the initial state
        pipe.reset()
        for t in range(cfg.n_intervals):
            iv = tr.interval(t)
            tok, off = tg.arena_host(tr, iv, 4)
            keys = pipe.interval(t, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen), d_u32(iv.slen),
                                 iv.g0, plan_next=t + 1 < cfg.n_intervals)
            assert (h_u64(keys) == ref["keys"][t]).all()
            pipe.wait_last()
            assert (h_u16(pipe.last_dest) == ref["dest"][t]).all()
            # the plans the interval was routed with equal the oracle's
            for (v, s), pl in zip(pipe.plan_keys, pipe.last_plans):
                opl = ref["plans"][t][(v, s)]
                got = pl.export()
                assert got["n_adm"] == opl.n_adm and (got["members"] == opl.members).all()
        pipe.sync()
        assert (h_u64(pipe.ctr) == ref["ctr"]).all()


@pytest.mark.parametrize("name,n,nint,depth,ps,rs,grp", [("70b", 40000, 6, 3, 2, 2, 1), ("8b", 8000, 9, 4, 3, 2, 1),
                                                          ("burst", 40000, 4, 2, 1, 3, 1),
                                                          ("large", 200000, 3, 8, 4, 4, 1),
                                                          ("tiny", 20000, 1, 8, 4, 4, 1),
                                                          ("70b", 40000, 7, 4, 2, 3, 3), ("8b", 8000, 9, 6, 2, 2, 4),
                                                          ("large", 200000, 3, 8, 4, 4, 2)])
def test_trace_pipeline_parity(P, ctx, name, n, nint, depth, ps, rs, grp):
    # several intervals in flight (plans and routes on several streams, the replay in order):
    # every interval's plans and destinations, and the counters, equal the oracle's
    from paper_2608_19677_gb300.pipeline import TracePipeline
    cfg = tg.CONFIGS[name]
    if name != "tiny":
        cfg = cfg.scaled(n, nint)
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=1024, keep=True)
    ivs = [tr.interval(t) for t in range(cfg.n_intervals)]
    keys = [d_u64(k) for k in ref["keys"]]
    plens = [d_u32(iv.plen) for iv in ivs]
    slens = [d_u32(iv.slen) for iv in ivs]
    pipe = TracePipeline(ctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, max_n=max(iv.n for iv in ivs),
                         batch_B=1024, depth=depth, plan_streams=ps, route_streams=rs, vnodes=cfg.vnodes,
                         replay_group=grp)
    for rep in range(2):   # twice: reset() restores the initial state
        pipe.reset()
        seen = []

        def check(t, dest, plans):
            pipe.sync()
            seen.append(t)
            assert (h_u16(dest) == ref["dest"][t]).all(), f"interval {t}: destinations differ"
            for (v, s_), pl in zip(pipe.plan_keys, plans):
                opl = ref["plans"][t][(v, s_)]
                got = pl.export()
                assert got["n_adm"] == opl.n_adm and (got["members"] == opl.members).all()
        pipe.run(keys, plens, slens, [iv.g0 for iv in ivs], on_interval=check if rep == 0 else None)
        pipe.sync()
        assert (h_u64(pipe.ctr) == ref["ctr"]).all()
    pipe.close()


@pytest.mark.parametrize("name,grp", [("8b", 4), ("70b", 2)])
def test_trace_pipeline_cuda_graph(P, ctx, name, grp):
    # the whole trace (reset + every interval's plans, routes and replay, on many streams)
    # captured once as a CUDA graph: each replay gives the oracle's counters again
    from paper_2608_19677_gb300.pipeline import TracePipeline
    cfg = tg.CONFIGS[name].scaled(40000, 8)
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=1024, keep=True)
    ivs = [tr.interval(t) for t in range(cfg.n_intervals)]
    keys = [d_u64(k) for k in ref["keys"]]
    plens = [d_u32(iv.plen) for iv in ivs]
    slens = [d_u32(iv.slen) for iv in ivs]
    g0s = [iv.g0 for iv in ivs]
    stream = torch.cuda.Stream()       # a graph is captured on a stream other than the default one
    gctx = P.Context(0, stream)
    pipe = TracePipeline(gctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, max_n=max(iv.n for iv in ivs),
                         batch_B=1024, depth=4, plan_streams=3, route_streams=2, vnodes=cfg.vnodes,
                         replay_group=grp)
    pipe.reset()
    pipe.run(keys, plens, slens, g0s)   # warm-up: scratch and inputs reach their sizes
    pipe.quiesce()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        pipe.reset()
        pipe.run(keys, plens, slens, g0s)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert (h_u64(pipe.ctr) == ref["ctr"]).all()
    del graph
    pipe.close()
    gctx.close()


@pytest.mark.parametrize("B", [1, 7, 1024])
def test_pipeline_parity_bounded_load_and_small_batches(P, ctx, B):
    # the 70B shape with the bounded-load comparison policy added, routed in
    # batches of 1 (exact sequential), 7 and 1024 requests
    import dataclasses
    from paper_2608_19677_gb300.pipeline import Pipeline
    cfg = dataclasses.replace(tg.CONFIGS["70b"].scaled(20000, 2), policies=["CR", "P2C", "HASH", "CHWBL"],
                              seeds=[0, 3])
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=B, keep=True)
    pipe = Pipeline(ctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, batch_B=B, overlap=True,
                    vnodes=cfg.vnodes)
    for t in range(cfg.n_intervals):
        iv = tr.interval(t)
        tok, off = tg.arena_host(tr, iv, 4)
        pipe.interval(t, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen), d_u32(iv.slen), iv.g0,
                      plan_next=t + 1 < cfg.n_intervals)
        pipe.wait_last()
        assert (h_u16(pipe.last_dest) == ref["dest"][t]).all()
    pipe.sync()
    assert (h_u64(pipe.ctr) == ref["ctr"]).all()


# ------------------------------------------------------------------ f2 replanning ---
def _diff_case(P, ctx, keys_a, keys_b, R, W, num_den_a, num_den_b, var_a="LPT", var_b="LPT"):
    oa = O.build_plan(keys_a, R, W, *num_den_a, variant=var_a, seed=1, epoch=0)
    ob = O.build_plan(keys_b, R, W, *num_den_b, variant=var_b, seed=2, epoch=1)
    da = P.build_plan(ctx, d_u64(keys_a), P.plan_params(R, W, *num_den_a, var_a, seed=1, epoch=0))
    db = P.build_plan(ctx, d_u64(keys_b), P.plan_params(R, W, *num_den_b, var_b, seed=2, epoch=1))
    got = P.plan_diff(ctx, da, db)
    want = O.plan_diff(oa, ob)
    assert got == want
    assert P.plan_diff(ctx, db, da) == O.plan_diff(ob, oa)
    assert P.plan_diff(ctx, da, da) == O.plan_diff(oa, oa)
    return got


@pytest.mark.parametrize("t", range(5))
def test_plan_diff_drift_transitions(P, ctx, t):
    # consecutive fresh LPT plans of the drift trace (70B shape, lognormal rate walk)
    cfg = tg.CONFIGS["drift"]
    tr = tg.Trace(cfg)
    ka = O.hash_prefixes(*tg.arena_host(tr, tr.interval(t), 4), tr.interval(t).plen)
    kb = O.hash_prefixes(*tg.arena_host(tr, tr.interval(t + 1), 4), tr.interval(t + 1).plen)
    d = _diff_case(P, ctx, ka, kb, cfg.R, cfg.W, tr.qcap(ka.size), tr.qcap(kb.size))
    cache, count = O.churn(d)
    assert 0 < cache <= 1 and 0 <= count < 1


@pytest.mark.parametrize("R,W,spread", [(1, 4, 50), (7, 3, 400), (64, 8, 3000), (1024, 16, 20000),
                                        (8192, 2, 30000)])
def test_plan_diff_shapes(P, ctx, R, W, spread):
    rng = np.random.default_rng(R)
    ka = _rates_keys(rng, spread, 60000)
    kb = np.concatenate([ka[: ka.size // 2], _rates_keys(rng, spread, 30000)])  # half the traffic changes
    n = ka.size
    _diff_case(P, ctx, ka, kb, R, W, (n, 4 * R), (n, 3 * R), "LPT", "RANDOM")  # replicated keys, k_b up to R


def test_plan_diff_empty_and_errors(P, ctx):
    keys = np.arange(1, 500, dtype=np.uint64) * np.uint64(7919)
    e = np.zeros(0, np.uint64)
    _diff_case(P, ctx, e, keys, 16, 4, (1, 1), (keys.size, 64))
    _diff_case(P, ctx, e, e, 16, 4, (1, 1), (1, 1))
    a = P.build_plan(ctx, d_u64(keys), P.plan_params(16, 4, keys.size, 64))
    b = P.build_plan(ctx, d_u64(keys), P.plan_params(17, 4, keys.size, 64))
    with pytest.raises(P.CacheRouteError):
        P.plan_diff(ctx, a, b)                                              # R differs
    with pytest.raises(P.CacheRouteError):
        P.plan_diff(ctx, a, P.Plan(ctx))                                    # not built


@pytest.mark.parametrize("fresh", [True, False])
def test_pipeline_parity_drift_fresh_and_stale(P, ctx, fresh):
    # the replanning comparison: every interval routed with a plan from its own keys
    # (fresh) or from the previous interval's (stale), replayed through persistent LRUs
    from paper_2608_19677_gb300.pipeline import Pipeline
    cfg = tg.CONFIGS["drift"].scaled(60000, 6)
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=1024, keep=True, fresh=fresh)
    pipe = Pipeline(ctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, batch_B=1024, overlap=True, fresh=fresh)
    for t in range(cfg.n_intervals):
        iv = tr.interval(t)
        tok, off = tg.arena_host(tr, iv, 4)
        pipe.interval(t, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen), d_u32(iv.slen), iv.g0,
                      plan_next=t + 1 < cfg.n_intervals)
        pipe.wait_last()
        assert (h_u16(pipe.last_dest) == ref["dest"][t]).all()
        for (v, s), pl in zip(pipe.plan_keys, pipe.last_plans):
            got = pl.export()
            opl = ref["plans"][t][(v, s)]
            assert got["n_adm"] == opl.n_adm and (got["members"] == opl.members).all()
    pipe.sync()
    assert (h_u64(pipe.ctr) == ref["ctr"]).all()


# ------------------------------------------------------------------ f3 token-weighted replay ---
def _fixed_len_stream(rng, n, nkeys, lo=16, hi=5000, spread=1.2):
    keys = _rates_keys(rng, nkeys, n, skew=spread)[:n]
    uk, inv = np.unique(keys, return_inverse=True)
    size_of = rng.integers(lo, hi, size=uk.size).astype(np.uint32)  # one prefix length per key
    return keys, size_of[inv]


@pytest.mark.parametrize("caps,lo,hi", [([24576], 16, 5000), ([1, 100, 3000], 16, 5000),
                                        ([4096, 65536, 2 ** 31], 16, 200),       # 1024-prefix bound
                                        ([5000, 10 ** 6], 1, 3)])
def test_token_replay_parity(P, ctx, caps, lo, hi):
    rng = np.random.default_rng(sum(caps) % 1000 + lo)
    n_rep, R, n = 3, 7, 24000
    keys, plen = _fixed_len_stream(rng, n, int(rng.integers(50, 3000)), lo, hi)
    n = keys.size
    slen = rng.integers(0, 200, size=n).astype(np.uint32)
    dest = tg.random_dest(n_rep, n, R, 5)
    orp = O.Replay(n_rep, R, caps, tokens=True)
    rp = P.Replay(ctx, n_rep, R, caps, tokens=True)
    ctr = torch.zeros((n_rep, len(caps), R, 5), dtype=torch.int64, device=DEV)
    dk, dp, ds, dd = d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest)
    cut = n // 3
    for a, b in ((0, cut), (cut, n)):  # state persists across calls
        orp.step(keys[a:b], plen[a:b], slen[a:b], dest[:, a:b])
        P.shadow_replay(ctx, rp, dk[a:b].contiguous(), dp[a:b].contiguous(), ds[a:b].contiguous(),
                        dd[:, a:b].contiguous(), ctr)
        ctx.sync()
        assert (h_u64(ctr) == orp.ctr).all()
    ci = caps.index(max(caps))
    for rep in range(n_rep):
        for r in range(R):
            assert (rp.state(rep, r) == orp.state(rep, ci, r)).all()


@pytest.mark.parametrize("caps,lo,hi,nkeys", [([24576], 16, 5000, 400), ([1, 100, 3000], 16, 5000, 2000),
                                              ([4096, 65536, 2 ** 31], 16, 200, 3000)])
def test_token_replay_parity_long_streams(P, ctx, caps, lo, hi, nkeys):
    # streams much longer than the chunks the byte-aware replay splits them into: every chunk
    # after a stream's first rebuilds its starting list by walking back over the stream and
    # the carried-in list, in both calls
    rng = np.random.default_rng(nkeys + lo)
    n_rep, R, n = 2, 2, 80000
    keys, plen = _fixed_len_stream(rng, n, nkeys, lo, hi)
    n = keys.size
    slen = rng.integers(0, 200, size=n).astype(np.uint32)
    dest = tg.random_dest(n_rep, n, R, 8)
    orp = O.Replay(n_rep, R, caps, tokens=True)
    rp = P.Replay(ctx, n_rep, R, caps, tokens=True)
    ctr = torch.zeros((n_rep, len(caps), R, 5), dtype=torch.int64, device=DEV)
    dk, dp, ds, dd = d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest)
    cut = n // 3
    for a, b in ((0, cut), (cut, n)):
        if a == cut:  # the second call's streams span several chunks at every capacity tested
            assert np.bincount(dest[0, a:b], minlength=R).min() > (16384 if max(caps) > (1 << 17) else 4096)
            # (capacities up to 2^16 tokens use chunks of 1,024 requests, up to 2^17 of 4,096)
        orp.step(keys[a:b], plen[a:b], slen[a:b], dest[:, a:b])
        P.shadow_replay(ctx, rp, dk[a:b].contiguous(), dp[a:b].contiguous(), ds[a:b].contiguous(),
                        dd[:, a:b].contiguous(), ctr)
        ctx.sync()
        assert (h_u64(ctr) == orp.ctr).all()
    ci = caps.index(max(caps))
    for rep in range(n_rep):
        for r in range(R):
            assert (rp.state(rep, r) == orp.state(rep, ci, r)).all()


def test_token_replay_saturating_sums(P, ctx):
    # prefixes near 2^31 tokens: sums past 2^32 saturate and are evicted like any over-capacity run
    caps = [2 ** 31, 2 ** 30]
    keys = np.array([1, 2, 1, 3, 4, 3, 2, 1, 1, 3, 4], np.uint64)
    size = {1: 2 ** 30, 2: 2 ** 31 - 5, 3: 2 ** 31, 4: 2 ** 32 - 1}  # 3 then 4: 3's sum passes 2^32
    plen = np.array([size[int(k)] for k in keys], np.uint32)
    slen = np.zeros(keys.size, np.uint32)
    dest = np.zeros((1, keys.size), np.uint16)
    orp = O.Replay(1, 1, caps, tokens=True)
    orp.step(keys, plen, slen, dest)
    rp = P.Replay(ctx, 1, 1, caps, tokens=True)
    ctr = torch.zeros((1, 2, 1, 5), dtype=torch.int64, device=DEV)
    P.shadow_replay(ctx, rp, d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest), ctr)
    ctx.sync()
    assert (h_u64(ctr) == orp.ctr).all()
    assert (rp.state(0, 0) == orp.state(0, 0, 0)).all()
    with pytest.raises(P.CacheRouteError):
        P.Replay(ctx, 1, 1, [2 ** 31 + 1], tokens=True)


def test_token_replay_changed_length_is_reported(P, ctx):
    rp = P.Replay(ctx, 1, 2, [10000], tokens=True)
    keys = d_u64(np.array([5, 6, 5], np.uint64))
    plen = d_u32(np.array([100, 200, 150], np.uint32))  # key 5 comes back with another length
    slen = d_u32(np.zeros(3, np.uint32))
    dest = d_u16(np.zeros((1, 3), np.uint16))
    ctr = torch.zeros((1, 1, 2, 5), dtype=torch.int64, device=DEV)
    P.shadow_replay(ctx, rp, keys, plen, slen, dest, ctr)
    with pytest.raises(P.CacheRouteError):
        ctx.sync()
    rp.reset()
    P.shadow_replay(ctx, rp, keys[:2].contiguous(), plen[:2].contiguous(), slen[:2].contiguous(),
                    dest[:, :2].contiguous(), ctr)
    ctx.sync()
    assert rp.state(0, 0).tolist() == [6, 5]


@pytest.mark.parametrize("name,n,nint", [("70b", 40000, 3), ("large", 100000, 2)])
def test_pipeline_parity_token_lru(P, ctx, name, n, nint):
    from paper_2608_19677_gb300.pipeline import Pipeline
    cfg = tg.CONFIGS[name].scaled(n, nint).token_lru()
    if name == "large":  # fewer replicas keep the oracle quick; R, caps and the 1024-prefix bound stay
        import dataclasses
        cfg = dataclasses.replace(cfg, seeds=[0, 1])
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=1024, keep=True)
    pipe = Pipeline(ctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, batch_B=1024, overlap=True,
                    lru_tokens=True)
    for t in range(cfg.n_intervals):
        iv = tr.interval(t)
        tok, off = tg.arena_host(tr, iv, 4)
        pipe.interval(t, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen), d_u32(iv.slen), iv.g0,
                      plan_next=t + 1 < cfg.n_intervals)
    pipe.sync()
    assert (h_u64(pipe.ctr) == ref["ctr"]).all()


@pytest.mark.parametrize("name,n,nint", [("8b", 6000, 5), ("70b", 30000, 3)])
def test_pipeline_cuda_graph_replay(P, ctx, name, n, nint):
    # a whole step captured once as a CUDA graph (planner and replay streams joined through
    # events) gives the counters of the ordinary step, replay after replay
    from paper_2608_19677_gb300.pipeline import Pipeline
    cfg = tg.CONFIGS[name].scaled(n, nint)
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=1024)
    s = torch.cuda.Stream(DEV)
    with torch.cuda.stream(s):
        gctx = P.Context(0, s)
        ins = []
        for t in range(cfg.n_intervals):
            iv = tr.interval(t)
            tok, off = tg.arena_host(tr, iv, 4)
            ins.append((t, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen), d_u32(iv.slen), iv.g0))
        pipe = Pipeline(gctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, batch_B=1024, overlap=True,
                        max_n=max(int(x[2].shape[0]) for x in ins))

        def step():
            pipe.reset()
            for i, (t, tok, off, pl, sl, g0) in enumerate(ins):
                pipe.interval(t, tok, off, pl, sl, g0, plan_next=i + 1 < len(ins))
            pipe.finish()

        step()
        torch.cuda.synchronize()
        assert (h_u64(pipe.ctr) == ref["ctr"]).all()
        pipe.quiesce()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            step()
        for _ in range(2):
            pipe.ctr.fill_(-1)
            graph.replay()
            torch.cuda.synchronize()
            assert (h_u64(pipe.ctr) == ref["ctr"]).all()
    gctx.sync()


# ------------------------------------------------------------------ f3 slot-capped placement ---
@pytest.mark.parametrize("R,W,nkeys,total,skew", [(2, 2, 4, 127, 0), (30, 3, 3000, 60000, 1),
                                                  (300, 2, 20000, 700000, 1), (1024, 4, 60000, 300000, 0),
                                                  (3000, 1, 5000, 40000, 1)])
def test_plan_parity_slotcap(P, ctx, R, W, nkeys, total, skew):
    # the capped LPT against the oracle, on the one-CTA build and on the device-wide build
    # (700,000 requests), with and without a skewed starting load (which trims replica counts)
    rng = np.random.default_rng(R + W)
    keys = _rates_keys(rng, nkeys, total)
    n = keys.size
    init = None
    if skew:
        init = rng.integers(0, 50, R).astype(np.uint64)
        init[: max(1, R // 4)] += np.uint64(10 ** 6)
    for num, den in ((5 * n, 4 * R), (n, 20 * R)):
        dl = d_u64(init) if init is not None else None
        got = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, num, den, "SLOTCAP", init_load=dl)).export()
        ref = O.build_plan(keys, R, W, num, den, variant="SLOTCAP", init_load=init)
        _cmp_plan(got, ref)
        assert np.bincount(got["members"].astype(np.int64), minlength=R).max() <= W


@pytest.mark.parametrize("n,R,W,n_rand", [(24576, 1024, 200, 1), (24577, 1024, 8, 1), (24577, 1024, 9, 1),
                                          (70000, 1024, 64, 1), (70000, 1024, 65, 1), (70000, 1024, 65, 3),
                                          (130000, 1024, 200, 1), (130000, 16, 300, 5), (4096, 1024, 200, 1),
                                          (4097, 1024, 200, 1), (24577, 1024, 4, 1), (24577, 241, 17, 1)])
def test_plan_parity_sort_and_admission_rules(P, ctx, n, R, W, n_rand):
    # both sides of the rules on interval and slot budget: histogram sorted by one CTA (up to
    # 4,096 requests or slots) or by the whole GPU, admission of all plans by one CTA each or
    # plan by plan
    rng = np.random.default_rng(n + R + W)
    pool = rng.integers(1, 2**63, n, dtype=np.int64).astype(np.uint64)
    keys = pool[np.minimum((rng.random(n) ** 2 * n).astype(np.int64), n - 1)]
    kinds = [("LPT", 0), ("NOREPL", 0), ("SLOTCAP", 0)] + [("RANDOM", s) for s in range(n_rand)]
    params = [P.plan_params(R, W, 5 * n, 4 * R, v, seed=s, epoch=1) for v, s in kinds]
    plans = [P.Plan(ctx) for _ in kinds]
    P.build_plans(ctx, d_u64(keys), params, plans)
    for (v, s), p in zip(kinds, plans):
        _cmp_plan(p.export(), O.build_plan(keys, R, W, 5 * n, 4 * R, variant=v, seed=s, epoch=1))


@pytest.mark.parametrize("n,U", [(66000, 1), (130000, 145), (130000, 4095), (130000, 4096), (130000, 4097),
                                 (524288, 2000), (524289, 2000)])
def test_every_plan_exports_its_histogram(P, ctx, n, U):
    # builds whose admission runs plan by plan and whose plans admit differently: every plan's
    # histogram comes out in key order, whichever kernel sorted it (few keys: by count, one CTA)
    rng = np.random.default_rng(n + U)
    pool = rng.choice(2**62, U, replace=False).astype(np.uint64)
    keys = pool[np.concatenate([np.arange(U), (rng.random(n - U) ** 2 * U).astype(np.int64)])]
    rng.shuffle(keys)
    R, W = 1024, 200
    kinds = [("LPT", R, W, 5 * n, 4 * R), ("NOREPL", R, W, 5 * n, 4 * R), ("LPT", 64, 3, n, 64)][: 2 if n < 10 ** 5 else 3]
    plans = [P.Plan(ctx) for _ in kinds]
    P.build_plans(ctx, d_u64(keys), [P.plan_params(r, w, a, b, v) for v, r, w, a, b in kinds], plans)
    uk, uc = O.histogram(keys)
    for (v, r, w, a, b), p in zip(kinds, plans):
        got = p.export()
        _cmp_plan(got, O.build_plan(keys, r, w, a, b, variant=v))
        assert (got["ukey"] == uk).all() and (got["ucnt"] == uc).all()


@pytest.mark.parametrize("pattern", ["random", "small", "high", "equal"])
@pytest.mark.parametrize("U", [4097, 6144, 6145, 32768, 32769, 70001])
def test_plan_wide_sort(P, ctx, U, pattern):
    # the sort of more than 4,096 keys by the whole GPU, at the edges of its tiles of 2,048: keys
    # that differ in every digit, only in the low or the high ones, counts of one to four digits
    # or all equal
    rng = np.random.default_rng(U)
    pool = {"random": rng.choice(2**62, U, replace=False).astype(np.uint64) * np.uint64(3),
            "small": np.arange(U, dtype=np.uint64), "high": np.arange(U, dtype=np.uint64) << np.uint64(44),
            "equal": np.arange(U, dtype=np.uint64) * np.uint64(2**46 + 1)}[pattern]
    cnt = np.ones(U, np.int64) if pattern == "equal" else 1 + (rng.pareto(1.0, U) * 0.7).astype(np.int64).clip(0, 70000)
    keys = np.repeat(pool, cnt)
    rng.shuffle(keys)
    n, R, W = keys.size, 64, 70  # C = 4,480
    got = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, 5 * n, 4 * R)).export()
    _cmp_plan(got, O.build_plan(keys, R, W, 5 * n, 4 * R))
    uk, uc = O.histogram(keys)
    assert (got["ukey"] == uk).all() and (got["ucnt"] == uc).all()


def test_plan_wide_sort_on_many_streams(P):
    # eight builds at once on streams of their own: a block of the sort waits only for work that
    # a running block holds, so they do not need the whole GPU to themselves
    rng = np.random.default_rng(8)
    n, R, W = 600000, 256, 256
    keys = rng.integers(0, 400000, n).astype(np.uint64) * np.uint64(0x9e3779b97f4a7c15)
    dk = d_u64(keys)
    torch.cuda.synchronize()
    ctxs = [P.Context(0, torch.cuda.Stream(DEV)) for _ in range(8)]
    plans = [P.Plan(c) for c in ctxs]
    prm = P.plan_params(R, W, 5 * n, 4 * R)
    for _ in range(5):
        for c, p in zip(ctxs, plans):
            P.build_plans(c, dk, [prm], [p])
    ref = O.build_plan(keys, R, W, 5 * n, 4 * R)
    for p in plans:
        _cmp_plan(p.export(), ref)
    for c, p in zip(ctxs, plans):
        p.close()
        c.close()


@pytest.mark.parametrize("R,W,kinds", [(1024, 66, ("SLOTCAP", "LPT")), (2048, 33, ("SLOTCAP", "LPT")),
                                       (2048, 33, ("SLOTCAP", "RANDOM")), (4096, 33, ("SLOTCAP", "SLOTCAP", "LPT", "RANDOM"))])
def test_plans_beside_a_trimmed_slotcap(P, ctx, R, W, kinds):
    # plan by plan, the slot-capped plan listed first: its replica counts are trimmed (an eighth
    # of the destinations starts too loaded to be chosen before the others are full), those of the
    # plans after it, which share its admission, are not
    rng = np.random.default_rng(R)
    lam = np.concatenate([rng.integers(R // 4, R // 3, 300), np.ones(9000, np.int64)])
    keys = np.repeat(rng.choice(2**62, lam.size, replace=False).astype(np.uint64), lam)
    rng.shuffle(keys)
    init = np.zeros(R, np.uint64)
    init[: R // 8] = 10 ** 6
    plans = [P.Plan(ctx) for _ in kinds]
    dl = d_u64(init)
    P.build_plans(ctx, d_u64(keys), [P.plan_params(R, W, 1, 1, v, seed=3, init_load=dl) for v in kinds], plans)
    refs = [O.build_plan(keys, R, W, 1, 1, variant=v, seed=3, init_load=init) for v in kinds]
    assert (refs[0].adm_k != refs[-1].adm_k).any()
    for p, ref in zip(plans, refs):
        _cmp_plan(p.export(), ref)


@pytest.mark.parametrize("R,W", [(2, 40), (33, 31), (64, 100), (700, 9), (1024, 40)])
@pytest.mark.parametrize("init", ["zero", "near", "far"])
def test_plan_parity_slotcap_runs(P, ctx, R, W, init):
    # long runs of equal counts over destinations whose slots run out one by one: every slot
    # is used, destinations start level, within a few requests, or far apart (the far ones
    # fill last), replicated keys in front
    rng = np.random.default_rng(R + W)
    C = R * W
    lam = np.concatenate([np.array([60, 41, 41, 17]), np.repeat([7, 5, 3, 2, 1], [C // 9, C // 7, C // 4, C // 3, C])])
    keys = np.repeat(rng.integers(1, 2**63, lam.size, dtype=np.int64).astype(np.uint64), lam)
    rng.shuffle(keys)
    load = None
    if init != "zero":
        load = rng.integers(0, 9, R).astype(np.uint64)
        if init == "far":
            load[:: 3] += np.uint64(2 * C)
    dl = d_u64(load) if load is not None else None
    got = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, 30, 1, "SLOTCAP", init_load=dl)).export()
    ref = O.build_plan(keys, R, W, 30, 1, variant="SLOTCAP", init_load=load)
    _cmp_plan(got, ref)
    assert np.bincount(got["members"].astype(np.int64), minlength=R).max() == W


def test_pipeline_parity_slotcap_policy(P, ctx):
    import dataclasses
    from paper_2608_19677_gb300.pipeline import Pipeline
    cfg = dataclasses.replace(tg.CONFIGS["8b"].scaled(8000, 4), policies=["CR", "CR_SLOTCAP", "P2C"], seeds=[0, 1])
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=1024, keep=True)
    pipe = Pipeline(ctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, batch_B=1024, overlap=True)
    for t in range(cfg.n_intervals):
        iv = tr.interval(t)
        tok, off = tg.arena_host(tr, iv, 4)
        pipe.interval(t, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen), d_u32(iv.slen), iv.g0,
                      plan_next=t + 1 < cfg.n_intervals)
        pipe.wait_last()
        assert (h_u16(pipe.last_dest) == ref["dest"][t]).all()
    pipe.sync()
    assert (h_u64(pipe.ctr) == ref["ctr"]).all()


@pytest.mark.parametrize("B,chwbl", [(1024, False), (1024, True), (1, True)])
def test_pipeline_split_routing_on_sm_partition(P, ctx, B, chwbl):
    # hashing and candidates on the large SM partition, the route resolution on the small one
    # (green contexts): same destinations and counters as the oracle, with the CTA resolution
    # (B = 1024) and the one-warp exact-sequential one (B = 1), with and without bounded-load
    # (ring) replicas
    import dataclasses
    from paper_2608_19677_gb300.pipeline import Pipeline
    try:
        part = P.Partition(0, 16)
    except P.CacheRouteError as e:
        pytest.skip(f"no SM partition on this driver: {e}")
    cfg = tg.CONFIGS["70b"].scaled(40000 if B > 1 else 12000, 4 if B > 1 else 2)
    if chwbl:
        cfg = dataclasses.replace(cfg, policies=["CR", "P2C", "CHWBL"], seeds=[0, 1])
    tr = tg.Trace(cfg)
    ref = OP.run_trace(tr, B=B, keep=True)
    with torch.cuda.stream(part.big):
        pctx = P.Context(0, part.big)
        pipe = Pipeline(pctx, cfg.R, cfg.W, cfg.caps, cfg.replicas, tr.qcap, batch_B=B, overlap=True,
                        resolve_stream=part.small, vnodes=cfg.vnodes)
        for t in range(cfg.n_intervals):
            iv = tr.interval(t)
            tok, off = tg.arena_host(tr, iv, 4)
            pipe.interval(t, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen), d_u32(iv.slen), iv.g0,
                          plan_next=t + 1 < cfg.n_intervals)
            pipe.wait_last()
            assert (h_u16(pipe.last_dest) == ref["dest"][t]).all()
        pipe.sync()
        assert (h_u64(pipe.ctr) == ref["ctr"]).all()
    pipe.close()  # what uses the partition's streams goes before the partition
    pctx.close()
    part.close()


def test_split_route_error_reported_by_sync(P):
    # a bounded-load replica whose load sum has wrapped past 2^64 leaves no destination below
    # cap: the resolution, enqueued on the resolve stream, raises the overflow flag, and the
    # next cr_sync must report it even though the context's own stream finished first
    c = P.Context(0)
    side = torch.cuda.Stream(DEV)
    try:
        R = 2
        ring = P.Ring(c, R, 4, 3)
        P.set_resolve_stream(c, side)
        keys = d_u64(np.arange(1, 65, dtype=np.uint64))
        # loads 2^63 and 2^63 + 2: their sum wraps to 2, so cap = ceil(5 * 3 / 8) = 2 < both
        load = d_u64(np.array([[2 ** 63, 2 ** 63 + 2]], np.uint64))
        P.route_batch(c, [None], ["CHWBL"], [5], R, keys, 0, 64, load, rings=[ring])
        with pytest.raises(P.CacheRouteError) as ei:
            c.sync()
        assert ei.value.code == P.CR_EOVERFLOW
        c.sync()   # reported once, then cleared
        P.set_resolve_stream(c, None)
        ring.close()
    finally:
        c.close()


def test_profile_events_time_each_launch(P):
    # per-launch timing: every timed kind of launch is counted once per call, with a positive duration
    c = P.Context(0)
    try:
        c.profile_enable(64)
        cfg = tg.CONFIGS["70b"].scaled(20000, 1)
        tr = tg.Trace(cfg)
        iv = tr.interval(0)
        tok, off = tg.arena_host(tr, iv, 4)
        keys = P.hash_prefixes(c, torch.from_numpy(tok).to(DEV), d_u64(off), d_u32(iv.plen))
        num, den = tr.qcap(iv.n)
        plan = P.build_plan(c, keys, P.plan_params(cfg.R, cfg.W, num, den, "LPT"))
        load = torch.zeros((2, cfg.R), dtype=torch.int64, device=DEV)
        dest = P.route_batch(c, [plan, None], ["CR", "P2C"], [0, 0], cfg.R, keys, iv.g0, 1024, load)
        rp = P.Replay(c, 2, cfg.R, cfg.caps)
        ctr = torch.zeros((2, 1, cfg.R, 5), dtype=torch.int64, device=DEV)
        P.shadow_replay(c, rp, keys, d_u32(iv.plen), d_u32(iv.slen), dest, ctr)
        c.sync()
        for tag in ("hash", "plan", "route_cand", "route_resolve", "partition", "replay"):
            n, ms = c.profile_read(tag)
            assert n == 1 and ms > 0.0, tag
        c.profile_enable(0)
        assert c.profile_read("replay") == (0, 0.0)
        import ctypes
        n_, ms_ = ctypes.c_uint64(), ctypes.c_double()
        assert P.lib().cr_profile_read(c.handle, 99, ctypes.byref(n_), ctypes.byref(ms_)) == P.CR_EINVAL
        rp.close()
        plan.close()
    finally:
        c.close()


def test_plan_import_routes_like_the_built_plan(P, ctx):
    # a plan exported from the device and installed again (as a host planner's table would
    # be) routes exactly as the plan it came from; bad tables are refused
    rng = np.random.default_rng(21)
    R, W = 64, 8
    keys = _rates_keys(rng, 3000, 60000)
    n = keys.size
    built = P.build_plan(ctx, d_u64(keys), P.plan_params(R, W, 5 * n, 4 * R, "LPT"))
    ex = built.export()
    imp = P.Plan(ctx).load(R, W, ex["adm_key"], ex["adm_cnt"], ex["adm_k"], ex["members"], ex["jobs"], ex["load"])
    got = imp.export()
    for f in ("adm_key", "adm_cnt", "adm_k", "koff", "members", "jobs", "load"):
        assert (got[f] == ex[f]).all(), f
    assert got["n_adm"] == ex["n_adm"] and got["sum_k"] == ex["sum_k"]
    load = torch.zeros((2, R), dtype=torch.int64, device=DEV)
    dk = d_u64(keys)
    d = P.route_batch(ctx, [built, imp], ["CR", "CR"], [3, 3], R, dk, 0, 1024, load)
    ctx.sync()
    h = h_u16(d)
    assert (h[0] == h[1]).all()
    # the oracle agrees with the imported plan's routes
    opl = O.build_plan(keys, R, W, 5 * n, 4 * R)
    od, _ = O.route([opl], ["CR"], [3], R, keys, 0, 1024)
    assert (h[1] == od[0]).all()
    for bad in (dict(adm_k=np.zeros_like(ex["adm_k"])),                       # k = 0
                dict(members=np.full_like(ex["members"], R)),                 # member >= R
                dict(adm_key=np.zeros_like(ex["adm_key"]))):                  # repeated key
        args = dict(adm_key=ex["adm_key"], adm_cnt=ex["adm_cnt"], adm_k=ex["adm_k"], members=ex["members"])
        args.update(bad)
        with pytest.raises(P.CacheRouteError):
            P.Plan(ctx).load(R, W, **args)


@pytest.mark.parametrize("caps", [[16], [64, 300], [1024]])
@pytest.mark.parametrize("ncoll", [9, 30, 60, 400])
def test_replay_parity_colliding_keys(P, ctx, caps, ncoll):
    # keys that share both index buckets and the tag (their products with the index's odd
    # multiplier differ in the low 22 bits only): past 8 of them the index's stash holds
    # them, past 40 it is degraded; mixed with ordinary keys, over several renumberings of
    # the window and two calls
    rng = np.random.default_rng(ncoll + sum(caps))
    inv = np.uint64(pow(0x9E3779B97F4A7C15, -1, 1 << 64))
    with np.errstate(over="ignore"):
        coll = (np.uint64(0xABCDEF0123 << 24) + rng.permutation(1 << 22)[:ncoll].astype(np.uint64)) * inv
    n_rep, R, n = 2, 2, 6000
    pool = np.concatenate([coll, _rates_keys(rng, 300, 300)])
    keys = pool[rng.integers(0, pool.size, size=n)]
    plen = rng.integers(16, 5000, size=n).astype(np.uint32)
    slen = np.full(n, 64, np.uint32)
    dest = tg.random_dest(n_rep, n, R, 7)
    orp = O.Replay(n_rep, R, caps)
    rp = P.Replay(ctx, n_rep, R, caps)
    ctr = torch.zeros((n_rep, len(caps), R, 5), dtype=torch.int64, device=DEV)
    dk, dp, ds, dd = d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest)
    cut = n // 2
    for a, b in ((0, cut), (cut, n)):
        orp.step(keys[a:b], plen[a:b], slen[a:b], dest[:, a:b])
        P.shadow_replay(ctx, rp, dk[a:b].contiguous(), dp[a:b].contiguous(), ds[a:b].contiguous(),
                        dd[:, a:b].contiguous(), ctr)
        ctx.sync()
        assert (h_u64(ctr) == orp.ctr).all()
    for rep in range(n_rep):
        for r in range(R):
            st = rp.state(rep, r)
            for c_i, c in enumerate(caps):
                assert (st[:c] == orp.state(rep, c_i, r)).all()


@pytest.mark.parametrize("R", [2, 191, 192, 193, 770, 800, 819, 820, 1024, 8192])
@pytest.mark.parametrize("n", [1, 33, 8191, 8192, 8193, 24577])
def test_replay_partition_edges(P, ctx, R, n):
    # every stream in arrival order (capacity 1 counts exactly the immediate repeats): both
    # ways of ranking equal destinations, tiles cut short, rows at odd addresses, and
    # destinations that are random, round robin, equal, or shared by pairs and runs of lanes
    # (from 768 to 819 destinations the dynamic shared memory alone is just below 48 KB)
    rng = np.random.default_rng(R * 31 + n)
    rows = [rng.integers(0, R, n), np.arange(n) % R, np.full(n, R - 1), (np.arange(n) // 2 * 7) % R,
            np.where(rng.random(n) < 0.5, R // 2, rng.integers(0, R, n)), (np.arange(n) // 16) % R]
    dest = np.stack(rows).astype(np.uint16)
    keys = rng.integers(1, 6, n).astype(np.uint64)
    plen = rng.integers(1, 5000, n).astype(np.uint32)
    slen = np.full(n, 64, np.uint32)
    caps = [1, 3]
    orp = O.Replay(len(rows), R, caps)
    rp = P.Replay(ctx, len(rows), R, caps)
    ctr = torch.zeros((len(rows), len(caps), R, 5), dtype=torch.int64, device=DEV)
    orp.step(keys, plen, slen, dest)
    P.shadow_replay(ctx, rp, d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest), ctr)
    ctx.sync()
    assert (h_u64(ctr) == orp.ctr).all()


@pytest.mark.parametrize("R,n,hot", [(1, 10007, 0.0), (3, 9001, 0.0), (600, 800000, 0.0), (8192, 60000, 0.5),
                                     (8191, 60000, 0.5), (2731, 50000, 0.3)])
def test_replay_items_of_many_chunks(P, ctx, R, n, hot):
    # streams of more than a few chunks (of 256 requests): one, three, 600 of them (more than one
    # CTA lists), a hot one among thousands; around 8,192 streams in one CTA or in four launches
    rng = np.random.default_rng(R)
    dest = rng.integers(0, R, (3 if R == 2731 else 1, n)).astype(np.uint16)
    dest[:, rng.random(n) < hot] = R // 2
    keys = rng.integers(1, 9, n).astype(np.uint64)
    plen = rng.integers(1, 5000, n).astype(np.uint32)
    slen = np.full(n, 64, np.uint32)
    orp = O.Replay(dest.shape[0], R, [3])
    rp = P.Replay(ctx, dest.shape[0], R, [3])
    ctr = torch.zeros((dest.shape[0], 1, R, 5), dtype=torch.int64, device=DEV)
    for _ in range(2):
        orp.step(keys, plen, slen, dest)
        P.shadow_replay(ctx, rp, d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest), ctr)
    ctx.sync()
    assert (h_u64(ctr) == orp.ctr).all()


@pytest.mark.parametrize("tokens", [False, True])
@pytest.mark.parametrize("R,n,hot,caps", [(900, 1800, 0.0, [64]), (900, 1801, 0.1, [2, 40, 1000]), (8192, 500, 0.0, [8]),
                                          (300, 600, 0.3, [33]), (50, 100, 0.0, [32, 31]), (400, 3200, 0.0, [100]),
                                          (400, 3201, 0.0, [5])])
def test_replay_short_streams(P, ctx, tokens, R, n, hot, caps):
    # streams of a few requests or none: lists that fit 32 entries with the call's requests, that
    # outgrow them over the calls, empty streams with longer lists; averages at and past the
    # lines of the kernel for them (two requests, eight for token capacities); a hot stream of
    # several chunks beside
    rng = np.random.default_rng(R + n)
    if tokens:
        caps = [c * 500 for c in caps]
    orp, rp = O.Replay(2, R, caps, tokens=tokens), P.Replay(ctx, 2, R, caps, tokens=tokens)
    ctr = torch.zeros((2, len(caps), R, 5), dtype=torch.int64, device=DEV)
    for call in range(12):
        dest = rng.integers(0, R, (2, n)).astype(np.uint16)
        dest[:, rng.random(n) < hot] = 1
        keys = rng.integers(1, 40 if call % 3 else 4000, n).astype(np.uint64)
        plen = (keys * np.uint64(7919) % np.uint64(900)).astype(np.uint32)  # 0 for some, above the least capacity for others
        slen = np.full(n, 64, np.uint32)
        orp.step(keys, plen, slen, dest)
        P.shadow_replay(ctx, rp, d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest), ctr)
    ctx.sync()
    assert (h_u64(ctr) == orp.ctr).all()
    top = int(np.argmax(caps))
    for r in list(range(0, R, max(1, R // 20))) + [1]:
        assert (rp.state(1, r) == orp.state(1, top, r)).all()


@pytest.mark.parametrize("tokens", [False, True])
@pytest.mark.parametrize("R,hot", [(40, [7]), (700, [3, 200, 699]), (700, list(range(0, 700, 9))), (33, [])])
def test_replay_items_of_long_streams(P, ctx, tokens, R, hot):
    # streams longer than twice the mean take the first work items: none, a few, and one in
    # nine of them, in whole chunks and in one, with empty streams between
    rng = np.random.default_rng(R + len(hot))
    n_rep, n = 3, 24000
    caps = [400000] if tokens else [16, 1000]
    keys = _rates_keys(rng, 4000, n)[:n]
    n = keys.size
    plen = (16 + keys % np.uint64(3000)).astype(np.uint32)
    slen = np.full(n, 64, np.uint32)
    dest = rng.integers(0, R, size=(n_rep, n)).astype(np.uint16)
    if hot:
        to = rng.random((n_rep, n)) < 0.8
        dest[to] = rng.choice(np.array(hot, np.uint16), size=int(to.sum()))
    dest[dest == 5] = 4
    orp = O.Replay(n_rep, R, caps, tokens=tokens)
    rp = P.Replay(ctx, n_rep, R, caps, tokens=tokens)
    ctr = torch.zeros((n_rep, len(caps), R, 5), dtype=torch.int64, device=DEV)
    dk, dp, ds, dd = d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest)
    cut = n // 3
    for a, b in ((0, cut), (cut, n)):
        orp.step(keys[a:b], plen[a:b], slen[a:b], dest[:, a:b])
        P.shadow_replay(ctx, rp, dk[a:b].contiguous(), dp[a:b].contiguous(), ds[a:b].contiguous(),
                        dd[:, a:b].contiguous(), ctr)
        ctx.sync()
        assert (h_u64(ctr) == orp.ctr).all()


def test_replay_state_import_resumes(P, ctx):
    # replay two calls in one simulator set; export every state after the first, import
    # it into a fresh set, and the second call's counters match
    rng = np.random.default_rng(5)
    caps, n_rep, R = [8, 64, 256], 2, 6
    keys = _rates_keys(rng, 2000, 30000)
    n = keys.size
    plen = rng.integers(16, 4000, size=n).astype(np.uint32)
    slen = np.full(n, 64, np.uint32)
    dest = tg.random_dest(n_rep, n, R, 9)
    cut = n // 2
    dk, dp, ds, dd = d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest)
    a = P.Replay(ctx, n_rep, R, caps)
    ctr_a = torch.zeros((n_rep, len(caps), R, 5), dtype=torch.int64, device=DEV)
    P.shadow_replay(ctx, a, dk[:cut].contiguous(), dp[:cut].contiguous(), ds[:cut].contiguous(),
                    dd[:, :cut].contiguous(), ctr_a)
    ctx.sync()
    b = P.Replay(ctx, n_rep, R, caps)
    for rep in range(n_rep):
        for r in range(R):
            b.set_state(rep, r, a.state(rep, r))
    ctr_a.zero_()
    ctr_b = torch.zeros_like(ctr_a)
    for rp, ctr in ((a, ctr_a), (b, ctr_b)):
        P.shadow_replay(ctx, rp, dk[cut:].contiguous(), dp[cut:].contiguous(), ds[cut:].contiguous(),
                        dd[:, cut:].contiguous(), ctr)
    ctx.sync()
    assert (h_u64(ctr_a) == h_u64(ctr_b)).all()
    with pytest.raises(P.CacheRouteError):
        b.set_state(0, 0, np.array([1, 2, 1], np.uint64))     # repeated key
    with pytest.raises(P.CacheRouteError):
        b.set_state(0, R, np.array([1], np.uint64))            # no such destination
    a.close()
    b.close()


def test_debug_build_runs_the_smoke_check_clean():
    # the bounds-checking build gives the oracle's results and raises no flag on a small
    # pass of the whole path (run in a child process that loads the debug library)
    import os
    import subprocess
    import sys
    from paper_2608_19677_gb300 import buildlib
    buildlib.build(debug=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, CR_DEBUG_LIB="1")
    code = ("import paper_2608_19677_gb300 as P, __graft_entry__ as g; "
            "assert P.LIB_PATH.endswith('libcacheroute_debug.so'); g.smoke()")
    r = subprocess.run([sys.executable, "-c", code], cwd=root, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    assert "smoke ok" in r.stdout


def test_replay_partition_then_simulate_equals_shadow_replay(P, ctx):
    # the two-call form (partition on one stream, simulation on another, ordered by an
    # event) gives the same counters and states as cr_shadow_replay, over two calls; an
    # input partitioned for another replay shape is refused
    rng = np.random.default_rng(17)
    caps, n_rep, R = [16, 64], 3, 9
    keys = _rates_keys(rng, 800, 24000)
    n = keys.size
    plen = rng.integers(16, 3000, size=n).astype(np.uint32)
    slen = np.full(n, 64, np.uint32)
    dest = tg.random_dest(n_rep, n, R, 4)
    dk, dp, ds, dd = d_u64(keys), d_u32(plen), d_u32(slen), d_u16(dest)
    a = P.Replay(ctx, n_rep, R, caps)
    b = P.Replay(ctx, n_rep, R, caps)
    ctr_a = torch.zeros((n_rep, len(caps), R, 5), dtype=torch.int64, device=DEV)
    ctr_b = torch.zeros_like(ctr_a)
    side = torch.cuda.Stream(DEV)
    pctx = P.Context(0, side)
    inp = P.ReplayInput(pctx)
    cut = n // 2
    for lo, hi in ((0, cut), (cut, n)):
        args = (dk[lo:hi].contiguous(), dp[lo:hi].contiguous(), ds[lo:hi].contiguous(), dd[:, lo:hi].contiguous())
        P.shadow_replay(ctx, a, *args, ctr_a)
        side.wait_stream(torch.cuda.current_stream(DEV))
        P.replay_partition(pctx, b, *args, inp)
        ev = torch.cuda.Event()
        ev.record(side)
        torch.cuda.current_stream(DEV).wait_event(ev)
        P.replay_simulate(ctx, b, inp, ctr_b)
        ctx.sync()
        pctx.sync()
    assert (h_u64(ctr_a) == h_u64(ctr_b)).all()
    for rep in range(n_rep):
        for r in range(R):
            assert (a.state(rep, r) == b.state(rep, r)).all()
    other = P.Replay(ctx, n_rep, R + 1, caps)
    with pytest.raises(P.CacheRouteError):
        P.replay_simulate(ctx, other, inp, torch.zeros((n_rep, len(caps), R + 1, 5), dtype=torch.int64, device=DEV))
    inp.close()
    pctx.close()


def test_replay_input_without_memory_is_refused(P, ctx):
    # a partition whose buffers cannot be had leaves its input without a partition: the simulation
    # refuses it (its pointers would be of the call before, or none), and works once memory is there
    n, R = 40_000_000, 16
    dk = torch.arange(n, dtype=torch.int64, device=DEV) % 1000
    one = torch.ones(n, dtype=torch.int32, device=DEV)
    dest = (torch.arange(n, dtype=torch.int32, device=DEV) % R).to(torch.int16)[None].contiguous()
    small = [x[..., :5000].contiguous() for x in (dk, one, one, dest)]
    rp = P.Replay(ctx, 1, R, [64])
    inp = P.ReplayInput(ctx)
    ctr = torch.zeros((1, 1, R, 5), dtype=torch.int64, device=DEV)
    P.replay_partition(ctx, rp, *small, inp)
    ctx.sync()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info(0)[0]
    hog = torch.empty(free - (500 << 20), dtype=torch.uint8, device=DEV)  # the records alone take 640 MB
    try:
        with pytest.raises(P.CacheRouteError, match="allocate"):
            P.replay_partition(ctx, rp, dk, one, one, dest, inp)
        with pytest.raises(P.CacheRouteError, match="another replay shape"):
            P.replay_simulate(ctx, rp, inp, ctr)
    finally:
        del hog
        torch.cuda.empty_cache()
    for args in (small, (dk, one, one, dest)):
        P.replay_partition(ctx, rp, *args, inp)
        P.replay_simulate(ctx, rp, inp, ctr)
    ctx.sync()
    assert int(ctr[..., 0].sum()) == n + 5000
    inp.close()


def test_plan_build_without_memory_leaves_no_plan(P, ctx):
    # a build whose buffers cannot be had leaves none of its plans built (their tables would not
    # be filled), and the same objects build again once memory is there
    rng = np.random.default_rng(3)
    keys = _rates_keys(rng, 2000, 100000)
    n, R = keys.size, 1024
    dk = d_u64(keys)
    small = P.plan_params(R, 4, n, R)
    plans = [P.Plan(ctx), P.Plan(ctx)]
    P.build_plans(ctx, dk, [small, small], plans)
    load = torch.zeros((1, R), dtype=torch.int64, device=DEV)
    ctx.sync()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info(0)[0] - (500 << 20), dtype=torch.uint8, device=DEV)
    try:
        with pytest.raises(P.CacheRouteError, match="allocate"):  # 102 M slots: 1 GB of jobs
            P.build_plans(ctx, dk, [small, P.plan_params(R, 100000, n, R)], plans)
        for p in plans:
            with pytest.raises(P.CacheRouteError, match="built"):
                P.route_batch(ctx, [p], ["CR"], [0], R, dk, 0, 64, load)
            with pytest.raises(P.CacheRouteError, match="never built"):
                p.info()
    finally:
        del hog
        torch.cuda.empty_cache()
    ctx.sync()
    P.build_plans(ctx, dk, [small, small], plans)
    ref = O.build_plan(keys, R, 4, n, R)
    for p in plans:
        _cmp_plan(p.export(), ref)
