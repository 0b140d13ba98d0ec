"""Bank-reading attention (Sec. 3.2): the tensor-core schedules against the oracle.

There are three (csrc/attn_schedule.h): one CTA per 128 queries with the key range split
between its two softmax groups (whole units), equal shares of the key tiles of all units with
the cut units merged (shares; on banks that hold too little for that the same kernel takes
whole units), and one CTA per 256 queries whose two query tiles share every key tile (two
tiles).  Every case asserts the schedule it is there for, from the rule itself and, for the
shares, from the list of cut units that the kernel leaves in the workspace.  The cases use
ragged occupancies and window lengths, query counts that leave a partial second tile or none,
and heads with no keys.  Outputs are compared with the oracle's softmax attention over
[bank | window] in float64, within 2e-2 absolute.
"""
import numpy as np
import pytest
import torch

import attn_schedule as A
import oracle
import synth
from gpu_util import load_state, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dkv():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2608_27922_gb300 import dkv as d
    return d


def _bf16(rng, shape, scale):
    return synth.round_to_bf16((rng.standard_normal(shape) * scale).astype(np.float32))


def _bank_with(dkv, occ, M, d=128, seed=0):
    """A bank whose head h holds occ[h] random bf16 states (the oracle's copy alongside)."""
    rng = np.random.default_rng(seed)
    H = len(occ)
    ob = oracle.LayerBank.empty([M] * H, d)
    for h, m in enumerate(occ):
        hb = ob.heads[h]
        hb.K = _bf16(rng, (m, d), 1.5).astype(np.float64)
        hb.V = _bf16(rng, (m, d), 1.0).astype(np.float64)
        hb.rho = np.ones(m, np.float32)
        hb.base = np.ones(m, np.float32)
        hb.step = np.zeros(m, np.int64)
        hb.src = np.arange(m, dtype=np.int64)
    bank = dkv.BankLayer(H, d, [M] * H, 64, torch.bfloat16, score_mode=dkv.DKV_SCORE_TENSOR)
    load_state(bank, ob)
    return bank, ob


@pytest.mark.parametrize("Nq,W,want", [(300, 200, A.WHOLE), (256, 0, A.TWO), (129, 77, A.TWO), (520, 128, A.TWO)])
def test_two_tile_attention_matches_oracle(dkv, Nq, W, want):
    H, M, d = 320, 400, 128   # >= 2 CTAs per SM in every case
    assert A.launched([M] * H, Nq, W, A.n_sm()) == want
    occ = [(37 * h) % (M + 1) for h in range(H)]   # 0 .. 400, ragged
    occ[5] = 0
    bank, ob = _bank_with(dkv, occ, M, seed=Nq + W)
    rng = np.random.default_rng(Nq)
    Q = _bf16(rng, (H, Nq, d), 1.5)
    Kw = _bf16(rng, (H, W, d), 1.5) if W else None
    Vw = _bf16(rng, (H, W, d), 1.0) if W else None
    O = bank.attend(to_dev(Q, torch.bfloat16), None if Kw is None else to_dev(Kw, torch.bfloat16),
                    None if Vw is None else to_dev(Vw, torch.bfloat16)).float().cpu().numpy()
    bank.sync()
    err = 0.0
    for h in range(H):
        kw = np.zeros((0, d)) if Kw is None else Kw[h]
        vw = np.zeros((0, d)) if Vw is None else Vw[h]
        if occ[h] + kw.shape[0] == 0:
            assert np.all(O[h] == 0), h            # no keys at all: zero output
            continue
        ref = oracle.attend(ob.heads[h], Q[h], kw, vw)
        err = max(err, float(np.abs(O[h] - ref).max()))
    assert err < 2e-2, err
    bank.close()


def _random_bank(dkv, M, occ, seed):
    """A bank with random states made on the GPU; heads with fewer states than M hold garbage beyond."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    bank = dkv.BankLayer(len(occ), 128, [M] * len(occ), 64, torch.bfloat16)
    for h in range(0, len(occ), 64):
        bank.k[h:h + 64].normal_(0, 1.5, generator=g)
        bank.v[h:h + 64].normal_(generator=g)
    bank.base.fill_(1.0)
    bank.import_state(occ)
    return bank, g


def _rand(g, scale, *shape):
    return (torch.randn(shape, device="cuda", generator=g) * scale).bfloat16()


def _check(bank, occ, Q, Kw, Vw, O, heads, rows):
    """O against the oracle at these heads and query rows."""
    bank.sync()
    assert bool(torch.isfinite(O).all())
    for h in heads:
        n = lambda x: x[h].double().cpu().numpy() if x is not None else np.zeros((0, 128))
        hb = oracle.LayerBank.empty([max(1, occ[h])], 128).heads[0]
        hb.K, hb.V = (x[h, :occ[h]].double().cpu().numpy() for x in (bank.k, bank.v))
        got = O[h, rows].double().cpu().numpy()
        if occ[h] == 0 and Kw is None:
            assert np.all(got == 0), h
            continue
        assert np.abs(got - oracle.attend(hb, Q[h, rows].double().cpu().numpy(), n(Kw), n(Vw))).max() < 2e-2, h


@pytest.mark.parametrize("H,M,Nq,want", [(444, 3000, 256, A.TWO), (444, 3000, 250, A.TWO), (152, 4000, 300, A.WHOLE)])
def test_long_banks_reuse_every_slot(dkv, H, M, Nq, want):
    """24 to 32 bank tiles and 6 of the window: the two key and three value slots of the two-tile
    kernel (those of each group with whole units) and their parities go round many times."""
    W = 700
    assert A.launched([M] * H, Nq, W, A.n_sm()) == want
    occ = [M - (h % 3) * 61 for h in range(H)]
    bank, g = _random_bank(dkv, M, occ, 7)
    Q, Kw, Vw = _rand(g, 1.5, H, Nq, 128), _rand(g, 1.5, H, W, 128), _rand(g, 1.0, H, W, 128)
    with A.taken(bank) as t:
        O = bank.attend(Q, Kw, Vw)
    assert not t.shares
    _check(bank, occ, Q, Kw, Vw, O, range(0, H, 21), slice(None))
    bank.close()


@pytest.mark.parametrize("M,occ,Nq,W,cut", [
    (9360, [9000] * 12, 1560, 333, True),                # more units than CTAs, most CTAs hold two parts
    (9000, [0, 9000, 0, 128, 1, 6000], 40, 0, True),     # heads without keys between cut units
    (5000, [5000, 1500] * 4, 300, 64, True),             # units too short to cut between cut ones
    (9000, [9000], 129, 1, True),                        # one head, a query tile of one row
    (6000, [700] * 10, 100, 0, False),                   # budgets that pay for shares, banks that do not
    (6000, [2100, 0, 1] * 4, 300, 5, False),
    (9360, [2200] * 12, 1560, 0, False),                 # the same, two waves of whole units
])
def test_shares_of_units_match_oracle(dkv, M, occ, Nq, W, cut):
    H = len(occ)
    n_sm = A.n_sm()
    assert A.launched([M] * H, Nq, W, n_sm) == A.SHARES and A.cuts(occ, Nq, W, n_sm) == cut
    bank, g = _random_bank(dkv, M, occ, M + Nq)
    Q = _rand(g, 1.5, H, Nq, 128)
    Kw, Vw = (_rand(g, 1.5, H, W, 128), _rand(g, 1.0, H, W, 128)) if W else (None, None)
    with A.taken(bank) as t:
        O = bank.attend(Q, Kw, Vw)
    assert t.shares and (t.cut > 0) == cut
    rows = sorted({r for r in (0, 1, 31, 127, 128, 200, 255, 256, Nq // 2, Nq - 129, Nq - 1) if 0 <= r < Nq})
    _check(bank, occ, Q, Kw, Vw, O, range(H), rows)
    # a second call, on new queries, writes all of its list and parts again
    Q = _rand(g, 1.5, H, Nq, 128)
    _check(bank, occ, Q, Kw, Vw, bank.attend(Q, Kw, Vw), range(H), rows)
    bank.close()


@pytest.mark.parametrize("occ,M,Nq,W", [
    ([5000], 5000, 16, 700),                  # one unit, cut into many parts
    ([0], 300, 1, 0),                         # no key at all
    ([1], 300, 130, 0),                       # one key, two query tiles
    ([0, 900, 0, 128, 1, 77], 900, 200, 0),   # heads without keys
    ([3000, 129], 3000, 128, 1),              # a window of one key after a bank that ends inside a tile
    ([2000] * 13, 2000, 1560, 333),           # more query tiles than SMs
])
def test_shared_key_tiles_match_oracle(dkv, occ, M, Nq, W):
    """Few units: the first case is cut into parts, the others are whole units.  The same call on
    a handle whose workspace lacks the parts' scratch takes whole units in every case, with the
    same bits where the first did; both match the oracle."""
    H, d = len(occ), 128
    cut = A.launched([M] * H, Nq, W, A.n_sm()) == A.SHARES
    assert cut == (len(occ) == 1 and M == 5000)
    bank, ob = _bank_with(dkv, occ, M, seed=Nq + W)
    rng = np.random.default_rng(Nq)
    Q = _bf16(rng, (H, Nq, d), 1.5)
    Kw = _bf16(rng, (H, W, d), 1.5) if W else None
    Vw = _bf16(rng, (H, W, d), 1.0) if W else None
    Qd = to_dev(Q, torch.bfloat16)
    Kd, Vd = (to_dev(Kw, torch.bfloat16), to_dev(Vw, torch.bfloat16)) if W else (None, None)
    p = dkv.dkv_params_default(d)
    p.score_mode = dkv.DKV_SCORE_FP32
    small = dkv.dkv_bank_workspace_size(H, d, [M] * H, 64, dkv.DKV_DTYPE_BF16, p)
    assert small < bank.workspace.numel()
    spare = torch.empty(small, dtype=torch.uint8, device="cuda")
    bufs = dkv.dkv_buffers_t(bank.k.data_ptr(), bank.v.data_ptr(), bank.rho.data_ptr(), bank.base.data_ptr(),
                             bank.knorm.data_ptr(), bank.prov_step.data_ptr(), bank.prov_src.data_ptr(),
                             bank.occupancy.data_ptr(), spare.data_ptr(), small)
    with A.taken(bank) as t:
        O = bank.attend(Qd, Kd, Vd)
    assert t.shares == cut and (t.cut > 0) == cut
    whole = torch.full_like(O, 7.0)
    other = dkv.dkv_bank_create(H, d, [M] * H, 64, dkv.DKV_DTYPE_BF16, bank.params, bufs)
    dkv.dkv_bank_attend(other, Qd, Nq, Kd, Vd, W, whole)
    bank.sync()
    dkv.dkv_bank_sync(other)
    dkv.dkv_bank_destroy(other)
    assert cut or torch.equal(O, whole)
    O, whole = O.float().cpu().numpy(), whole.float().cpu().numpy()
    for h in range(H):
        if occ[h] + W == 0:
            assert np.all(O[h] == 0) and np.all(whole[h] == 0), h
            continue
        kw = np.zeros((0, d)) if Kw is None else Kw[h]
        vw = np.zeros((0, d)) if Vw is None else Vw[h]
        ref = oracle.attend(ob.heads[h], Q[h], kw, vw)
        assert np.abs(O[h] - ref).max() < 2e-2 and np.abs(whole[h] - ref).max() < 2e-2, h
    bank.close()


@pytest.mark.parametrize("occ", [2200, 9000])
def test_attention_bits_follow_the_bank_alone(dkv, occ):
    """156 units on the SMs, 9,360 states of budget: whole units pay with 2,200 states (18 key
    tiles), equal shares with 9,000.  The same bank and queries give the same bits on the handle
    that imported the bank, on one that was only handed its buffers, in a replayed graph, and on
    a handle that held another bank before."""
    H, M, d, Nq = 12, 9360, 128, 1560
    assert A.launched([M] * H, Nq, 0, A.n_sm()) == A.SHARES and A.cuts([occ] * H, Nq, 0, A.n_sm()) == (occ > 5000)
    g = torch.Generator(device="cuda")
    g.manual_seed(occ)
    bank = dkv.BankLayer(H, d, [M] * H, 64, torch.bfloat16)
    bank.k.normal_(generator=g)
    bank.v.normal_(generator=g)
    bank.base.fill_(1.0)
    bank.import_state([occ] * H)
    Q = torch.randn(H, Nq, d, device="cuda", generator=g).bfloat16()
    want = bank.attend(Q, None, None)
    bufs = dkv.dkv_buffers_t(bank.k.data_ptr(), bank.v.data_ptr(), bank.rho.data_ptr(), bank.base.data_ptr(),
                             bank.knorm.data_ptr(), bank.prov_step.data_ptr(), bank.prov_src.data_ptr(),
                             bank.occupancy.data_ptr(), bank.workspace.data_ptr(), bank.workspace.numel())
    bank.sync()
    other = dkv.dkv_bank_create(H, d, [M] * H, 64, dkv.DKV_DTYPE_BF16, bank.params, bufs)
    handed = torch.zeros_like(want)
    dkv.dkv_bank_attend(other, Q, Nq, None, None, 0, handed)
    dkv.dkv_bank_sync(other)
    dkv.dkv_bank_destroy(other)
    assert torch.equal(want, handed)

    captured = torch.zeros_like(want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        bank.attend(Q, None, None, captured)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(want, captured)

    again = dkv.BankLayer(H, d, [M] * H, 64, torch.bfloat16)
    again.k.copy_(bank.k)
    again.v.copy_(bank.v)
    again.base.fill_(1.0)
    again.import_state([M] * H)
    again.attend(Q, None, None)
    again.import_state([occ] * H)
    assert torch.equal(want, again.attend(Q, None, None))
    bank.sync()
    again.sync()
    bank.close()
    again.close()


@pytest.mark.parametrize("captured", [False, True])
def test_attention_on_two_streams_shares_the_scratch_in_turn(dkv, captured):
    """Attends of one handle on two streams, without events between them, whose units are cut
    (the handle's scratch holds the parts): each gives the bits that it gives alone."""
    H, M, d, Nq, W, reps = 2, 9000, 128, 200, 300, 6
    assert A.launched([M] * H, Nq, W, A.n_sm()) == A.SHARES and A.cuts([M, M - 700], Nq, W, A.n_sm())
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    bank = dkv.BankLayer(H, d, [M] * H, 64, torch.bfloat16)
    bank.k.normal_(generator=g)
    bank.v.normal_(generator=g)
    bank.base.fill_(1.0)
    bank.import_state([M, M - 700])
    Qs = [torch.randn(H, Nq, d, device="cuda", generator=g).bfloat16() for _ in range(2 * reps)]
    Kw, Vw = (torch.randn(H, W, d, device="cuda", generator=g).bfloat16() for _ in range(2))
    want = [bank.attend(q, Kw, Vw) for q in Qs]
    out = [torch.zeros_like(q) for q in Qs]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()

    def both(main):
        side.wait_stream(main)
        for i in range(reps):
            bank.attend(Qs[2 * i], Kw, Vw, out[2 * i], stream=main.cuda_stream)
            bank.attend(Qs[2 * i + 1], Kw, Vw, out[2 * i + 1], stream=side.cuda_stream)
        main.wait_stream(side)

    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            both(torch.cuda.current_stream())
        graph.replay()
    else:
        both(torch.cuda.current_stream())
    torch.cuda.synchronize()
    bank.sync()
    for i, (a, b) in enumerate(zip(want, out)):
        assert torch.equal(a, b), i
    bank.close()
