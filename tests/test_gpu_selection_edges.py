"""Edges of three dispatches of the bank update, and of its commit.

Selection: banks of 8,192 slots and more run on a cluster of blocks per head; its lists must be
those of Step 3 computed from the call's own crossings and projected densities, also when every
key ties and the provenance decides.  Projection: a prefix that is the whole tested range takes
the crossing pass's final sums, around multiples of the 128-column snapshots.  Norms: the wide
form of the candidates' norms and the one used after an import give the same bits.  Commit: a warp copies eight rows of 128, 256 or 512 bytes.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

INT_MAX = 2 ** 31 - 1


@pytest.fixture(scope="module")
def dkv():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2608_27922_gb300 import dkv as d
    return d


def _full_bank(dkv, H, M, N, seed, **kw):
    """A full bank of random keys around a few centres, every state from step 0."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    bank = dkv.BankLayer(H, 128, [M] * H, N, torch.bfloat16, **kw)
    mu = torch.randn(H, 8, 128, generator=g, device="cuda")

    def keys(n):
        which = torch.randint(0, 8, (H, n, 1), generator=g, device="cuda").expand(-1, -1, 128)
        return (torch.gather(mu, 1, which) + 0.3 * torch.randn(H, n, 128, generator=g, device="cuda")).bfloat16()
    bank.k.copy_(keys(M))
    bank.v.normal_(generator=g)
    bank.rho.uniform_(200, 400, generator=g)
    bank.base.copy_(bank.rho / torch.empty_like(bank.rho).uniform_(0.9, 1.9, generator=g))
    bank.prov_step.zero_()
    bank.prov_src.copy_(torch.argsort(torch.rand(H, M, generator=g, device="cuda")).int())   # order != slot
    bank.import_state([M] * H)
    return bank, keys(N), torch.randn(H, N, 128, generator=g, device="cuda").bfloat16()


@pytest.mark.parametrize("H,M,N", [(2, 8192, 300), (1, 16385, 129), (3, 9001, 512)])
@pytest.mark.parametrize("eviction", [0, 1, 2])
def test_cluster_selection_matches_step_3(dkv, H, M, N, eviction):
    bank, K, V = _full_bank(dkv, H, M, N, M + N, eviction=eviction)
    src = bank.prov_src.cpu().numpy().copy()
    bank.admit(K, V, 1)
    bank.evict()
    bank.sync()
    mid = {k: v.cpu().numpy() for k, v in bank.intermediates().items()}
    bank.commit()
    bank.sync()
    slot_new = bank.intermediates()["slot_new"].cpu().numpy()    # written by the commit
    _, hs = bank.stats()
    step, now = bank.prov_step.cpu().numpy(), bank.prov_src.cpu().numpy()
    for h in range(H):
        r, e = hs[h].admitted, hs[h].evicted
        assert r > 0 and e == r          # a full bank
        mand = mid["cross"][h, :M] <= r
        assert hs[h].mandatory == mand.sum() <= e
        rt = mid["rho_tilde"][h, :M]
        # (class, density, provenance) of Step 3 in the policy: crossers, then the fill's order
        cls = np.where(mand, 0, 1) if eviction != dkv.DKV_EVICT_DENSEST else np.zeros(M, int)
        dens = -rt if eviction != dkv.DKV_EVICT_MANDATORY_SOURCE else np.zeros(M)
        dens = np.where(cls == 0, 0.0, dens) if eviction != dkv.DKV_EVICT_DENSEST else dens
        expect = np.sort(np.lexsort((src[h], dens, cls))[:e])
        gone = np.nonzero(step[h] == 1)[0]   # evicted slots hold the admitted states
        assert np.array_equal(gone, expect), h
        # in ascending slot order, the admitted candidates in score order
        assert np.array_equal(slot_new[h, :e], expect)
        assert np.array_equal(now[h, gone], mid["perm"][h, :r])
    bank.close()


@pytest.mark.parametrize("N", [1, 127, 128, 129, 257])
@pytest.mark.parametrize("mode", ["tensor", "fp32"])
def test_projection_of_the_whole_range(dkv, N, mode):
    """tau far above any growth: r* = N, nothing evicted, every state's density grows by its
    interactions with the whole block."""
    H, m, M = 2, 300, 1000
    g = torch.Generator(device="cuda").manual_seed(N)
    bank = dkv.BankLayer(H, 128, [M] * H, N, torch.bfloat16, tau=1e6,
                         score_mode=dkv.DKV_SCORE_TENSOR if mode == "tensor" else dkv.DKV_SCORE_FP32)
    bank.k.normal_(generator=g)
    bank.rho.uniform_(1, 2, generator=g)
    bank.base.copy_(bank.rho)
    bank.import_state([m] * H)
    rho0 = bank.rho.double()
    K = torch.randn(H, N, 128, generator=g, device="cuda").bfloat16()
    bank.update(K, K, 1)
    bank.sync()
    assert bank.occupancy_host() == [m + N] * H
    a, b = bank.k[:, :m].double(), K.double()
    d2 = (a * a).sum(-1)[:, :, None] + (b * b).sum(-1)[:, None] - 2 * a @ b.transpose(1, 2)
    ref = rho0[:, :m] + ((1 + d2 / 64) ** -2).sum(-1)
    # fp32 sums of up to 257 positive terms, each within 2^-20 in tensor mode
    assert ((bank.rho[:, :m].double() - ref).abs() / ref).max().item() < 1e-5
    bank.close()


@pytest.mark.parametrize("N", [1, 7, 63, 65, 300])
@pytest.mark.parametrize("desc", [0, 1])
def test_candidate_norms_equal_the_imported_ones(dkv, N, desc):
    H, M = 3, 512
    g = torch.Generator(device="cuda").manual_seed(N)
    bank = dkv.BankLayer(H, 128, [M] * H, N, torch.bfloat16, descriptor=desc)
    bank.reset()
    K = torch.randn(H, N, 128, generator=g, device="cuda").bfloat16()
    V = torch.randn(H, N, 128, generator=g, device="cuda").bfloat16()
    bank.update(K, V, 0)
    bank.sync()
    m = min(N, M)
    got = bank.knorm[:, :m].clone()
    bank.knorm.fill_(-1)
    bank.import_state([m] * H)
    bank.sync()
    assert torch.equal(got, bank.knorm[:, :m])
    bank.close()


@pytest.mark.parametrize("N,M", [(1, 3), (7, 20), (9, 41), (64, 72), (130, 515)])
@pytest.mark.parametrize("d,dtype,desc", [(64, torch.bfloat16, 0), (128, torch.bfloat16, 1), (64, torch.float32, 1),
                                          (128, torch.float32, 0)])
def test_every_state_is_its_candidate(dkv, N, M, d, dtype, desc):
    """Appending and evicting commits: each state holds the key and value that its provenance
    names, and the norm that an import computes from them."""
    H, T = 3, 12
    g = torch.Generator(device="cuda").manual_seed(N)
    K, V = (torch.randn(T, H, N, d, generator=g, device="cuda").to(dtype) for _ in range(2))
    bank = dkv.BankLayer(H, d, [M, M - 1, max(1, M // 2)], N, dtype, sync_heads=0, descriptor=desc,
                         score_mode=dkv.DKV_SCORE_FP32 if d == 64 or dtype == torch.float32 else dkv.DKV_SCORE_TENSOR)
    bank.reset()
    for t in range(T):
        bank.update(K[t], V[t], t)
    bank.sync()
    occ = bank.occupancy_host()
    norms = bank.knorm.clone()
    steps = set()
    for h in range(H):
        t, i = bank.prov_step[h, :occ[h]].long(), bank.prov_src[h, :occ[h]].long()
        assert occ[h] > 0 and len(set(zip(t.tolist(), i.tolist()))) == occ[h]
        assert torch.equal(bank.k[h, :occ[h]], K[t, h, i]) and torch.equal(bank.v[h, :occ[h]], V[t, h, i])
        steps |= set(t.tolist())
    assert len(steps) > 1
    bank.import_state(occ)
    bank.sync()
    for h in range(H):
        assert torch.equal(norms[h, :occ[h]], bank.knorm[h, :occ[h]])
    bank.close()
