"""Updates and attention captured in CUDA graphs (no call of the hot path reads the device back,
so a whole step can be captured): every step's graph is captured before any of them runs, then
replayed in order on a bank that starts empty, fills and evicts.  Buffers and outputs must be
bit for bit those of a handle that makes the same calls directly, after every step; so must the
outputs of one attend captured on the empty bank and replayed after each step.
"""
import pytest
import torch

import attn_schedule as A

pytestmark = pytest.mark.gpu

BUFFERS = ("k", "v", "rho", "base", "knorm", "prov_step", "prov_src", "occupancy")


@pytest.fixture(scope="module")
def dkv():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2608_27922_gb300 import dkv as d
    return d


@pytest.mark.parametrize("mode,H,d,dtype,N,M,Nq,W,opts", [
    ("tensor", 2, 128, torch.bfloat16, 900, 4000, 200, 300, {"tau": 1e3}),   # attention in shares from step 4 on
    ("tensor", 4, 128, torch.bfloat16, 1700, 8500, 64, 0, {"sync_heads": 0, "tau": 1e3}),   # selection on clusters
    ("tensor", 160, 128, torch.bfloat16, 200, 500, 300, 128, {"layer_heads": 40, "tau": 1e3}),   # persistent passes
    ("tensor", 2, 128, torch.bfloat16, 200, 700, 64, 64, {"descriptor": 1, "tau": 1e3}),
    ("fp32", 2, 64, torch.float32, 256, 512, 256, 256, {"tau": 1e3}),                # chains over clusters
    ("fp32", 3, 128, torch.bfloat16, 150, 400, 40, 0, {"order": 1, "tau": 1e3}),
    ("tensor", 2, 128, torch.bfloat16, 900, 4000, 200, 300, {}),                 # prefixes that the growth gate cuts
])
def test_captured_steps_are_the_direct_ones(dkv, mode, H, d, dtype, N, M, Nq, W, opts):
    sm = dkv.DKV_SCORE_TENSOR if mode == "tensor" else dkv.DKV_SCORE_FP32
    steps = 6
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    mk = lambda *shape: torch.randn(shape, device="cuda", generator=g).to(dtype)
    blocks = [(mk(H, N, d), mk(H, N, d)) for _ in range(steps)]
    Q = [mk(H, Nq, d) for _ in range(steps)]
    Kw, Vw = (mk(H, W, d), mk(H, W, d)) if W else (None, None)
    banks = [dkv.BankLayer(H, d, [M] * H, N, dtype, score_mode=sm, **opts) for _ in range(2)]
    for b in banks:
        b.reset()
    torch.cuda.synchronize()
    eager, cap = banks
    out, fixed = [torch.zeros_like(q) for q in Q], torch.zeros_like(Q[0])

    def step(bank, t, O):
        bank.admit(*blocks[t], t)
        bank.compress()
        bank.attend(Q[t], Kw, Vw, O)

    graphs = [torch.cuda.CUDAGraph() for _ in range(steps)]
    once = torch.cuda.CUDAGraph()
    with torch.cuda.graph(once):
        cap.attend(Q[0], Kw, Vw, fixed)
    for t, graph in enumerate(graphs):
        with torch.cuda.graph(graph):
            step(cap, t, out[t])
    for t in range(steps):
        graphs[t].replay()
        once.replay()
        want = torch.zeros_like(Q[t])
        step(eager, t, want)
        torch.cuda.synchronize()
        assert torch.equal(want, out[t]), t
        assert torch.equal(eager.attend(Q[0], Kw, Vw), fixed), t
        for name in BUFFERS:
            assert torch.equal(getattr(eager, name), getattr(cap, name)), (t, name)
    for b in banks:
        b.sync()
    if "tau" in opts:   # whole blocks admitted: the banks fill up and evict
        assert eager.occupancy_host() == [M] * H
        assert sum(x.evicted for x in eager.stats()[1]) > 0
    if mode == "tensor" and H <= 4 and M > 1000:
        assert A.launched([M] * H, Nq, W, A.n_sm()) == A.SHARES
    for b in banks:
        b.close()
