"""The kernels' own edges: sizes at which a tile, a piece, a replica count or a dispatch rule changes."""
import numpy as np
import pytest
import torch

import oracle
import test_gpu_parity as parity
from gpu_harness import Round, check_round, close, make_gpu, make_oracle, to_cpu
from helpers import WALK_SHAPES
from paper_2609_22098_b200 import binding
from paper_2609_22098_b200.binding import TreeSpark

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V,B", [(1, 3), (7, 5), (31, 300), (4095, 2), (4097, 9), (33000, 1), (50257, 40)])
def test_row_statistics_by_pieces(dtype, V, B):
    """One-node trees with proposal probability 1: the edge statistic is p(x) itself, that is the row's maximum and
    log-sum-exp; greedy bonus tokens are the first of planted equal maxima.  Rows and pieces start anywhere."""
    ts = TreeSpark(V, 2, 8, 1, 2, B, dtype=dtype)
    g = torch.Generator().manual_seed(V)
    Z = (torch.randn(2 * B, V, generator=g) * 4).to(dtype)
    Z[::3] -= torch.linspace(3e3, 0.0, V).to(dtype)   # rising rows: the sums' reference moves many times
    for i in range(2 * B):
        Z[i, torch.randint(0, V, (3,), generator=g)] = 20.0   # equal maxima
    Z[0, 0] = Z[0, V - 1] = 20.0
    if B > 1:
        Z[2] = torch.where(torch.rand(V, generator=g) < 0.5, -0.0, 0.0).to(dtype)   # -0 equals 0
    tree = ts.alloc_tree(B)
    x = torch.randint(0, V, (B,), generator=g, dtype=torch.int32)
    for k, v in (("n_nodes", 1), ("parent", -1), ("depth", 1), ("sib_rank", 0), ("logqT", 0.0), ("node_hash", 0), ("node_lseT", 0.0)):
        tree[k].fill_(v)
    tree["tok"][:, 0] = x.cuda()
    U, A, W = (torch.zeros(s, dtype=dtype, device="cuda") for s in ((B, 2, V), (V, 8), (8, V)))
    off = torch.arange(0, 2 * B + 1, 2, dtype=torch.int64).cuda()
    anchor = torch.zeros(B, dtype=torch.int32, device="cuda")
    first = Z.float().numpy().argmax(1)
    out = ts.verify_tree(U, A, W, Z.cuda(), off, anchor, tree, 0.0, 5)
    for b in range(B):
        hit = int(first[2 * b]) == int(x[b])
        assert int(out["bonus_tok"][b]) == int(first[2 * b + (1 if hit else 0)])
    for T in (1.0, 0.05):
        out = ts.verify_tree(U, A, W, Z.cuda(), off, anchor, tree, T, 5)
        assert (out["status"] == 0).all()
        lp = torch.log_softmax(Z[::2].double() / T, 1)[torch.arange(B), x.long()].numpy()
        e = out["edge_stat"][:, 0].double().cpu().numpy()
        # fp32 exponents of size |z| / T carry half an ulp each, the sum of positive terms a few more
        rel = 2.0 ** -23 * (2 * 20.0 / T + 16)
        assert np.all(np.abs(e - np.exp(lp)) <= rel * np.exp(lp) + 1e-37)


def check_scores(dtype, V, r, K, P, T, mode=0):
    wl = parity.small("tiny", V=V, r=r, K=K, D=3, Nmax=100, dtype=dtype, B=3, calib_mode=0)
    rnd = Round(wl, seed=3 + V)
    ts, orc = make_gpu(wl, None, max_batch=3, test_mode=mode), make_oracle(wl, None)
    g = torch.Generator().manual_seed(P)
    req, dep, tok, hsh = (torch.randint(0, n, (P,), generator=g) for n in (3, 3, V, 2 ** 62))
    out = to_cpu(ts.score_parents(rnd.U, rnd.A, rnd.W, req.int().cuda(), dep.int().cuda(), tok.int().cuda(), hsh.cuda(), T, seed=99))
    c = rnd.cpu()
    Af, Wf, Uf = c["A"].float().numpy(), c["W"].float().numpy(), c["U"].float().numpy()
    n, near = min(K, V), 0
    for i in range(P):
        o = orc.score_parent(Uf[req[i], dep[i]], Af[tok[i]], Wf, T, 99, int(req[i]), int(hsh[i]))
        assert close(out["lse0"][i], o["lse0"]) and close(out["lseT"][i], o["lseT"]), i
        for margin, name in zip(o["margins"], ("top", "draw")):
            if margin < oracle.TOPK_MARGIN:
                near += 1
                continue
            assert out[name + "_tok"][i, :n].tolist() == o[name + "_tok"][:n].tolist(), (i, name)
            assert all(close(out[name + "_logit"][i, j], o[name + "_logit"][j]) for j in range(n)), (i, name)
    assert near <= 2 + 0.02 * P


# parents at the replica counts' borders (32, 64, 128 rows of a tile) and beyond one group; ranks that are no multiple of 16
# or 64; vocabularies with 32-byte rows, with 16-byte rows only, and ragged ones (padded copies)
@pytest.mark.parametrize("P", [1, 32, 33, 64, 65, 128, 129, 260])
@pytest.mark.parametrize("V,r,K,mode", [(2048, 8, 8, 0), (2056, 24, 16, 0), (2049, 72, 4, 0), (2044, 64, 8, binding.TEST_NO_TMA), (65, 16, 8, 0)])
def test_scoring_tile_edges(V, r, K, mode, P):
    check_scores("bf16", V, r, K, P, 0.7, mode)


# fp32 lists up to what the few-parents kernel's records hold (95 at this size), and one more
@pytest.mark.parametrize("V,P", [(64000, 1), (64000, 9), (64000, 95), (64000, 96), (264, 8), (260, 8)])
def test_few_parents_edges(V, P):
    check_scores("f32", V, 4, 8, P, 1.0)


# bf16 lists up to what goes to the few-parents kernel (by parents, by pairs of parent and tile, by rank), and one more; the
# same lengths on the tensor cores
@pytest.mark.parametrize("V,r,P,mode", [(2048, 8, 64, 0), (2048, 8, 65, 0), (64000, 24, 11, 0), (64000, 24, 12, 0), (64000, 24, 13, 0), (1000, 128, 5, 0),
                                        (1000, 136, 5, 0), (1001, 64, 5, 0), (2048, 8, 1, binding.TEST_NO_FEW), (2048, 8, 32, binding.TEST_NO_FEW)])
def test_short_bf16_lists(V, r, P, mode):
    for T in (0.0, 0.7):
        check_scores("bf16", V, r, 8, P, T, mode)


@pytest.mark.parametrize("over,theta,T,mode", [
    (dict(V=3000, B=3, Nmax=96, K=8, D=6, r=16), 0.005, 0.7, 0),            # the last size of the single-owner form
    (dict(V=3001, B=3, Nmax=97, K=16, D=6, r=16), 0.005, 0.7, 0),           # shared merges and seed bounds, ragged rows
    (dict(V=4104, B=5, Nmax=256, K=16, D=16, r=40), 0.002, 1.0, 0),
    (dict(V=4104, B=2, Nmax=200, K=16, D=16, r=256), 0.002, 1.0, binding.TEST_NO_TMA),
    (dict(V=2500, B=70, Nmax=12, K=4, D=4, r=8), 0.02, 1.0, 0),             # the walk: more than 64 requests in a step
    (dict(V=5003, B=1, Nmax=24, K=8, D=5, r=64), 0.02, 0.7, 0),             # one request, ragged
    (dict(V=19000, B=65, Nmax=12, K=4, D=4, r=8), 0.03, 1.0, 0),            # base logits by boxes of all requests: a partial last slab,
    (dict(V=2501, B=128, Nmax=12, K=4, D=4, r=16), 0.03, 1.0, 0),           # padded rows and several groups of parents,
    (dict(V=2504, B=128, Nmax=12, K=4, D=4, r=256), 1.0, 0.7, 0),           # the chain,
    (dict(V=2504, B=129, Nmax=12, K=4, D=4, r=16), 0.03, 1.0, 0),           # and one request more than a box holds
    (dict(V=60008, B=9, Nmax=24, K=8, D=5, r=256), 0.02, 1.0, 0),           # the walk streams its range of W
])
def test_round_edges(over, theta, T, mode):
    wl = parity.small("wide", dtype="bf16", **over)
    rnd = Round(wl, seed=over["V"])
    rnd.theta.fill_(theta)
    ts = make_gpu(wl, rnd.table, max_batch=rnd.B, test_mode=mode)
    st = check_round(ts, make_oracle(wl, rnd.table), rnd, T, round_seed=9)
    assert st["nodes"] > rnd.B and st["trees_exempt"] <= 0.05 * st["trees"] + 2


@pytest.mark.parametrize("big,small", [
    (dict(V=19000, r=64, B=128), dict(V=19000, r=64, B=4)),                     # the form with the base-logit ring
    (dict(V=19000, r=64, B=3), dict(V=19000, r=32, B=3)),                       # one-launch expansion
    (dict(V=50001, r=64, B=2, dtype="f32"), dict(V=9001, r=4, B=2, dtype="f32")),   # fp32 tiles
    (dict(V=3000, r=4, B=2, dtype="f32", Nmax=256, K=16), dict(V=3000, r=4, B=2, dtype="f32", Nmax=160, K=16)),   # fp32 level step
    (dict(V=3000, r=4, B=2, dtype="f32", Nmax=128, K=15), dict(V=3000, r=4, B=2, dtype="f32", Nmax=8, K=2)),      # its 48 KB beside static arrays
])
def test_a_context_still_runs_after_another_one_was_made(big, small):
    """A kernel's shared-memory limit belongs to the process: a context with a smaller plan must not lower it."""
    def make(over):
        wl = parity.small("serve32", **dict(dict(D=4, Nmax=24, K=4), **over))
        rnd = Round(wl, seed=12)
        return rnd, make_gpu(wl, rnd.table, max_batch=rnd.B)
    rnd, ts = make(big)
    want = to_cpu(ts.expand_tree(rnd.U, rnd.A, rnd.W, rnd.anchor, rnd.theta, 1.0, 5))
    other = make(small)
    got = to_cpu(ts.expand_tree(rnd.U, rnd.A, rnd.W, rnd.anchor, rnd.theta, 1.0, 5))
    assert int(want["n_nodes"].sum()) > rnd.B and torch.equal(got["n_nodes"], want["n_nodes"])
    for b in range(rnd.B):
        n = int(want["n_nodes"][b])
        assert torch.equal(got["tok"][b, :n], want["tok"][b, :n])
    other[1].expand_tree(other[0].U, other[0].A, other[0].W, other[0].anchor, other[0].theta, 1.0, 5)


def test_scoring_that_gives_up_says_so_in_its_outputs():
    """ts_score_parents has no status array: when a bounded wait runs out, log-normalisers are NaN and tokens -1."""
    wl = parity.small("serve32", V=20000, B=3)
    rnd = Round(wl, seed=14)
    ts = make_gpu(wl, rnd.table, max_batch=3)
    P = 150
    g = torch.Generator().manual_seed(1)
    req, dep, tok, hsh = (torch.randint(0, n, (P,), generator=g) for n in (3, wl.D, wl.V, 2 ** 62))
    args = (rnd.U, rnd.A, rnd.W, req.int().cuda(), dep.int().cuda(), tok.int().cuda(), hsh.cuda(), 1.0, 3)
    want = to_cpu(ts.score_parents(*args))
    for call in (ts.score_parents, ts.score_parents_static):
        out = ts.alloc_score_outputs(P)
        for t in out.values():
            t.fill_(1)
        ts.set_test_mode(binding.TEST_SHORT_WAITS | binding.TEST_LOST_ARRIVAL)
        bad = to_cpu(call(*args, out=out))
        ts.set_test_mode(0)
        assert torch.isnan(bad["lse0"]).all() and torch.isnan(bad["lseT"]).all()
        assert (bad["top_tok"] == -1).all() and (bad["draw_tok"] == -1).all()
    again = to_cpu(ts.score_parents(*args))
    for k in want:
        assert torch.equal(again[k], want[k]), k


def test_candidates_that_nobody_waits_for_any_more_are_reported():
    """With waits of 4096 polls the warp that takes the candidates loses patience in ranges of 100,000 tokens when the only
    ones (planted far above the rest) stand at the ranges' ends.  They would be missing from the lists: the call says so."""
    V, P = 1 << 24, 128
    ts = TreeSpark(V, 1, 8, 4, P, 1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    TV = ((V + sms - 1) // sms + 63) // 64 * 64
    g = torch.Generator(device="cuda").manual_seed(4)
    U, A, W = ((torch.randn(s, generator=g, device="cuda") * x).bfloat16() for s, x in (((1, 1, V), 2.0), ((V, 8), 0.3), ((8, V), 0.3)))
    for i in range(16):
        U[0, 0, (i * (sms // 16) + 1) * TV - 3 - i] = 64.0 + i
    tok = torch.randint(0, V, (P,), generator=g, device="cuda", dtype=torch.int32)
    hsh = torch.randint(0, 2 ** 62, (P,), generator=g, device="cuda", dtype=torch.int64)
    zero = torch.zeros(P, dtype=torch.int32, device="cuda")
    want = to_cpu(ts.score_parents(U, A, W, zero, zero, tok, hsh, 1.0, 3))
    assert (want["top_tok"] >= 0).all()
    ts.set_test_mode(binding.TEST_SHORT_WAITS)
    got = to_cpu(ts.score_parents(U, A, W, zero, zero, tok, hsh, 1.0, 3))
    lost = (got["top_tok"] != want["top_tok"]).any(1) | (got["draw_tok"] != want["draw_tok"]).any(1)
    assert torch.isnan(got["lse0"][lost]).all(), f"{int(lost.sum())} lists are incomplete without a word"


class HardRound(Round):
    """A round whose target avoids what was drafted, so that walks reject sibling after sibling."""

    def target_logits(self, tree, sigma=None):
        Z, off = super().target_logits(tree, sigma)
        for b in range(self.B):
            n = int(tree["n_nodes"][b])
            rows, cols = int(off[b]) + tree["parent"][b, :n].long() + 1, tree["tok"][b, :n].long()
            Z[rows, cols] -= 3.0
        return Z, off


@pytest.mark.parametrize("over,T", [
    (dict(V=4104, B=33, Nmax=24, K=8, D=3, r=64), 1.0),       # an odd number of requests, one tile for four sets of warps
    (dict(V=3001, B=3, Nmax=40, K=16, D=3, r=16), 0.7),       # sixteen rejections: more coefficients than one reduction evaluates; ragged rows
    (dict(V=3003, B=2, Nmax=8, K=2, D=3, r=8), 1.3),          # two children
    (dict(V=60008, B=2, Nmax=24, K=8, D=3, r=256), 1.0),      # W through the ring
    (dict(V=240008, B=2, Nmax=12, K=8, D=2, r=8), 1.0),       # a range of more tiles than tensor memory holds at a time
])
def test_walks_that_reject_every_sibling(over, T):
    """The residual masses after several rejections come from one reduction at guessed coefficients: the walk has to be the
    oracle's, sibling by sibling, and it has to count the sums that it needed."""
    check_hard_walks(over, T)


def check_hard_walks(over, T, reqs=None, mode=0):
    wl = parity.small("wide", dtype="bf16", **over)
    rnd = HardRound(wl, seed=over["V"])
    rnd.theta.fill_(0.01)
    ts = make_gpu(wl, rnd.table, max_batch=rnd.B, test_mode=mode)
    st = check_round(ts, make_oracle(wl, rnd.table), rnd, T, round_seed=4, reqs=reqs)
    assert st["walks_exempt"] <= 0.1 * st["walks"] + 1
    tree = ts.expand_tree(rnd.U, rnd.A, rnd.W, rnd.anchor, rnd.theta, T, 4)
    Z, off = rnd.target_logits(tree)
    v = ts.verify_tree(rnd.U, rnd.A, rnd.W, Z, off, rnd.anchor, tree, T, 4)
    sums = (v["flags"] >> 8).cpu()
    for b in range(rnd.B):   # one sum a rejection, and the bonus draw's at a node without children
        n, kids = int(tree["n_nodes"][b]), {}
        for i in range(n):
            kids.setdefault(int(tree["parent"][b, i]), []).append(i)
        cur, want = -1, 0
        for i in range(int(v["acc_len"][b])):
            x = int(v["acc_node"][b, i])
            want += kids[cur].index(x)
            cur = x
        want += max(len(kids.get(cur, [])), 1)
        assert int(sums[b]) == want
    assert int(sums.max()) >= wl.K   # the case was reached


@pytest.mark.parametrize("V,r,B", list(WALK_SHAPES))
def test_every_form_of_the_walk_under_hard_targets(V, r, B):
    """A sample of the requests against the oracle, the ends of every pass among them; the sums of all."""
    size = WALK_SHAPES[V, r, B][1]
    ends = {b for k in range(0, B, size) for b in (k, min(k + size, B) - 1)} | {B // 2}   # (of every pass of the first step)
    check_hard_walks(dict(V=V, r=r, B=B, Nmax=12, K=8, D=3), 0.9, sorted(ends))


@pytest.mark.parametrize("V,r,B", [(64008, 32, 18), (200008, 64, 20)])   # (the second: passes of 16 and 4 beside a resident range)
def test_walk_without_a_tensor_map(V, r, B):
    check_hard_walks(dict(V=V, r=r, B=B, Nmax=12, K=8, D=3), 0.9, [0, B // 2, B - 1], binding.TEST_NO_TMA)


# several groups of 128 parents whose last is held once, twice or four times over
@pytest.mark.parametrize("P", [129, 160, 161, 192, 193])
def test_last_group_of_a_list(P):
    check_scores("bf16", 2048, 8, 8, P, 0.7)


def test_expansions_repeat_to_the_last_bit():
    """A level's list holds its parents in the order in which their owners are done, another one on every run: no sum may
    depend on the place.  Lists of 129 to 192 parents, whose second group is short, must be among the levels."""
    wl = parity.small("wide", V=20008, B=40, Nmax=32, K=8, D=5, r=32, dtype="bf16")
    rnd = Round(wl, seed=77)
    ts = make_gpu(wl, rnd.table, max_batch=rnd.B)
    levels, first = set(), None
    for scale in (1.0, 1.4, 2.0, 2.8, 4.0):
        rnd.theta.fill_(0.02 * scale)
        first = None
        for _ in range(25):
            t = to_cpu(ts.expand_tree(rnd.U, rnd.A, rnd.W, rnd.anchor, rnd.theta, 1.0, 5))
            live = torch.arange(wl.Nmax)[None] < t["n_nodes"][:, None]
            got = [t[k][live].contiguous().view(torch.int32) for k in ("logS", "q0", "logqT", "logkey")] + [t["tok"][live], t["node_lseT"][:, 1:][live].contiguous().view(torch.int32)]
            if first is None:
                first = got
                scored = live & ~torch.isnan(t["node_lseT"][:, 1:])
                levels |= {int((scored & (t["depth"] == d)).sum()) for d in range(1, wl.D)}
            assert all(torch.equal(a, b) for a, b in zip(first, got))
    assert any(128 < n <= 192 for n in levels), levels
