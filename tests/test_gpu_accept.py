"""GPU acceptance kernel (sd2_accept_logits) against the oracle: emitted tokens bit-exact.

Both sides see the same logits and the same Philox stream; every decision (accept/reject, the
replacement drawn from the residual, the bonus token, greedy matches) must be identical.
"""
import numpy as np
import pytest
import torch

from oracle import sampling
from paper_2511_09844_gb300 import sd2
from paper_2511_09844_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _oracle(target, draft, xhat, temps, seed, step):
    t = target.float().cpu().numpy()
    d = draft.float().cpu().numpy()
    x = xhat.cpu().numpy()
    out = []
    for b in range(t.shape[0]):
        out.append(sampling.accept_block(t[b], d[b], list(x[b]), float(temps[b]), seed, b, step))
    return out


def _compare(target, draft, xhat, temps, seed, step):
    tt = torch.tensor(temps, dtype=torch.float32, device="cuda")
    tok, n = sd2.accept_logits(target.cuda(), draft.cuda(), xhat.cuda(), tt, seed, step)
    torch.cuda.synchronize()
    tok, n = tok.cpu(), n.cpu()
    ref = _oracle(target, draft, xhat, temps, seed, step)
    js = []
    for b, (emitted, j) in enumerate(ref):
        assert int(n[b]) == j + 1, (b, int(n[b]), j)
        assert tok[b, :j + 1].tolist() == emitted, (b, tok[b].tolist(), emitted)
        js.append(j)
    return js


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V,B,k", [(4096, 8, 4), (32000, 4, 8), (1000, 16, 1)])
def test_sweep_logits_bit_exact(dtype, V, B, k):
    target, draft, xhat = W.make_sweep_logits(B, k, V, seed=V + B + k)
    temps = [[0.0, 0.7, 1.0][b % 3] for b in range(B)]
    _compare(target.to(dtype), draft.to(dtype), xhat, temps, seed=99, step=3)


def test_high_acceptance_reaches_bonus_and_residual_paths():
    """Draft rows close to the target rows: many accepts, full blocks (bonus), and rejections."""
    B, k, V = 32, 6, 2048
    g = torch.Generator().manual_seed(5)
    target = torch.randn(B, k + 1, V, generator=g) * 2
    noise = torch.randn(B, k, V, generator=g) * torch.linspace(0.0, 1.5, B)[:, None, None]
    draft = target[:, :k] + noise
    # drafts: the draft row's most likely token (what a sampler would usually pick)
    xhat = draft.argmax(-1).to(torch.int32)
    temps = [1.0 if b % 4 else 0.7 for b in range(B)]
    js = _compare(target, draft, xhat, temps, seed=2024, step=11)
    assert max(js) == k and min(js) < k and len(set(js)) >= 3


def test_identical_rows_always_accept():
    B, k, V = 4, 5, 512
    g = torch.Generator().manual_seed(6)
    target = torch.randn(B, k + 1, V, generator=g)
    draft = target[:, :k].clone()
    xhat = torch.randint(0, V, (B, k), generator=g, dtype=torch.int32)
    js = _compare(target, draft, xhat, [1.0] * B, seed=3, step=1)
    assert js == [k] * B          # u*q <= p with q == p and u < 1


def test_greedy_prefix_match():
    B, k, V = 6, 4, 300
    g = torch.Generator().manual_seed(7)
    target = torch.randn(B, k + 1, V, generator=g)
    am = target.argmax(-1)
    xhat = am[:, :k].clone().to(torch.int32)
    for b in range(B):                 # sequence b mismatches at draft b (none for b >= k)
        if b < k:
            xhat[b, b] = (xhat[b, b] + 1) % V
    draft = torch.randn(B, k, V, generator=g)
    js = _compare(target, draft, xhat, [0.0] * B, seed=1, step=1)
    assert js == [min(b, k) for b in range(B)]


def test_step_and_seed_change_the_stream():
    B, k, V = 16, 4, 4096
    target, draft, xhat = W.make_sweep_logits(B, k, V, seed=8, std=0.5, boost=1.0)   # flat rows
    tt = torch.ones(B, device="cuda")

    def emitted(step):
        tok, n = sd2.accept_logits(target.cuda(), draft.cuda(), xhat.cuda(), tt, 1, step)
        tok, n = tok.cpu(), n.cpu()
        return [tok[b, :n[b]].tolist() for b in range(B)]        # entries past n are not written

    a, b, c = emitted(1), emitted(2), emitted(1)
    assert a == c and a != b


def test_nonfinite_logits_are_reported_not_trapped():
    """A NaN logit is latched in the error word; the context stays usable."""
    B, k, V = 2, 2, 256
    target = torch.randn(B, k + 1, V)
    target[1, 0, 7] = float("nan")
    draft = torch.randn(B, k, V)
    xhat = torch.zeros(B, k, dtype=torch.int32)
    L = sd2.load_library()
    ws = torch.zeros(L.sd2_accept_workspace_bytes(B, k), dtype=torch.uint8, device="cuda")
    sd2.accept_logits(target.cuda(), draft.cuda(), xhat.cuda(), torch.ones(B, device="cuda"), 1, 1, workspace=ws)
    torch.cuda.synchronize()
    # the error word sits right after the scratch tables
    R = B * (2 * k + 1)
    off = 8 * 2 * R + 8 * 2 * B + 4 * B + 8 * B
    word = int(ws[off:off + 4].cpu().view(torch.int32)[0])
    assert word & 1
    torch.cuda.synchronize()                      # no sticky error


# More than 152 rows (B (2k + 1); 96 of a vocabulary up to 65536) take the path that decides from approximate
# normalisers, which all of these have: rows whose last group is partial, rows of 8-byte alignment (bf16, V % 8 == 4), vocabularies below one pass.
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V,B,k", [(4, 110, 1), (36, 120, 3), (1004, 70, 4), (8196, 64, 2), (33000, 40, 4)])
def test_many_rows_bit_exact(dtype, V, B, k):
    target, draft, xhat = W.make_sweep_logits(B, k, V, seed=V + B + k, share_prob=0.8)
    mix = torch.rand(B, 1, 1, generator=torch.Generator().manual_seed(V))
    draft = (mix * target[:, :k].float() + (1 - mix) * draft.float())       # some pairs close, some not
    xhat[::3] = draft.argmax(-1)[::3].to(torch.int32)
    temps = [[0.0, 0.7, 1.0, 1.3][b % 4] for b in range(B)]
    js = _compare(target.to(dtype), draft.to(dtype), xhat, temps, seed=17, step=5)
    assert min(js) == 0 and max(js) == k


def test_close_calls_are_decided_exactly():
    """u q and p within a few ulps of each other: no approximate normaliser can tell, so each such
    draft is settled by its exact rows, and must agree with the oracle bit for bit."""
    from oracle import philox
    B, k, V, seed, step = 60, 3, 2000, 31, 2
    g = torch.Generator().manual_seed(9)
    draft = torch.randn(B, k, V, generator=g, dtype=torch.float64) * 2
    xhat = draft.argmax(-1).to(torch.int32)
    target = torch.randn(B, k + 1, V, generator=g, dtype=torch.float64) * 2
    for b in range(B):
        for i in range(k):
            x, u = int(xhat[b, i]), float(philox.accept_uniform(seed, i + 1, b, step))
            q = float(torch.softmax(draft[b, i], 0)[x])
            want = min(u * q * (1 + 2e-7 * float(torch.randn(1, generator=g))), 0.999)
            rest = torch.cat([target[b, i, :x], target[b, i, x + 1:]]).logsumexp(0)
            target[b, i, x] = float(rest) + np.log(want / (1 - want))        # p(x) = want
    js = _compare(target.float(), draft.float(), xhat, [1.0] * B, seed, step)
    assert len(set(js)) == k + 1


@pytest.mark.parametrize("B", [3, 120])              # the few-rows and the many-rows kernels
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("value,place,flagged", [(float("nan"), "target", True), (float("inf"), "target", True),
                                                 (float("-inf"), "target", True), (float("-inf"), "draft", True),
                                                 (float("nan"), "greedy draft", False), (0.0, "target", False)])
def test_every_nonfinite_logit_is_reported(B, dtype, value, place, flagged):
    """In any row, also one past the first rejection; a greedy sequence's draft rows are not read."""
    k, V = 2, 516
    g = torch.Generator().manual_seed(10)
    target, draft = torch.randn(B, k + 1, V, generator=g), torch.randn(B, k, V, generator=g)
    temps = torch.ones(B)
    temps[1] = 0.0
    if place == "target":
        target[B - 1, k, V - 1] = value
    else:
        draft[1 if place == "greedy draft" else 0, k - 1, 5] = value
    L = sd2.load_library()
    ws = torch.full((L.sd2_accept_workspace_bytes(B, k),), 0xA5, dtype=torch.uint8, device="cuda")
    sd2.accept_logits(target.to(dtype).cuda(), draft.to(dtype).cuda(), torch.zeros(B, k, dtype=torch.int32).cuda(),
                      temps.cuda(), 1, 1, workspace=ws)
    torch.cuda.synchronize()
    off = 8 * 2 * B * (2 * k + 1) + 8 * 2 * B + 4 * B + 8 * B
    assert (int(ws[off:off + 4].cpu().view(torch.int32)[0]) & 1) == (1 if flagged else 0)


def test_zero_residual_falls_back_to_the_target_row():
    """Equal rows but for one token far below the others, e^-70 under the draft and 0 under the target:
    both normalisers are the same, so the rejected draft leaves no positive residual anywhere, and the
    replacement is drawn from the target row."""
    for B, k in ((2, 1), (160, 1)):
        g = torch.Generator().manual_seed(11)
        target = torch.randn(B, k + 1, 600, generator=g)
        target[:, :, 3] = -100.0
        draft = target[:, :k].clone()
        draft[:, :, 3] = -67.0
        js = _compare(target, draft, torch.full((B, k), 3, dtype=torch.int32), [1.0] * B, seed=5, step=1)
        assert js == [0] * B


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V,B,k", [(4, 1, 1), (8, 2, 2), (36, 1, 5), (132, 3, 4), (516, 5, 3), (1020, 9, 4)])
def test_vocabularies_shorter_than_a_cluster_s_slices(dtype, V, B, k):
    """Few rows of so short a vocabulary that CTAs of a row's cluster have no entries and are at once where they
    exchange their maxima; many blocks in a row, so that clusters start at all times."""
    target, draft, xhat = W.make_sweep_logits(B, k, V, seed=V + B + k, share_prob=0.8)
    temps = [[1.0, 0.0, 0.7][b % 3] for b in range(B)]
    tt = torch.tensor(temps, dtype=torch.float32, device="cuda")
    t, d, x = target.to(dtype).cuda(), draft.to(dtype).cuda(), xhat.cuda()
    got = [sd2.accept_logits(t, d, x, tt, 7, step) for step in range(40)]
    torch.cuda.synchronize()
    for step, (tok, n) in enumerate(got):
        for b, (emitted, j) in enumerate(_oracle(t, d, xhat, temps, 7, step)):
            assert int(n[b]) == j + 1 and tok[b, :j + 1].tolist() == emitted, (step, b)


def test_close_calls_on_rows_whose_maximum_keeps_rising():
    """The largest vocabulary, logits that rise along it, so that every thread raises its reference in every pass;
    u q and p within a few ulps of each other."""
    from oracle import philox
    B, k, V, seed, step = 52, 1, 152064, 33, 4
    g = torch.Generator().manual_seed(12)
    rise = torch.linspace(0, 9, V, dtype=torch.float64)
    draft = torch.randn(B, k, V, generator=g, dtype=torch.float64) * 0.05 + rise
    target = torch.randn(B, k + 1, V, generator=g, dtype=torch.float64) * 0.05 + rise
    xhat = torch.randint(0, V, (B, k), generator=g, dtype=torch.int32)
    for b in range(B):
        x, u = int(xhat[b, 0]), float(philox.accept_uniform(seed, 1, b, step))
        q = float(torch.softmax(draft[b, 0], 0)[x])
        want = u * q * (1 + 2e-7 * float(torch.randn(1, generator=g)))
        rest = torch.cat([target[b, 0, :x], target[b, 0, x + 1:]]).logsumexp(0)
        target[b, 0, x] = float(rest) + np.log(want / (1 - want))            # p(x) = want
    js = _compare(target.float(), draft.float(), xhat, [1.0] * B, seed, step)
    assert set(js) == {0, 1}
