"""The paged causal attention kernel (sd2_attention) against the oracle's attention (Sec. 3.2 decoder).

Each case builds a bf16 KV pool whose blocks are scattered through a random block table, row groups
at chosen positions of ragged sequences, and checks every output against oracle.model.causal_attention
evaluated in float64 on the same bf16 keys/values and bf16-rounded queries (the kernel stages queries
and probabilities in bf16). Covered: 1 to 16 context splits with empty splits, chunks of one and
several tiles, verifier-, drafter- and prompt-shaped groups, GQA ratios 1, 4 and 8, head dims 64 and
128, and the decode-step path whose cache rows below a pre-step length are read before the
programmatic wait (boundaries inside a tile, on a tile edge, on a split edge, at zero), with finite
stale rows between the last row and the planned bound; K/V rings of 2 to 4 tiles and split-merge
buffers laid over the ring. A row beyond the planned bound must raise the range bit of the error
word, not fault.
"""
import pytest
import torch

from conftest import kernels_of
from oracle import model as oracle_model
from paper_2511_09844_gb300 import sd2

pytestmark = pytest.mark.gpu

ERR_TIMEOUT, ERR_RANGE = 2, 4


def _case(seed, seq_lens, rows_per_group, H, Hkv, hd, n_layers=2, layer=1):
    """Random pool/table/queries; group g = the last rows_per_group[g] positions of sequence g."""
    g = torch.Generator().manual_seed(seed)
    n_seq = len(seq_lens)
    bt_stride = max((L + 15) // 16 for L in seq_lens) + 1
    n_blocks = n_seq * bt_stride + 3
    pool = (torch.randn(n_layers, n_blocks, 2, Hkv, 16, hd, generator=g)).to(torch.bfloat16)
    perm = torch.randperm(n_blocks, generator=g)[: n_seq * bt_stride]
    table = perm.view(n_seq, bt_stride).to(torch.int32)
    row_pos, grp_row0, grp_nrows, grp_seq = [], [], [], []
    for s, (L, nr) in enumerate(zip(seq_lens, rows_per_group)):
        grp_row0.append(len(row_pos))
        grp_nrows.append(nr)
        grp_seq.append(s)
        row_pos += list(range(L - nr, L))
    M = len(row_pos)
    q = torch.randn(M, H, hd, generator=g) * 2.0
    return dict(pool=pool, table=table, q=q, row_pos=torch.tensor(row_pos, dtype=torch.int32),
                grp_row0=torch.tensor(grp_row0, dtype=torch.int32), grp_nrows=torch.tensor(grp_nrows, dtype=torch.int32),
                grp_seq=torch.tensor(grp_seq, dtype=torch.int32), layer=layer, seq_lens=seq_lens, H=H, hd=hd)


def _reference(c):
    """Oracle attention per sequence: dense K/V gathered through the table, queries at their positions."""
    pool, table, layer = c["pool"], c["table"], c["layer"]
    H, hd = c["H"], c["hd"]
    q_bf = c["q"].to(torch.bfloat16).double()
    out = torch.zeros(c["q"].shape[0], H * hd, dtype=torch.float64)
    for g in range(len(c["grp_row0"])):
        s, r0, nr = int(c["grp_seq"][g]), int(c["grp_row0"][g]), int(c["grp_nrows"][g])
        pos = c["row_pos"][r0:r0 + nr].tolist()
        T = max(pos) + 1
        blocks = table[s, : (T + 15) // 16].long()
        kv = pool[layer, blocks].double()                          # [nb, 2, Hkv, 16, hd]
        k = kv[:, 0].permute(0, 2, 1, 3).reshape(-1, kv.shape[2], hd)[:T]
        v = kv[:, 1].permute(0, 2, 1, 3).reshape(-1, kv.shape[2], hd)[:T]
        qf = torch.zeros(T, H, hd, dtype=torch.float64)
        for i, p in enumerate(pos):
            qf[p] = q_bf[r0 + i]
        o = oracle_model.causal_attention(qf, k, v, row_block=512)
        for i, p in enumerate(pos):
            out[r0 + i] = o[p].reshape(-1)
    return out


def _run(c, n_splits, chunk, pre_len=None, pre_stable=0, pre_fresh=0, max_rows=None):
    dev = {k: v.cuda() for k, v in c.items() if isinstance(v, torch.Tensor)}
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = sd2.attention(dev["q"].float().contiguous(), dev["pool"], dev["table"], c["layer"], dev["row_pos"],
                        dev["grp_row0"], dev["grp_nrows"], dev["grp_seq"],
                        max_rows or int(c["grp_nrows"].max()), n_splits, chunk,
                        pre_len=None if pre_len is None else torch.tensor(pre_len, dtype=torch.int32, device="cuda"),
                        pre_stable=pre_stable, pre_fresh=pre_fresh, err=err)
    torch.cuda.synchronize()
    return out.float().cpu(), int(err.item())


def _check(out, ref):
    assert torch.isfinite(out).all()
    torch.testing.assert_close(out.double(), ref, atol=1.5e-2, rtol=1e-2)


@pytest.mark.parametrize("n_splits,chunk", [(1, 1152), (9, 128), (16, 128), (5, 256), (16, 64 * 18)])
def test_verify_shaped_groups_over_splits(n_splits, chunk):
    """Verify blocks (6 rows x 4 heads per KV head, hd 128) of ragged sequences; the large-chunk
    cases leave most splits empty."""
    c = _case(1, seq_lens=[1030, 517, 70], rows_per_group=[6, 6, 6], H=32, Hkv=8, hd=128)
    out, err = _run(c, n_splits, chunk)
    assert err == 0
    _check(out, _reference(c))


@pytest.mark.parametrize("hd,H,Hkv,rows", [(64, 32, 8, [1, 2, 1]), (64, 8, 8, [2, 1, 2]), (128, 64, 8, [6, 3, 1])])
def test_drafter_and_gqa_shapes(hd, H, Hkv, rows):
    """Drafter rows (1 or 2 per sequence), GQA ratios 1, 4 and 8."""
    c = _case(2, seq_lens=[700, 129, 64], rows_per_group=rows, H=H, Hkv=Hkv, hd=hd)
    out, err = _run(c, 11, 64)
    assert err == 0
    _check(out, _reference(c))


def test_prompt_shaped_group():
    """A prompt chunk: 16 rows x 4 heads = 64 query vectors (the per-CTA maximum)."""
    c = _case(3, seq_lens=[300, 16], rows_per_group=[16, 16], H=16, Hkv=4, hd=64)
    out, err = _run(c, 3, 128)
    assert err == 0
    _check(out, _reference(c))


@pytest.mark.parametrize("stable_off", [0, 3, 6])
@pytest.mark.parametrize("lens", [[517, 1030, 7], [512, 640, 6], [1024, 200, 13]])
def test_decode_step_reads_pre_step_rows_early(lens, stable_off):
    """pre_len places the boundary inside a tile, on a tile edge, on a split edge and at zero. The rows
    between the last row and pre_len + pre_stable + pre_fresh hold finite stale values, masked."""
    k1 = 6
    c = _case(4, seq_lens=lens, rows_per_group=[k1] * 3, H=32, Hkv=8, hd=128)
    ref = _reference(c)
    # verifier convention: rows at n-1 .. n-1+k, cache [0, n-1) written before the step
    pre_len = [L - k1 + 1 - stable_off for L in lens]
    pre_len = [max(0, p) for p in pre_len]
    out, err = _run(c, 9, 128, pre_len=pre_len, pre_stable=-1, pre_fresh=k1 + stable_off + 1)
    assert err == 0
    _check(out, ref)
    # the same with more splits than the context needs and one-tile chunks
    out, err = _run(c, 16, 64 * 2, pre_len=pre_len, pre_stable=-1, pre_fresh=k1 + stable_off + 1)
    assert err == 0
    _check(out, ref)


def test_row_beyond_the_planned_bound_is_reported():
    """pre_fresh one short: each sequence's last key row is zero-filled instead of read, and the
    kernel reports the range error instead of reading outside the planned rows."""
    k1 = 6
    c = _case(5, seq_lens=[600, 300], rows_per_group=[k1, k1], H=32, Hkv=8, hd=128)
    pre_len = [600 - k1 + 1, 300 - k1 + 1]
    out, err = _run(c, 9, 128, pre_len=pre_len, pre_stable=-1, pre_fresh=k1 - 1)
    assert err & ERR_RANGE
    assert torch.isfinite(out).all()


@pytest.mark.parametrize("hd,H,Hkv,n_seq,n_splits,chunk,kernel", [(64, 32, 8, 8, 4, 1024, "attn_few"), (128, 16, 4, 1, 16, 256, "attn_stream"),
                                                                  (128, 16, 4, 1, 9, 128, "attn")])
def test_rows_past_the_table_and_past_the_splits(hd, H, Hkv, n_seq, n_splits, chunk, kernel):
    """Every kernel alike: a row at a position that the block table does not cover is reported; positions beyond
    n_splits * chunk are not seen by a row that lies past them, and that is no error."""
    L = 700 if n_splits != 16 else 4000
    c = _case(14, [L] * n_seq, [1] * n_seq, H, Hkv, hd)
    pre = dict(pre_len=[L - 1] * n_seq, pre_stable=0, pre_fresh=1)
    assert _kernel(c, n_splits, chunk, **pre) == kernel
    out, err = _run(c, n_splits, chunk, **pre)
    assert err == 0
    _check(out, _reference(c))
    short = dict(c, table=c["table"][:, : L // 16 - 4].contiguous())
    out, err = _run(short, n_splits, chunk, **pre)
    assert err == ERR_RANGE and torch.isfinite(out).all()
    fewer = 64 if n_splits == 9 else chunk * 3 // 4 if n_splits == 16 else 128       # n_splits * fewer < L
    out, err = _run(c, n_splits, fewer, **pre)
    assert err == 0
    seen = dict(c, row_pos=torch.full_like(c["row_pos"], n_splits * fewer - 1))
    _check(out, _reference(seen))


def test_bad_arguments_are_rejected_on_the_host():
    c = _case(6, seq_lens=[100], rows_per_group=[2], H=32, Hkv=8, hd=128)
    with pytest.raises(sd2.SD2Error):
        _run(c, 17, 64)                 # more splits than a cluster takes
    with pytest.raises(sd2.SD2Error):
        _run(c, 2, 96)                  # chunk not a multiple of 64
    with pytest.raises(sd2.SD2Error):
        _run(c, 2, 64, max_rows=17)     # 17 rows x 4 heads per KV head > 64 query vectors


@pytest.mark.parametrize("hd,k1,n_splits,chunk", [(128, 9, 2, 768), (128, 9, 16, 128), (64, 2, 2, 768), (64, 1, 9, 256)])
def test_ring_depths_and_merge_over_the_ring(hd, k1, n_splits, chunk):
    """K/V rings of 2 to 4 tiles and, where two CTAs per SM fit only that way (48 query vectors at
    16 splits), the split-merge buffers laid over the ring; decode steps and plain launches."""
    lens = [1030, 517, 70]
    c = _case(7, seq_lens=lens, rows_per_group=[k1] * 3, H=32, Hkv=8, hd=hd)
    ref = _reference(c)
    pre_len = [max(0, L - k1 + 1) for L in lens]
    out, err = _run(c, n_splits, chunk, pre_len=pre_len, pre_stable=-1, pre_fresh=k1 + 1)
    assert err == 0
    _check(out, ref)
    out, err = _run(c, n_splits, chunk)
    assert err == 0
    _check(out, ref)


def test_many_sequences_four_ctas_per_sm():
    """16 drafter-shaped groups x 8 KV heads x 4 splits = 512 CTAs: the hd = 64 launch sized for four
    resident CTAs per SM (its shared-memory share), in a decode step and a plain launch."""
    lens = [70 + 61 * i for i in range(16)]
    c = _case(8, seq_lens=lens, rows_per_group=[1] * 16, H=32, Hkv=8, hd=64)
    ref = _reference(c)
    pre_len = [L - 1 for L in lens]
    out, err = _run(c, 4, 320, pre_len=pre_len, pre_stable=0, pre_fresh=1)
    assert err == 0
    _check(out, ref)
    out, err = _run(c, 4, 320)
    assert err == 0
    _check(out, ref)


def _run_flat(c, slots, max_ctx, pre_len, pre_stable, pre_fresh, workspace=None):
    dev = {k: v.cuda() for k, v in c.items() if isinstance(v, torch.Tensor)}
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = sd2.attention_flat(dev["q"].float().contiguous(), dev["pool"], dev["table"], c["layer"], dev["row_pos"],
                             dev["grp_row0"], dev["grp_nrows"], dev["grp_seq"], int(c["grp_nrows"].max()), slots,
                             max_ctx, torch.tensor(pre_len, dtype=torch.int32, device="cuda"), pre_stable=pre_stable,
                             pre_fresh=pre_fresh, workspace=workspace, err=err)
    torch.cuda.synchronize()
    return out.float().cpu(), int(err.item())


def test_flat_mode_sixty_four_ragged_sequences():
    """Flat mode (sd2_attention_flat) with the most groups a launch takes, 64 drafter-shaped groups of
    ragged lengths: groups 32..63 take the slot map's second lane half; most of the 150 slots a KV
    head has are idle. A second call on the same workspace checks that its counters reset."""
    lens = [30 + (97 * i) % 301 for i in range(64)]
    k1 = 2
    c = _case(9, seq_lens=lens, rows_per_group=[k1] * 64, H=8, Hkv=2, hd=64)
    ref = _reference(c)
    pre_len = [L - k1 for L in lens]
    ws = torch.zeros(sd2.load_library().sd2_attention_flat_workspace_bytes(2, 150, 64), dtype=torch.uint8,
                     device="cuda")
    for _ in range(2):
        out, err = _run_flat(c, 150, max(lens) + 8, pre_len, 0, k1, workspace=ws)
        assert err == 0
        _check(out, ref)


@pytest.mark.parametrize("slots", [100, 3])
def test_flat_mode_long_sequence_over_many_slots(slots):
    """Verify-shaped groups (6 rows x 4 heads, hd 128), one sequence of 2100 positions among two
    short ones. With 100 slots the per-group cap of 32 slots sets the tiles per slot (2: the long
    sequence over 17 slots); with 3 slots every group takes one."""
    lens = [2100, 70, 150]
    k1 = 6
    c = _case(10, seq_lens=lens, rows_per_group=[k1] * 3, H=8, Hkv=2, hd=128)
    ref = _reference(c)
    pre_len = [L - k1 + 1 for L in lens]      # verifier convention: rows at n-1 .. n-1+k
    out, err = _run_flat(c, slots, max(lens) + 8, pre_len, -1, k1 + 1)
    assert err == 0
    _check(out, ref)


def test_flat_mode_bad_arguments_are_rejected_on_the_host():
    c = _case(11, seq_lens=[100, 90], rows_per_group=[2, 2], H=32, Hkv=8, hd=128)
    with pytest.raises(sd2.SD2Error):
        _run_flat(c, 1, 120, [98, 88], 0, 2)       # fewer slots than groups
    with pytest.raises(sd2.SD2Error):
        _run_flat(c, 8, 64, [98, 88], 0, 2)        # a context bound of one tile


def _prompt_case(seed, seq_lens, first_rows, H, Hkv, hd):
    """Every row of each prompt from position first_rows[s] on, in groups of at most 64 query vectors;
    the cache past a prompt's end holds NaN."""
    c = _case(seed, seq_lens, [1] * len(seq_lens), H, Hkv, hd)
    cap = 64 // (H // Hkv)
    pos, r0, nr, sq = [], [], [], []
    for s, (L, f) in enumerate(zip(seq_lens, first_rows)):
        for t in range(f, L, cap):
            r0.append(len(pos))
            nr.append(min(cap, L - t))
            sq.append(s)
            pos += list(range(t, min(L, t + cap)))
        for p in range(L, 16 * c["table"].shape[1]):
            c["pool"][:, int(c["table"][s, p // 16]), :, :, p % 16] = float("nan")
    i32 = lambda v: torch.tensor(v, dtype=torch.int32)
    c.update(row_pos=i32(pos), grp_row0=i32(r0), grp_nrows=i32(nr), grp_seq=i32(sq),
             q=torch.randn(len(pos), H, hd, generator=torch.Generator().manual_seed(seed)) * 2.0)
    return c


def _prompt_reference(c):
    """_reference with the groups of a sequence taken together."""
    seqs = c["grp_seq"].tolist()
    first = [seqs.index(s) for s in sorted(set(seqs))]
    rows = [sum(int(n) for n, q in zip(c["grp_nrows"], seqs) if q == s) for s in sorted(set(seqs))]
    whole = dict(c, grp_row0=c["grp_row0"][first], grp_nrows=torch.tensor(rows), grp_seq=c["grp_seq"][first])
    return _reference(whole)


@pytest.mark.parametrize("hd,H,Hkv", [(128, 32, 8), (64, 32, 8), (64, 14, 2), (128, 4, 4), (64, 64, 1)])
@pytest.mark.parametrize("lens,first", [([300], [0]), ([64], [0]), ([17, 130, 1], [0, 0, 0]), ([200, 450], [150, 33])])
def test_prompt_rows(hd, H, Hkv, lens, first):
    """Whole prompts and the later rows of prompts (the tcgen05 kernel, which takes launches of eight tiles): pairs of groups within one
    sequence and across two, an odd number of groups, groups of 64, 63 and fewer query vectors, tiles
    partly past the prompt's end whose cache rows are not finite."""
    c = _prompt_case(12, lens, first, H, Hkv, hd)
    ref = _prompt_reference(c)
    for chunk in (64 * ((max(lens) + 63) // 64), 64 * 8):      # by its length a short prompt runs on the general kernel
        out, err = _run(c, 1, chunk, max_rows=64 // (H // Hkv))
        assert err == 0
        _check(out, ref)


def test_prompt_scores_that_keep_rising():
    """Keys that grow along the context: every tile raises the rows' maxima by far more than the
    factor at which the accumulator is rescaled."""
    c = _prompt_case(13, [400], [0], 8, 2, 128)
    ramp = torch.ones(c["pool"].shape[1] * 16)
    for b in range(c["table"].shape[1]):
        ramp[16 * int(c["table"][0, b]):][:16] = torch.arange(16 * b, 16 * b + 16) / 40.0
    c["pool"][:, :, 0] = (c["pool"][:, :, 0].float() * ramp.view(1, -1, 1, 16, 1)).to(torch.bfloat16)
    out, err = _run(c, 1, 448, max_rows=16)
    assert err == 0
    _check(out, _prompt_reference(c))


@pytest.mark.parametrize("hd,H,Hkv,k1", [(128, 32, 8, 1), (128, 32, 8, 6), (128, 16, 4, 9), (128, 64, 8, 8),
                                         (64, 8, 2, 2), (64, 14, 2, 4), (64, 32, 8, 9), (64, 14, 2, 9)])
@pytest.mark.parametrize("stable_off", [None, 0, 5])
def test_long_context_kernel_beside_the_general_one(hd, H, Hkv, k1, stable_off):
    """16 splits of 256 positions run on the long-context kernel, of 192 on the general one unless there are 48 or
    more query vectors of 128 per KV head. 8 to 64 query vectors per KV head; contexts of one position, a block's
    and a tile's edge, one row past them, and several tiles a split, with most splits empty at the short ones; with
    and without rows read early. Two sequences a launch where there are 8 KV heads: more clusters of 16 than two
    waves of them stay on the general kernel."""
    lens = [k1, 16 + k1, 128, 129, 1153, 2999]
    N = k1 * (H // Hkv)
    per = 2 if Hkv == 8 else 6
    for i in range(0, 6, per):
        some = lens[i:i + per]
        c = _case(20 + i, seq_lens=some, rows_per_group=[k1] * per, H=H, Hkv=Hkv, hd=hd)
        ref = _reference(c)
        kw = {}
        if stable_off is not None:
            kw = dict(pre_len=[max(0, L - k1 + 1 - stable_off) for L in some], pre_stable=-1, pre_fresh=k1 + stable_off + 1)
        wide = hd == 128 and N > 32
        whole = "attn_prompt" if stable_off is None and N > 32 else "attn_stream"
        outs = []
        for n_splits, chunk, kernel in ((16, 192, "attn_stream" if wide else "attn"), (16, 256, "attn_stream"),
                                        (6, 1024, "attn_stream"), (1, 4096, whole)):
            if i == 0:
                assert _kernel(c, n_splits, chunk, **kw) == kernel, (n_splits, chunk)
            out, err = _run(c, n_splits, chunk, **kw)
            assert err == 0
            _check(out, ref)
            outs.append(out)
        torch.testing.assert_close(outs[1], outs[0], atol=1.5e-2, rtol=1e-2)


@pytest.mark.parametrize("hd,k1,slots,spread", [(128, 1, 38, 12), (128, 4, 38, 12), (128, 9, 38, 12), (128, 16, 38, 12), (64, 9, 36, 24)])
def test_flat_mode_long_context_kernel(hd, k1, slots, spread):
    """Flat launches of enough tiles per slot: ragged sequences of 8 to 64 query vectors per KV head, some of
    one slot, some of several; twice on one workspace, whose counters must reset."""
    lens = [k1 + (311 * i) % (64 * spread) for i in range(13)]
    c = _case(21, seq_lens=lens, rows_per_group=[k1] * 13, H=8, Hkv=2, hd=hd)
    ref = _reference(c)
    ws = torch.zeros(sd2.load_library().sd2_attention_flat_workspace_bytes(2, slots, hd), dtype=torch.uint8, device="cuda")
    assert _kernel(c, slots, 64 * spread + 64, [L - k1 + 1 for L in lens], -1, k1 + 1, run=_run_flat) == "attn_stream"
    for _ in range(2):
        out, err = _run_flat(c, slots, 64 * spread + 64, [L - k1 + 1 for L in lens], -1, k1 + 1, workspace=ws)
        assert err == 0
        _check(out, ref)


@pytest.mark.parametrize("k1", [2, 9])
def test_long_context_scores_that_keep_rising(k1):
    """Keys that grow along the context: every tile raises the references of most query vectors."""
    c = _case(22, seq_lens=[2300], rows_per_group=[k1], H=16, Hkv=4, hd=128)
    ramp = torch.ones(c["pool"].shape[1] * 16)
    for b in range(c["table"].shape[1]):
        ramp[16 * int(c["table"][0, b]):][:16] = torch.arange(16 * b, 16 * b + 16) / 200.0
    c["pool"][:, :, 0] = (c["pool"][:, :, 0].float() * ramp.view(1, -1, 1, 16, 1)).to(torch.bfloat16)
    for n_splits, chunk in ((1, 4096), (4, 1024)):
        out, err = _run(c, n_splits, chunk)
        assert err == 0
        _check(out, _reference(c))


@pytest.mark.parametrize("hd,H,Hkv", [(128, 32, 8), (64, 14, 2), (128, 8, 1)])
@pytest.mark.parametrize("lens,first", [([1000], [0]), ([513], [385]), ([40, 33, 20, 600], [0, 1, 0, 0]), ([129, 128, 127], [0, 0, 0]),
                                        ([16, 5, 16, 3, 17, 48], [0, 0, 0, 0, 0, 0]), ([700, 30], [670, 0])])
def test_prompt_rows_four_groups_a_cta(hd, H, Hkv, lens, first):
    """CTAs whose four groups lie in one, two and more sequences (a pass each), halves of unequal contexts and
    empty ones, contexts that end in a partial cache block, on a tile's edge and one row past it."""
    c = _prompt_case(23, lens, first, H, Hkv, hd)
    out, err = _run(c, 1, max(64 * 8, 64 * ((max(lens) + 63) // 64)), max_rows=64 // (H // Hkv))
    assert err == 0
    _check(out, _prompt_reference(c))


def _kernel(c, *args, run=_run, **kw):
    """The attention kernel a launch of c runs on."""
    names = [n for n in kernels_of(lambda: run(c, *args, **kw)) if "attn" in n]
    assert len(names) == 1, names
    return next(k for k in ("attn_prompt", "attn_few", "attn_stream", "attn") if k + "_kernel" in names[0])


@pytest.mark.parametrize("hd,H,Hkv,lens,kernel", [
    (128, 32, 8, [17], "attn"), (128, 32, 8, [64, 27, 1, 1], "attn"), (128, 32, 8, [256], "attn"),
    (128, 32, 8, [192, 155, 118, 81], "attn_prompt"), (128, 32, 8, [321], "attn_prompt"), (128, 8, 2, [300], "attn"),
    (64, 32, 8, [256], "attn_prompt"),
    (64, 14, 2, [192, 155, 118, 81], "attn"), (64, 14, 2, [256, 219, 182, 145], "attn_prompt"), (64, 14, 2, [384], "attn_prompt")])
def test_short_prompts_run_on_the_general_kernel(hd, H, Hkv, lens, kernel):
    """Prompts of a few tiles and few CTAs are quicker on many small CTAs than on the tcgen05 kernel's."""
    c = _prompt_case(28, lens, [0] * len(lens), H, Hkv, hd)
    assert _kernel(c, 1, 64 * ((max(lens) + 63) // 64), max_rows=64 // (H // Hkv)) == kernel


@pytest.mark.parametrize("H,Hkv,k1,n_seq", [(32, 8, 1, 8), (32, 8, 4, 9), (14, 2, 1, 32), (14, 2, 2, 40), (16, 16, 9, 8), (32, 8, 2, 30)])
@pytest.mark.parametrize("stable_off", [0, 5])
def test_few_query_vectors_over_many_sequences(H, Hkv, k1, n_seq, stable_off):
    """Heads of 64, 4 to 16 query vectors, 64 CTAs and more (one and two to an SM): the kernel for few query
    vectors, beside the general one (without pre-step lengths, in more clusters of 16 than two waves hold). Contexts of one row, of a
    cache block's edges, shorter than the warps, of a warp's 32 blocks and one more, ragged; then flat mode."""
    edges = [k1, 16, 17, 127 + k1, 129, 8 * 16 * 6, 8 * 16 * 6 + 1, 4097 + k1]
    lens = [max(k1, edges[i] if i < len(edges) else 20 + (131 * i) % 700) for i in range(n_seq)]
    c = _case(24, lens, [k1] * n_seq, H, Hkv, 64)
    ref = _reference(c)
    kw = dict(pre_len=[max(0, L - k1 + 1 - stable_off) for L in lens], pre_stable=-1, pre_fresh=k1 + stable_off + 1)
    assert _kernel(c, 4, 1088, **kw) == "attn_few" and _kernel(c, 16, 320) == "attn"
    out, err = _run(c, 4, 1088, **kw)
    assert err == 0
    _check(out, ref)
    other, err = _run(c, 16, 320)
    assert err == 0
    _check(other, ref)
    torch.testing.assert_close(out, other, atol=1.5e-2, rtol=1e-2)
    if n_seq * Hkv >= 128:
        assert _kernel(c, n_seq, max(lens) + 16, kw["pre_len"], -1, kw["pre_fresh"], run=_run_flat) == "attn_few"
        out, err = _run_flat(c, n_seq, max(lens) + 16, kw["pre_len"], -1, kw["pre_fresh"])
        assert err == 0
        _check(out, ref)


@pytest.mark.parametrize("kind,hd,H,Hkv,k1", [("prompt", 128, 8, 2, 0), ("prompt", 64, 14, 2, 0), ("splits", 128, 32, 8, 1),
                                              ("splits", 128, 16, 4, 6), ("splits", 128, 8, 2, 16), ("splits", 64, 8, 2, 4),
                                              ("flat", 128, 8, 2, 9), ("flat", 64, 8, 2, 9)])
def test_probabilities_enter_the_products_unrounded(kind, hd, H, Hkv, k1):
    """The tcgen05 kernels form probabilities about a reference below the row's maximum, so even the largest is
    not exactly 1: they enter P V in two bf16 parts. What is left of the error against 64 bits on the same bf16
    queries, keys and values is the rounding of the result (2^-9 at most; the parts leave 2^-17, sums in f32 less):
    one bf16 part alone adds as much again, 1.2 to 1.4 times the rounding's error in all."""
    if kind == "prompt":
        c = _prompt_case(25, [900], [0], H, Hkv, hd)
        ref = _prompt_reference(c)
        out, err = _run(c, 1, 960, max_rows=64 // (H // Hkv))
    elif kind == "splits":
        c = _case(26, [4096], [k1], H, Hkv, hd)
        ref = _reference(c)
        out, err = _run(c, 16, 256)
    else:
        lens = [k1 + (311 * i) % (64 * 24) for i in range(13)]
        c = _case(27, lens, [k1] * 13, H, Hkv, hd)
        ref = _reference(c)
        out, err = _run_flat(c, 36, 64 * 24 + 64, [L - k1 + 1 for L in lens], -1, k1 + 1)
    assert err == 0
    rounding = (ref.to(torch.bfloat16).double() - ref).norm()
    assert (out.double() - ref).norm() <= 1.05 * rounding


@pytest.mark.parametrize("hd,H,Hkv", [(128, 8, 2), (64, 14, 2)])
@pytest.mark.parametrize("at", [0, 31, 32, 63, 64, 127, 128, 200, 511])
def test_prompt_scores_that_jump(hd, H, Hkv, at):
    """One key far above the others (its scores pass the reference by up to 2^80 either way), in every 32 positions
    of a tile and in later tiles: what was formed of the tile before it is rescaled with the sums and O."""
    c = _prompt_case(29, [512], [0], H, Hkv, hd)
    c["pool"][:, int(c["table"][0, at // 16]), 0, :, at % 16] *= 12.0
    out, err = _run(c, 1, 512, max_rows=64 // (H // Hkv))
    assert err == 0
    _check(out, _prompt_reference(c))
