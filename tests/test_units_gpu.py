"""GPU parity at the edges of the decode kernel's work split: contexts that
end just before, at and after the edges of a 16-token box and of a unit (16
tokens at d = 128, 32 at d = 64), against the fp64 oracle.

Bars as in test_parity_gpu.py (max |err| <= 1.5e-2, mean |err| <= 2e-3, the
pool bit-exact): bf16 outputs of fp32 sums over N(0, 1) values.
"""
import numpy as np
import pytest

import oracle
from paper_2606_12950_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MAX_ABS = 1.5e-2
MEAN_ABS = 2e-3


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _check(got, ref, what):
    err = np.abs(got - ref)
    assert np.isfinite(got).all(), what
    assert err.max() <= MAX_ABS and err.mean() <= MEAN_ABS, (what, err.max(), err.mean())


def _nan_past_contexts(b):
    """NaN bit patterns in every row of a sequence's blocks past its context,
    and in every block that no sequence holds."""
    view = b.pool.reshape(b.n_pages, 2, b.Hkv, b.bs, b.d)
    held = np.zeros(b.n_pages, bool)
    for s in range(b.S):
        n = int(b.ctx_lens[s])
        blocks = b.table[s, : -(-n // b.bs)]
        held[blocks] = True
        if n % b.bs:
            view[blocks[-1], :, :, n % b.bs:, :] = 0xFFFF
    view[~held] = 0xFFFF


@pytest.mark.parametrize("fused", [False, True], ids=["separate", "fused"])
@pytest.mark.parametrize("variant", [1, 2])
@pytest.mark.parametrize("bs", [16, 32, 64])
@pytest.mark.parametrize("d", [64, 128])
def test_context_lengths_at_box_and_unit_edges(d, bs, variant, fused):
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    pre = [0, 14, 15, 16, 30, 31, 32, 46, 47, 48, 62, 63, 64, 95, 127, 500, 1023]
    b = W.make_batch(7000 + d + bs, pre, Hq=8, Hkv=2, d=d, bs=bs, extra_blocks=5)
    _nan_past_contexts(b)
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(b.Hkv, b.d)])
    pool.upload(b.pool)
    pool.set_variant(variant)
    db = DeviceBatch(pool, 0, b)
    if fused:
        db.append_attend()
    else:
        db.append()
        db.attend()
    torch.cuda.synchronize()
    ref_pool = oracle.batch_append(b)
    assert np.array_equal(pool.download(), ref_pool)
    _check(db.out_f64(), oracle.batch_attention(b, pool=ref_pool), (d, bs, variant, fused))
    assert pool.error() == 0


def _attend(b, max_blocks=None):
    """Fused append + attention of batch b, its table widened to max_blocks."""
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    if max_blocks is not None:
        wide = np.full((b.S, max_blocks), -1, np.int32)
        wide[:, : b.max_blocks] = b.table
        b.table, b.max_blocks = wide, max_blocks
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(b.Hkv, b.d)])
    pool.upload(b.pool)
    db = DeviceBatch(pool, 0, b)
    db.append_attend()
    torch.cuda.synchronize()
    assert pool.error() == 0
    return pool, db


@pytest.mark.parametrize("G,d", [(1, 64), (4, 128), (5, 64), (8, 128)])
@pytest.mark.parametrize("S", [1, 2, 76, 77, 152, 153])
def test_combine_with_few_and_many_runs(S, G, d):
    """One KV head, so S runs: either side of the lines at which the combine
    spreads a run's columns over 8, 4 or 1 CTAs (152 SMs), with runs of one
    record and, with one or two sequences, of several hundred: 60000 tokens are
    six units or more for each of 304 CTAs, more records than the 16 groups of
    a combine CTA take at once (8 each)."""
    lens = [60000 if S < 3 else 700] + [17 + 41 * s % 333 for s in range(1, S)]
    b = W.make_batch(7100 + S + G, lens, Hq=G, Hkv=1, d=d, bs=16, extra_blocks=3)
    pool, db = _attend(b)
    ref_pool = oracle.batch_append(b)
    assert np.array_equal(pool.download(), ref_pool)
    _check(db.out_f64(), oracle.batch_attention(b, pool=ref_pool), (S, G, d))


MERGE_LENS = {
    "one_token": [0],
    "under_a_warp": [15, 40],
    "many_short": [1 + 37 * s % 90 for s in range(40)],
    "one_long": [5000],
    "long_and_short": [3000, 5, 700, 31, 1, 2047, 16, 64],
}


@pytest.mark.parametrize("lens", MERGE_LENS.values(), ids=MERGE_LENS.keys())
@pytest.mark.parametrize("G,Hkv,d", [(1, 4, 128), (4, 8, 128), (8, 1, 128), (5, 2, 64), (4, 8, 64)])
def test_cta_level_parts_against_the_oracle_and_the_general_path(G, Hkv, d, lens):
    """A small batch merges its warps' records inside each CTA; the same batch
    with a table too wide for that takes the general path.  Both against the
    oracle, and against each other.  The two paths round a token's weight to
    bf16 against different running maxima, 2^-9 of it at most on each side, so
    they differ by at most 2 * 2^-9 * sum(p |v|) <= 2^-8 max|v|, and by the
    outputs' own rounding, 2^-9 |out| on each side (the fp32 sums add less
    than 2^-16 of that)."""
    outs = []
    for width in (None, 16384):
        b = W.make_batch(7200 + G + d, lens, Hq=G * Hkv, Hkv=Hkv, d=d, bs=16, extra_blocks=3)
        _nan_past_contexts(b)
        pool, db = _attend(b, width)
        ref_pool = oracle.batch_append(b)
        assert np.array_equal(pool.download(), ref_pool)
        outs.append(db.out_f64())
        _check(outs[-1], oracle.batch_attention(b, pool=ref_pool), (G, Hkv, d, width))
    vals = W.bf16_bits_to_f64(ref_pool)
    vmax = np.abs(vals[np.isfinite(vals)]).max()
    assert np.all(np.abs(outs[0] - outs[1]) <= 2.0 ** -8 * (vmax + np.abs(outs[1])))


def test_cta_level_parts_with_a_shared_prefix():
    """Short suffixes beside the prefix kernel: every member leaves a record,
    also where its suffix lies inside one CTA."""
    from paper_2606_12950_gb300 import kvpool as K
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    pre = [256 + n for n in (0, 3, 16, 47, 300, 64)] + [90, 33]
    groups = [(list(range(6)), 256)]
    b = W.make_batch(7300, pre, Hq=8, Hkv=2, d=128, bs=16, extra_blocks=3)
    W.share_prefix(b, groups)
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(b.Hkv, b.d)])
    pool.upload(b.pool)
    db = DeviceBatch(pool, 0, b)
    db.cascade(K.PrefixPlan(groups))
    torch.cuda.synchronize()
    ref_pool = oracle.batch_append(b)
    assert np.array_equal(pool.download(), ref_pool)
    _check(db.out_f64(), oracle.batch_attention(b, pool=ref_pool), "prefix")
    assert pool.error() == 0


@pytest.mark.parametrize("G,Hkv,d", [(4, 8, 128), (8, 1, 128), (2, 2, 64)])
@pytest.mark.parametrize("tokens", [64, 192, 448, 576, 4160])
def test_key_splits_of_a_shared_prefix(tokens, G, Hkv, d):
    """Few members, so the prefix is cut into as many key splits as it has
    64-token chunks, eight at most: splits of one chunk (a half tile), of an
    odd number of chunks, and of more tiles than are asked of L2 ahead."""
    from paper_2606_12950_gb300 import kvpool as K
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    groups = [([0, 1, 2], tokens), ([4, 5], tokens)]
    pre = [tokens, tokens + 16, tokens + 333, 50, tokens, tokens + 100]
    b = W.make_batch(7400 + tokens + G, pre, Hq=G * Hkv, Hkv=Hkv, d=d, bs=16, extra_blocks=3)
    W.share_prefix(b, groups)
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(b.Hkv, b.d)])
    pool.upload(b.pool)
    db = DeviceBatch(pool, 0, b)
    db.cascade(K.PrefixPlan(groups))
    torch.cuda.synchronize()
    ref_pool = oracle.batch_append(b)
    assert np.array_equal(pool.download(), ref_pool)
    _check(db.out_f64(), oracle.batch_attention(b, pool=ref_pool), (tokens, G))
    assert pool.error() == 0


@pytest.mark.parametrize("lens", MERGE_LENS.values(), ids=MERGE_LENS.keys())
@pytest.mark.parametrize("G,Hkv,d,variant", [(1, 4, 128, 2), (4, 8, 128, 2), (8, 1, 128, 2), (4, 2, 64, 2), (4, 2, 64, 1)])
def test_records_per_warp_and_per_cta_give_the_same_bits(G, Hkv, d, variant, lens):
    """A table too wide for the small-batch rule: alone a call merges its warps'
    records in the CTAs, after another call's combine (step overlap) it leaves
    them to the combine.  The same bits, also with fewer units than warps, with
    one CTA and with several."""
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    b = W.make_batch(7500 + G + d, lens, Hq=G * Hkv, Hkv=Hkv, d=d, bs=16, extra_blocks=3)
    wide = np.full((b.S, 16384), -1, np.int32)
    wide[:, : b.max_blocks] = b.table
    b.table, b.max_blocks = wide, 16384
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(b.Hkv, b.d)])
    pool.upload(b.pool)
    pool.set_variant(variant)
    for splits in (0, 1, 3):
        db = DeviceBatch(pool, 0, b, splits)
        db.append_attend()
        torch.cuda.synchronize()
        alone = db.out_bits()
        pool.set_step_overlap(True)
        for _ in range(3):
            db.append_attend()
        torch.cuda.synchronize()
        pool.set_step_overlap(False)
        assert np.array_equal(alone, db.out_bits()), splits
    _check(db.out_f64(), oracle.batch_attention(b, pool=oracle.batch_append(b)), (G, Hkv, d))
    assert pool.error() == 0


@pytest.mark.parametrize("G,Hkv,d", [(1, 8, 128), (4, 4, 64)])
@pytest.mark.parametrize("splits", [1, 2, 3, 16, 40, 0])
def test_combine_by_part(splits, G, Hkv, d):
    """Many more runs than parts (with the splits given; at 0, 2560 runs on 304
    CTAs): the combine has a CTA per part, for the run that starts there.  Runs
    inside a part, over two and over many, empty sequences, and parts without
    units; against the oracle, and bit for bit against the same call overlapping
    another's combine, which has a CTA per run."""
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    S = 2560 // Hkv if splits == 0 else 200 // Hkv * 2
    lens = [7 + 29 * s % 150 for s in range(S)]
    lens[3], lens[S // 2], lens[S - 1] = 6000, 900, 2000
    width = None
    if splits == 40:  # one unit a run, so most of the CTAs have none
        lens, width = [3 + s % 12 for s in range(400 // Hkv)], 4096
    b = W.make_batch(7600 + G + d, lens, Hq=G * Hkv, Hkv=Hkv, d=d, bs=16, extra_blocks=3, max_blocks=width)
    post = b.ctx_lens.copy()
    post[[0, 5, 6]] = 0  # empty
    b.ctx_lens = post
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(b.Hkv, b.d)])
    pool.upload(b.pool)
    db = DeviceBatch(pool, 0, b, splits)
    db.attend()
    torch.cuda.synchronize()
    alone = db.out_bits()
    _check(db.out_f64(), oracle.batch_attention(b, pool=b.pool), (splits, G))
    pool.set_step_overlap(True)
    for _ in range(3):
        db.attend()
    torch.cuda.synchronize()
    assert np.array_equal(alone, db.out_bits())
    assert pool.error() == 0


def _long_run_units(span, short_runs, P, min_units, before=5):
    """Units of a run that starts after `before` one-unit runs and ends `span`
    parts after the one it starts in, by the kernel's cut: W units in NC equal
    ranges, NC = min(max(W // (6 * min_units), 1), P)."""
    for n in range(2, 1 << 16):
        w = short_runs + n
        nc = min(max(w // (6 * min_units), 1), P)
        begin = np.arange(nc + 1) * w // nc
        first, last = np.searchsorted(begin, [before, before + n - 1], "right") - 1
        if last - first == span:
            return n
    raise AssertionError(span)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("G", [1, 2, 4, 5, 8])
def test_combine_by_part_finds_the_end_of_a_run(G, d):
    """A combine CTA per part, and a run that ends 1 to 49 parts after the one it
    starts in: the look for its end takes one pass or two, by warps of 32 lanes
    and, with 80 threads a CTA (G = 5 at d = 64), of 16.  Every output is
    written (NaN before the call), against the oracle, and bit for bit as the
    overlapped form, which has a combine CTA per run.

    Contexts of a token or a few have outputs as large as the values, so the bar
    is the roundings' bound: a weight to bf16, 2^-9 of it, so 2^-9 max|v| of the
    output; the output itself, 2^-9 |out|; fp32 sums, below 2^-6 of those."""
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    P, S, unit = 60, 600, 32 if d == 64 else 16
    for span in (1, 15, 16, 17, 31, 32, 33, 49):
        lens = [s % 15 for s in range(S)]
        lens[5] = _long_run_units(span, S - 1, P, 64 // unit) * unit - 3
        b = W.make_batch(7800 + span + G, lens, Hq=G, Hkv=1, d=d, bs=16, extra_blocks=3)
        pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(1, d)])
        pool.upload(b.pool)
        db = DeviceBatch(pool, 0, b, P)
        db.out.fill_(float("nan"))
        db.attend()
        torch.cuda.synchronize()
        alone = db.out_bits()
        ref = oracle.batch_attention(b, pool=b.pool)
        vmax = np.abs(W.bf16_bits_to_f64(b.pool)).max()
        assert np.all(np.abs(db.out_f64() - ref) <= (2.0 ** -9 + 2.0 ** -15) * (vmax + np.abs(ref))), (span, G, d)
        pool.set_step_overlap(True)
        db.attend()
        db.out.fill_(float("nan"))
        db.attend()
        torch.cuda.synchronize()
        assert np.array_equal(alone, db.out_bits()), (span, G, d)
        assert pool.error() == 0


@pytest.mark.parametrize("G,d,S", [(1, 64, 14302), (1, 64, 15100), (1, 64, 16349), (8, 64, 15901), (4, 128, 13725)])
def test_the_most_sequences_a_call_takes(G, d, S):
    """S up to what the sequence index of a CTA leaves room for beside a 16-token
    box of K and of V for each of six warps, whatever a unit holds: the last S
    of each form is that limit, and one more is refused."""
    from paper_2606_12950_gb300 import kvpool as K
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    lens = [s % 19 for s in range(S)]
    lens[7], lens[S - 3] = 3000, 700
    b = W.make_batch(7900 + G, lens, Hq=G, Hkv=1, d=d, bs=16, extra_blocks=3)
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(1, d)])
    pool.upload(b.pool)
    db = DeviceBatch(pool, 0, b)
    db.append_attend()
    torch.cuda.synchronize()
    alone = db.out_bits()
    ref_pool = oracle.batch_append(b)
    assert np.array_equal(pool.download(), ref_pool)
    ref = oracle.batch_attention(b, pool=ref_pool)
    # contexts of a token or a few: the bound of the roundings (see above)
    vmax = np.abs(W.bf16_bits_to_f64(ref_pool)).max()
    assert np.all(np.abs(db.out_f64() - ref) <= (2.0 ** -9 + 2.0 ** -15) * (vmax + np.abs(ref)))
    pool.set_step_overlap(True)
    for _ in range(3):
        db.append_attend()
    torch.cuda.synchronize()
    assert np.array_equal(alone, db.out_bits())
    assert pool.error() == 0
    if S in (16349, 15901, 13725):
        with pytest.raises(K.KVError):
            K.kv_workspace_bytes(pool.handle, 0, S + 1, G, b.max_blocks, 0)


def _exact(b, pool, s):
    """Sequence s of batch b in 64 bits (NaN and infinities as IEEE has them)."""
    n = int(b.ctx_lens[s])
    kv = W.bf16_bits_to_f64(pool).reshape(-1, 2, b.Hkv, b.bs, b.d)[b.table[s, : -(-n // b.bs)]]
    k, v = (kv[:, i].transpose(1, 0, 2, 3).reshape(b.Hkv, -1, b.d)[:, :n] for i in (0, 1))
    q = W.bf16_bits_to_f64(b.q[s]).reshape(b.Hkv, b.G, b.d)
    with np.errstate(all="ignore"):
        x = q @ k.transpose(0, 2, 1) * b.scale
        w = np.exp(x - x.max(-1, keepdims=True))
        return ((w / w.sum(-1, keepdims=True)) @ v).reshape(b.Hq, b.d)


@pytest.mark.parametrize("path", ["small", "per_cta", "per_warp", "cuda_cores", "prefix"])
@pytest.mark.parametrize("d", [64, 128])
def test_nan_and_infinite_scores(d, path):
    """A token whose score is NaN makes its sequence's output NaN, and one whose
    score is -inf has no weight, wherever the token is: alone in the run's last
    unit (the new token), the first token, all of the first units, one in the
    middle.  In every form of the records; the other sequences are as ever."""
    from paper_2606_12950_gb300 import kvpool as K
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    pre = [448, 448, 1000, 1000, 2048, 2048, 700, 330, 5000]
    b = W.make_batch(8000 + d, pre, Hq=8, Hkv=2, d=d, bs=16, extra_blocks=3)
    groups = [([4, 5, 6], 256)]
    if path == "prefix":
        W.share_prefix(b, groups)
    one, nan, ninf = 0x3F80, 0x7FC0, 0xFF80
    b.q[:, :, 0] = one
    rows = b.pool.reshape(b.n_pages, 2, b.Hkv, b.bs, b.d)

    def set_k(s, pos, bits):
        rows[b.table[s, pos // b.bs], 0, 1, pos % b.bs, 0] = bits  # KV head 1

    b.k_new[0, 1, 0] = nan      # the new token, the only one of its unit
    b.k_new[1, 1, 0] = ninf
    set_k(2, 0, nan)
    for pos in range(64):       # whole units without a score
        set_k(3, pos, ninf)
    if path == "prefix":        # in the shared prefix: a NaN that all members see
        set_k(4, 130, nan)
        nan_seqs = [0, 2, 4, 5, 6]
    else:
        set_k(4, 1030, nan)
        for pos in range(512):
            set_k(5, pos, ninf)
        nan_seqs = [0, 2, 4]
    if path in ("per_cta", "per_warp", "cuda_cores"):  # a table too wide for the small batches' rule
        wide = np.full((b.S, 16384), -1, np.int32)
        wide[:, : b.max_blocks] = b.table
        b.table, b.max_blocks = wide, 16384
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(b.Hkv, b.d)])
    pool.upload(b.pool)
    pool.set_variant(1 if path == "cuda_cores" else 2)
    db = DeviceBatch(pool, 0, b)
    if path == "prefix":
        db.cascade(K.PrefixPlan(groups))
    else:
        db.append_attend()
    if path == "per_warp":
        pool.set_step_overlap(True)
        for _ in range(2):
            db.append_attend()
    torch.cuda.synchronize()
    got, ref_pool = db.out_f64().reshape(b.S, b.Hq, d), oracle.batch_append(b)
    for s in range(b.S):
        ref = _exact(b, ref_pool, s)
        if s in nan_seqs:
            assert np.isnan(got[s, 4:]).all() and np.isnan(ref[4:]).all(), s
            _check(got[s, :4], ref[:4], (s, path))
        else:
            _check(got[s], ref, (s, path))
    assert pool.error() == 0


@pytest.mark.parametrize("d", [64, 128])
def test_shared_prefix_whose_first_keys_have_no_weight(d):
    """-inf scores in the first 192 keys of a shared prefix: more than the first
    128-key tile of the prefix kernel."""
    from paper_2606_12950_gb300 import kvpool as K
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    groups = [([0, 1, 2], 2048)]
    b = W.make_batch(8100 + d, [2048, 2100, 2500, 40], Hq=8, Hkv=2, d=d, bs=16, extra_blocks=3)
    W.share_prefix(b, groups)
    b.q[:, :, 0] = 0x3F80
    rows = b.pool.reshape(b.n_pages, 2, b.Hkv, b.bs, b.d)
    for pos in range(192):
        rows[b.table[0, pos // b.bs], 0, :, pos % b.bs, 0] = 0xFF80
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(b.Hkv, b.d)])
    pool.upload(b.pool)
    db = DeviceBatch(pool, 0, b)
    db.cascade(K.PrefixPlan(groups))
    torch.cuda.synchronize()
    ref_pool = oracle.batch_append(b)
    got = db.out_f64().reshape(b.S, b.Hq, d)
    for s in range(b.S):
        _check(got[s], _exact(b, ref_pool, s), s)
    assert pool.error() == 0


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("lens", [[[30]] * 3, [[200, 90], [700, 33, 5, 260, 1, 64], [500]], [[3000], [2900, 64], [2500] * 3],
                                  [[0], [900] * 6, [15, 16, 17]], [[100, 600], [30, 500, 7], [20] * 39 + [3900]]],
                         ids=["one_cta", "ragged", "long", "uneven", "beside_a_large_one"])
def test_small_batches_in_one_call(lens, d):
    """Co-located batches that are small: from one unit a warp on, by the room of
    all of them, CTAs without units among the chained kernels.  The same bits
    in each of 20 steps; against the oracle, and against the calls one by one within the roundings of two work splits
    (see test_cta_level_parts_against_the_oracle_and_the_general_path)."""
    from paper_2606_12950_gb300 import kvpool as K
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    heads = [(8, 2), (8, 8), (32, 4)]
    for order in (slice(None), slice(None, None, -1)):
        batches = [W.make_batch(8200 + d + i, pre, Hq=Hq, Hkv=Hkv, d=d, bs=16, extra_blocks=3)
                   for i, (pre, (Hq, Hkv)) in enumerate(zip(lens[order], heads))]
        page = 2 * 2 * 16 * d  # elements of the smallest block
        first, n_pages, parts = [], 0, []
        for b in batches:  # each batch's blocks in pages of their own
            k = b.block_elems // page
            b.table = np.where(b.table >= 0, b.table * k + n_pages, -1).astype(np.int32)
            parts.append(b.pool)
            first.append(n_pages)
            n_pages += b.n_pages * k
        host = np.concatenate(parts)
        outs = []
        for multi in (False, True):
            pool = DevicePool(n_pages, page * 2, 16, [(b.Hkv, d) for b in batches])
            pool.upload(host)
            dbs = [DeviceBatch(pool, i, b) for i, b in enumerate(batches)]
            if multi:
                calls = K.attn_batches([db.batch() for db in dbs])
                steps = []
                for _ in range(20):
                    K.paged_decode_attn_multi(pool.handle, calls)
                    steps.append([db.out.clone() for db in dbs])
                torch.cuda.synchronize()
                for s in steps[:-1]:
                    assert all(torch.equal(x, y) for x, y in zip(s, steps[-1]))
            else:
                for db in dbs:
                    db.append_attend()
            torch.cuda.synchronize()
            assert pool.error() == 0
            outs.append([db.out_f64() for db in dbs])
            got_pool = pool.download()
            ref_pool = host.copy()
            for i, b in enumerate(batches):
                oracle.append(ref_pool, n_pages, page, 16, b.Hkv, d, b.k_new, b.v_new, b.table, b.ctx_lens, inplace=True)
            assert np.array_equal(got_pool, ref_pool)
        vmax = np.abs(W.bf16_bits_to_f64(ref_pool)).max()
        for i, b in enumerate(batches):
            ref = oracle.paged_attention(ref_pool, n_pages, page, 16, b.Hkv, d, b.q, b.table, b.ctx_lens, b.scale)
            for got in (outs[0][i], outs[1][i]):
                assert np.all(np.abs(got - ref) <= (2.0 ** -9 + 2.0 ** -15) * (vmax + np.abs(ref))), i
            assert np.all(np.abs(outs[0][i] - outs[1][i]) <= 2.0 ** -8 * (vmax + np.abs(ref))), i


@pytest.mark.parametrize("splits", [303, 305, 700, 3000])
@pytest.mark.parametrize("lens", [[8000], [40, 700, 3, 1500, 64, 333, 900, 1999], [s % 40 for s in range(60)]],
                         ids=["one", "some", "short"])
@pytest.mark.parametrize("G,Hkv,d", [(4, 8, 128), (5, 2, 64)])
def test_more_splits_than_resident_ctas(G, Hkv, d, lens, splits):
    """num_splits either side of the CTAs that are resident (304 on 152 SMs) and far
    above, in small batches: against the oracle (the bound of the roundings, see
    above), and the same bits overlapping another call's combine."""
    from paper_2606_12950_gb300.runner import DeviceBatch, DevicePool

    b = W.make_batch(8300 + G, lens, Hq=G * Hkv, Hkv=Hkv, d=d, bs=16, extra_blocks=3)
    pool = DevicePool(b.n_pages, b.page_elems * 2, b.bs, [(Hkv, d)])
    pool.upload(b.pool)
    db = DeviceBatch(pool, 0, b, splits)
    db.append_attend()
    torch.cuda.synchronize()
    alone, ref_pool = db.out_bits(), oracle.batch_append(b)
    assert np.array_equal(pool.download(), ref_pool)
    ref = oracle.batch_attention(b, pool=ref_pool)
    vmax = np.abs(W.bf16_bits_to_f64(ref_pool)).max()
    assert np.all(np.abs(db.out_f64() - ref) <= (2.0 ** -9 + 2.0 ** -15) * (vmax + np.abs(ref)))
    pool.set_step_overlap(True)
    for _ in range(3):
        db.append_attend()
    torch.cuda.synchronize()
    assert np.array_equal(alone, db.out_bits())
    assert pool.error() == 0
