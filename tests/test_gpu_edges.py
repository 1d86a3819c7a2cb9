"""Sizes at which the kernels change over or could slip: remainders and edges of tiles, lots and passes, the smallest and
largest of a range, runs that are merged by a warp or a block, candidates of equal D.  Everything against the CPU oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def U():
    import gpu_util
    return gpu_util


def _text(rng, n, vocab, period=60):
    """Repeats itself with a few fresh tokens in between: many equal suffixes, few nodes."""
    base = rng.integers(0, vocab, size=period)
    t = np.tile(base, n // period + 1)[:n].astype(np.int32)
    hit = rng.random(n) < 20.0 / max(n, 40)
    t[hit] = rng.integers(0, vocab, size=int(hit.sum()))
    return t


@pytest.mark.parametrize("longest,D,vocab", [(1, 1, 2), (33, 32, 3), (1024, 17, 130), (1025, 32, 50), (2049, 2, 7), (4096, 24, 128256),
                                             (4097, 32, 300), (8193, 31, 65), (16384, 32, 40), (16385, 32, 40),
                                             (32768, 32, 40), (32769, 9, 30)])
def test_prompts_at_the_edges_of_the_sorts(U, longest, D, vocab):
    """Up to eight prompts in a call: a block each up to 1,024 tokens, then a cluster of eight blocks each, above 32,768 tokens the sort of a
    whole corpus."""
    _check_prompts(U, longest, D, vocab, 0)


@pytest.mark.parametrize("n,longest,D,vocab", [(33, 1024, 32, 70), (33, 1025, 32, 50), (34, 2048, 24, 90), (33, 2049, 2, 7), (33, 4096, 17, 130),
                                               (40, 4097, 32, 300), (33, 8192, 9, 128256), (33, 8193, 31, 65), (33, 16384, 32, 40),
                                               (33, 16385, 8, 40)])
def test_prompts_at_the_edges_of_the_block_sort(U, n, longest, D, vocab):
    """More than 32 prompts in a call: a block each up to 16,384 tokens."""
    _check_prompts(U, longest, D, vocab, n)


@pytest.mark.parametrize("n,longest,D,vocab", [(17, 1025, 32, 50), (32, 2049, 24, 128256), (18, 4097, 32, 30), (17, 8193, 17, 300), (32, 16384, 32, 40),
                                               (17, 16385, 32, 40)])
def test_prompts_at_the_edges_of_clusters_of_four_blocks(U, n, longest, D, vocab):
    """17 to 32 prompts in a call: a cluster of four blocks each up to 16,384 tokens."""
    _check_prompts(U, longest, D, vocab, n)


def test_one_long_prompt_is_sorted_as_a_small_corpus(U):
    rng = np.random.default_rng(40)
    text = _text(rng, 40000, 90)
    pr = U.Pair([], vocab=90, D=16, n_slots=1, max_req_tokens=40100)
    pr.g.build_requests(np.arange(1), np.array([0, text.size]), U.dev_i32(text))
    pr.o.slot_append_batch([0], [text])
    pr.check_tree(0)
    pr.append([0], [text[:9]])
    pr.check_speculate([0], 12, 2.0, 32)
    pr.close()


def _check_prompts(U, longest, D, vocab, n):
    rng = np.random.default_rng(longest)
    lens = sorted({1, 2, 15, 16, 17, max(1, longest - 1), longest} & set(range(1, longest + 1)))
    lens += [3 + k for k in range(n - len(lens) - 1)]            # n prompts in all, if that is more
    prompts = [_text(rng, n, vocab) for n in lens] + [np.zeros(0, np.int32)]
    pr = U.Pair([], vocab=vocab, D=D, n_slots=len(prompts), max_req_tokens=longest + 8, M=32)
    off, flat = U.ragged(prompts)
    for _ in range(2):                                          # the second time over trees that are there
        pr.g.build_requests(np.arange(len(prompts)), off, U.dev_i32(flat))
    pr.o.slot_append_batch(list(range(len(prompts))), prompts)
    for s in range(len(prompts)):
        pr.check_tree(s)
    pr.append(list(range(len(prompts))), [_text(rng, 5, vocab) for _ in prompts])       # the active nodes are right
    for s in range(len(prompts)):
        pr.check_tree(s)
    pr.check_speculate(list(range(len(prompts))), 8, 2.0, 32)
    pr.close()


@pytest.mark.parametrize("n,D,vocab", [(1, 32, 5), (1023, 32, 9), (1025, 17, 4000), (9000, 24, 60), (8193, 32, 500), (65536, 32, 700),
                                       (65537, 31, 700), (303104, 3, 12), (303137, 6, 90)])
def test_corpora_at_the_edges_of_the_sort(U, n, D, vocab):
    rng = np.random.default_rng(n)
    text = _text(rng, n, vocab, period=200)
    cuts = np.unique(np.concatenate([[0, n, n], rng.integers(0, n + 1, size=6), [min(n, 1), min(n, 34)]]))
    seqs = [text[a:b] for a, b in zip(cuts[:-1], cuts[1:])]
    seqs.insert(1, np.zeros(0, np.int32))
    pr = U.Pair(seqs, vocab=vocab, D=D, n_slots=1, max_req_tokens=64)
    pr.check_tree(-1)
    want = pr.o.entropy(-1)
    assert abs(pr.g.entropy(-1) - want) <= 1e-9 * max(1.0, want)            # the tree as built
    pr.append([-1], [text[:1]])
    want = pr.o.entropy(-1)
    assert abs(pr.g.entropy(-1) - want) <= 1e-9 * max(1.0, want)            # ... and inserted into: by traversal
    pr.close()


@pytest.mark.parametrize("distinct,length,copies,halves", [(40, 40, 1500, False), (4096, 1, 1030, False), (3000, 2, 1030, False),
                                                           (900, 6, 1100, True), (1500, 2, 1024, True), (700, 1, 1023, False)])
def test_entropy_of_short_sequences_that_occur_again_and_again(distinct, length, copies, halves):
    """Every token in one place of one sequence: below the root every child is an only one, so the sum is the root's alone.  Counts on both
    sides of what is counted in shared memory, and more leaves with large ones than a block lists itself."""
    import paper_2411_04975_b200 as sfx
    D = 8
    seqs = [np.arange(distinct * length, dtype=np.int32).reshape(distinct, length)]
    if halves:
        seqs.append(seqs[0][:, :length // 2])                    # sequences end in the middle of others
    flat = np.concatenate([np.tile(s, (copies, 1)).reshape(-1) for s in seqs])
    off = np.concatenate([[0], np.cumsum(np.repeat([s.shape[1] for s in seqs], copies * distinct))])
    st = sfx.SuffixStore(torch.as_tensor(flat, device="cuda:0"), torch.as_tensor(off, device="cuda:0"), vocab=distinct * length, depth_cap=D,
                         max_requests=1, max_req_tokens=16, max_spec_cap=8, global_extra_nodes=0)
    counts = np.bincount(flat).astype(np.longdouble)
    root = counts.sum() * np.log2(counts.sum()) - (counts * np.log2(counts)).sum()
    nodes = sum(copies * distinct * sum(min(D, s.shape[1] - i) for i in range(s.shape[1])) for s in seqs)     # counts of all nodes
    want = float(root / nodes)
    assert abs(st.entropy(-1) - want) <= 1e-13 * want            # (a few roundings of 2^-53)
    st.free()


@pytest.mark.parametrize("sizes,D,vocab,fresh", [([1], 32, 4, False), ([7, 8, 9], 32, 6, False), ([511, 1, 0, 2], 17, 30, False),
                                                 ([513], 32, 2, False), ([2015], 32, 5, False), ([2016], 8, 700, True),
                                                 ([2017, 3], 32, 40, False), ([1000, 1000, 1000, 1100], 24, 900, True),
                                                 ([1920], 32, 50, False), ([1919, 2], 32, 800, True), ([961, 960, 1920], 17, 3, False)])
def test_global_insert_at_the_edges_of_a_pass(U, sizes, D, vocab, fresh):
    rng = np.random.default_rng(sum(sizes) + D)
    base = [_text(rng, 400, vocab), rng.integers(0, vocab, size=300).astype(np.int32)]
    pr = U.Pair(base, vocab=vocab, D=D, n_slots=2, max_req_tokens=64)
    for _ in range(2):
        seqs = [rng.integers(0, vocab, size=n).astype(np.int32) if fresh else _text(rng, n, vocab, 45) for n in sizes]
        pr.append([-1] * len(seqs) + [1], seqs + [base[0][:3]])
        pr.check_tree(-1)
    pr.append([0], [base[0][:20]])
    pr.check_speculate([0, 1], 12, 2.0, 32)
    pr.close()


@pytest.mark.parametrize("n,fits", [(1990, True), (1990, False), (2016, True), (2016, False), (2017, False)])
def test_what_a_full_pool_takes_goes_by_lots_of_2016(U, n, fits):
    """New strings throughout, D nodes per start position but for the last ones: a lot that does not fit adds no node, whatever part of it
    would; the one in front of it stays."""
    D, vocab = 4, 4096
    tokens = np.random.default_rng(n).permutation(vocab)[:n].astype(np.int32)
    nodes = sum(min(D, n - i) for i in range(n))
    last = sum(min(D, n - i) for i in range(2016)) if n > 2016 else 0    # nodes of the lots in front of the last one
    pr = U.Pair([], vocab=vocab, D=D, n_slots=1, max_req_tokens=16, global_extra_nodes=nodes if fits else nodes - 1)
    off, flat = U.ragged([tokens])
    pr.g.append(U.dev_i32([-1]), torch.as_tensor(off, device=U.DEV), U.dev_i32(flat))
    st = pr.g.stats()
    assert st["global_pool_cap"] == (nodes if fits else nodes - 1)
    assert st["global_status"] == (0 if fits else 4)
    assert st["global_nodes"] == (nodes if fits else last)
    pr.close()


@pytest.fixture
def small_clusters():
    import paper_2411_04975_b200 as sfx
    sfx.library().sd_debug_small_clusters(1)
    yield
    sfx.library().sd_debug_small_clusters(0)


@pytest.mark.parametrize("sizes,D,vocab,fresh", [([7, 8, 9], 32, 6, False), ([513], 32, 2, False), ([2015], 32, 5, False), ([2016], 8, 700, True),
                                                 ([2017, 3], 32, 40, False), ([1000, 1000, 1000, 1100], 24, 900, True)])
def test_global_insert_without_a_cluster(U, small_clusters, sizes, D, vocab, fresh):
    test_global_insert_at_the_edges_of_a_pass(U, sizes, D, vocab, fresh)


@pytest.mark.parametrize("n,fits", [(2016, True), (2016, False), (2017, False)])
def test_what_a_full_pool_takes_without_a_cluster(U, small_clusters, n, fits):
    test_what_a_full_pool_takes_goes_by_lots_of_2016(U, n, fits)


@pytest.mark.parametrize("n,D,vocab", [(1025, 17, 4000), (32768, 32, 500), (32769, 24, 60), (65536, 32, 700)])
def test_corpora_without_large_clusters(U, small_clusters, n, D, vocab):
    test_corpora_at_the_edges_of_the_sort(U, n, D, vocab)


def test_global_insert_merges_long_runs(U):
    """One token with hundreds of children: runs that move and runs with room, merged by a block, children of which get children."""
    rng = np.random.default_rng(5)
    vocab = 4000
    def fan(tokens):
        return np.stack([np.zeros(len(tokens), np.int64), tokens], 1).reshape(-1).astype(np.int32)
    perm = 1 + rng.permutation(vocab - 1)
    pr = U.Pair([fan(perm[:600])], vocab=vocab, D=4, n_slots=1, max_req_tokens=64)
    for lo, hi in ((550, 950), (950, 960), (0, 300), (960, 1500), (1500, 1501)):
        pr.append([-1, -1], [fan(perm[lo:hi]), fan(perm[hi - 1:lo:-7])])
        pr.check_tree(-1)
    pr.append([0], [np.array([3, 0], np.int32)])
    pr.check_speculate([0], 4, 4.0, 64)
    pr.close()


@pytest.mark.parametrize("fan,deep,budget", [(2, 20, 64), (31, 3, 64), (32, 2, 64), (33, 2, 64), (30, 1, 64), (40, 6, 48)])
def test_candidates_of_equal_d(U, fan, deep, budget):
    """A node with `fan` children that all occur equally often, each the start of a chain, and of further fans: equal D in
    numbers up to and above a warp and the pool."""
    rng = np.random.default_rng(fan * 100 + deep)
    seqs = []
    for c in range(fan):
        chain = (rng.permutation(500)[:deep] + 100 * (c % 3)).tolist()
        for e in range(3 if deep < 4 else 1):
            seqs.append(np.array([7, 8, 10 + c] + chain + [900 + (e * 37 + c) % 60, 960 + e], np.int32))
    wide = [np.array([7, 9, 10 + c, 700 + e], np.int32) for c in range(min(fan, 30)) for e in range(30)]
    pr = U.Pair(seqs + wide, vocab=1024, D=32, n_slots=3, max_req_tokens=64)
    pr.append([0, 1, 2], [np.array([7, 8], np.int32), np.array([7, 9], np.int32), np.array([5, 7], np.int32)])
    for flags in (0, 4):
        pr.check_speculate([0, 1, 2], 3, 32.0, budget, flags=flags)
    pr.close()


def test_a_bad_token_leaves_the_slots_as_they_are(U):
    import paper_2411_04975_b200 as sfx
    rng = np.random.default_rng(9)
    pr = U.Pair([], vocab=20, D=8, n_slots=3, max_req_tokens=200)
    pr.append([0, 1, 2], [_text(rng, 50, 20) for _ in range(3)])
    prompts = [_text(rng, 120, 20), _text(rng, 90, 20)]
    off, flat = U.ragged(prompts)
    flat[130] = 20
    for _ in range(2):
        with pytest.raises(sfx.SuffixSpecError) as e:
            pr.g.build_requests([2, 0], off, U.dev_i32(flat))
        assert e.value.code == -1
        for s in range(3):
            pr.check_tree(s)
        pr.check_speculate([0, 1, 2], 8, 2.0, 32)
    pr.close()


def test_memory_kept_between_stores_is_bounded():
    import paper_2411_04975_b200 as sfx
    torch.cuda.synchronize()
    free0, total = torch.cuda.mem_get_info()
    for k in range(6):
        stores = [sfx.SuffixStore(None, None, vocab=1000, depth_cap=32, max_requests=64, max_req_tokens=2000 + 997 * j + 311 * k, max_spec_cap=64)
                  for j in range(3)]
        for s in stores:
            s.free()
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= total // 32 + (64 << 20)


@pytest.mark.parametrize("name,bad,error", [
    ("slots", lambda t: t.long(), TypeError), ("slots", lambda t: t.cpu(), TypeError), ("slots", lambda t: None, Exception),
    ("offsets", lambda t: t.int(), TypeError), ("new_tokens", lambda t: t.repeat(2)[::2], TypeError),
    ("new_tokens", lambda t: t.tolist(), Exception), ("P", lambda t: "4", TypeError), ("alpha", lambda t: None, TypeError),
    ("budget_cap", lambda t: torch.ones(3, dtype=torch.float32, device="cuda"), TypeError), ("out", lambda t: {}, KeyError)])
def test_arguments_of_the_calls_of_every_step(U, name, bad, error):
    pr = U.Pair([], vocab=20, D=8, n_slots=3, max_req_tokens=200)
    pr.append([0, 1, 2], [np.arange(9, dtype=np.int32) % 4 for _ in range(3)])
    args = dict(slots=U.dev_i32(np.arange(3)), offsets=torch.zeros(4, dtype=torch.int64, device="cuda"), new_tokens=U.dev_i32(np.zeros(2)),
                P=4, alpha=2.0, max_spec=8, flags=0, budget_cap=None, out=None, tau=0.0)
    bad_args = dict(args, **{name: bad(args[name])})
    with pytest.raises(error):
        pr.g.step(**bad_args)
    if name in ("slots", "P", "alpha", "budget_cap", "out"):
        with pytest.raises(error):
            pr.g.speculate(**{k: v for k, v in bad_args.items() if k not in ("offsets", "new_tokens")})
    host = {k: v.pin_memory() if isinstance(v, torch.Tensor) else v for k, v in
            dict(args, slots=args["slots"].cpu(), offsets=args["offsets"].cpu(), new_tokens=args["new_tokens"].cpu()).items()}
    a, b = pr.g.step(**args), pr.g.step(**host)                 # the store is as it was; pinned host tensors are taken
    for k in ("n_draft", "chosen_tree", "chosen_p", "score", "status"):
        assert torch.equal(a[k], b[k])
    pr.close()


@pytest.mark.parametrize("children,most", [(33, 3), (128, 9), (129, 1), (300, 2), (300, 40), (140, 140),
                                           (62, 4), (63, 1), (63, 5), (64, 2), (65, 7), (127, 60)])
def test_long_runs_without_a_ready_list_in_the_middle_of_a_tree(U, children, most):
    rng = np.random.default_rng(children + most)
    counts = np.full(children, 131) if most == 140 else rng.integers(1, most + 1, children)
    heads = rng.permutation(np.repeat(np.arange(children), counts))
    text = np.concatenate([np.stack([np.full(heads.size, 1), np.full(heads.size, 2), 10 + heads], 1).reshape(-1), [5, 1]]).astype(np.int32)
    pr = U.Pair([], vocab=1024, D=6, n_slots=1, max_req_tokens=text.size + 8)
    off, flat = U.ragged([text])
    pr.g.build_requests(np.arange(1), off, U.dev_i32(flat))
    pr.o.slot_append_batch([0], [text])
    for budget in (8.0, 63.0):
        for flags in (0, 4):
            pr.check_speculate([0], 2, budget, 64, flags=flags)
    pr.close()


@pytest.mark.parametrize("budget", [33, 35, 36, 37, 39, 41, 64])
def test_the_least_of_a_long_runs_best_children_stays_a_candidate(U, budget):
    """40 children: the first occurs 50 times, the last 12 times, those between ten times or once.  The first one's children need more places
    than are left: what goes then goes by the least of the best, wherever it stands in the run."""
    first = [60] * 20 + list(range(61, 91))
    seqs = [np.array([7, 10, e, 95], np.int32) for e in first]
    seqs += [np.array([7, 10 + c, 60 + e, 95], np.int32) for c, k in zip(range(1, 40), [10] * 34 + [1] * 4 + [12]) for e in range(k)]
    pr = U.Pair(seqs, vocab=100, D=8, n_slots=200, max_req_tokens=16)
    slots = list(range(200))
    pr.append(slots, [np.array([7], np.int32)] * 200)
    for some in (slots[:1], slots):                             # one block per SM, and two
        for flags in (0, 4):
            pr.check_speculate(some, 1, float(budget), 64, flags=flags)
    pr.close()


def test_trim_gives_back_what_freed_stores_left():
    import paper_2411_04975_b200 as sfx
    sfx.sd_trim()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    store = sfx.SuffixStore(None, None, vocab=1000, depth_cap=32, max_requests=64, max_req_tokens=4000, max_spec_cap=64)
    store.free()
    assert free0 - torch.cuda.mem_get_info()[0] > (100 << 20)            # kept for the next store
    sfx.sd_trim()
    assert free0 - torch.cuda.mem_get_info()[0] < (8 << 20)


@pytest.mark.parametrize("outer,inner", [(31, 32), (40, 20), (40, 30), (60, 32), (64, 5), (70, 31), (31, 3), (31, 5), (28, 17), (32, 9)])
def test_more_candidates_than_a_job_has_places_for(U, outer, inner):
    """Candidates of equal D from several fans until there is no place: the best stay, by token and parent where D is equal."""
    rng = np.random.default_rng(outer * 100 + inner)
    seqs = [np.array([7, 10 + c, 100 + e, 300 + (c + e) % 9], np.int32) for c in rng.permutation(outer) for e in rng.permutation(inner)]
    pr = U.Pair(seqs, vocab=400, D=8, n_slots=1, max_req_tokens=16)
    pr.append([0], [np.array([7], np.int32)])
    for budget in (64.0, 41.0):
        for flags in (0, 4):
            pr.check_speculate([0], 1, budget, 64, flags=flags)
    pr.close()


@pytest.mark.parametrize("total", [2, 510, 511, 512, 1023])
def test_quotients_on_both_sides_of_the_table_of_reciprocals(U, total):
    rng = np.random.default_rng(total)
    cuts = np.sort(rng.choice(np.arange(1, total), size=min(total - 1, 11), replace=False))
    counts = np.diff(np.concatenate([[0], cuts, [total]]))
    seqs = [np.array([7, 10 + c, 50 + (c + e) % 3, 60], np.int32) for c, k in enumerate(counts) for e in range(k)]
    pr = U.Pair(seqs, vocab=100, D=8, n_slots=1, max_req_tokens=16)
    pr.append([0], [np.array([7], np.int32)])
    pr.check_speculate([0], 1, 40.0, 64)
    pr.close()


@pytest.mark.parametrize("n_slots,new", [(2, 1), (12, 2), (40, 9)])
def test_match_nodes_found_while_prompts_are_sorted(U, n_slots, new):
    """New prompts of more than a block's step: their match nodes, and those an insert has made stale, come with the sort."""
    rng = np.random.default_rng(n_slots)
    base = [_text(rng, 3000, 60), _text(rng, 500, 60)]
    pr = U.Pair(base, vocab=60, D=32, n_slots=n_slots, max_req_tokens=1700)
    every = list(range(n_slots))

    def build(slots, bad=False):
        prompts = [_text(rng, 1100 + 37 * k, 60, 90) for k in range(len(slots))]
        off, flat = U.ragged(prompts)
        if bad:
            flat[-1] = 60
            with pytest.raises(Exception):
                pr.g.build_requests(np.array(slots), off, U.dev_i32(flat))
            return
        pr.g.build_requests(np.array(slots), off, U.dev_i32(flat))
        for k in slots:
            pr.o.slot_reset(k)
        pr.o.slot_append_batch(slots, prompts)

    for k in range(0, n_slots, 9):
        build(every[k:k + 9])
    for turn in range(3):
        pr.check_speculate(every, 20, 2.0, 40)
        pr.append([-1, 0], [_text(rng, 700, 60, 30), base[1][:5]])               # (the drafts' match nodes are stale now)
        if turn == 1:
            build(every[:new], bad=True)                                         # a refused call leaves them right, too
        else:
            build(every[-new:])
        pr.append(every, [base[0][k:k + 1 + k % 4] for k in every])
    pr.check_speculate(every, 20, 2.0, 40)
    pr.close()


@pytest.mark.parametrize("n", [40, 200, 400])
def test_slots_that_appear_twice_in_batches_of_every_shape(U, n):
    """One block per SM, two and four: the later appearances are refused, also while the first ones' match nodes are out of date."""
    rng = np.random.default_rng(n)
    pr = U.Pair([_text(rng, 2000, 50)], vocab=50, D=16, n_slots=n, max_req_tokens=100)
    pr.append(list(range(n)), [_text(rng, int(k), 50) for k in rng.integers(20, 80, n)])
    call = rng.integers(0, n, n)
    call[:3] = call[-1]
    first = np.sort(np.unique(call, return_index=True)[1])
    again = np.setdiff1d(np.arange(n), first)
    for turn in range(6):
        got = {k: v.cpu().numpy() for k, v in pr.g.speculate(U.dev_i32(call), 12, 2.0, 40).items()}
        got["mask"] = got["mask"].view(np.uint32)
        assert (got["status"][first] == 0).all() and (got["status"][again] == 1).all()
        assert (got["n_draft"][again] == 0).all() and (got["chosen_tree"][again] == -1).all()
        U.assert_same_drafts({k: v[first] for k, v in got.items()}, pr.o.speculate(call[first].tolist(), 12, 2.0, 40, M=64, n_threads=4))
        some = rng.permutation(n)[:n // 2].tolist()              # every other turn the global tree changes, too
        pr.append(some + [-1] * (turn % 2), [_text(rng, 2, 50) for _ in some] + [_text(rng, 90, 50)] * (turn % 2))
    pr.close()


def test_prompts_sorted_beside_steps_and_inserts_on_other_streams(U):
    """sd_build_requests has nothing to do with the other slots and the global tree: steps of those and inserts into that may be at work on
    other streams.  What it finds out for them meanwhile is taken for the text that it was found for only."""
    rng = np.random.default_rng(12)
    vocab, old, new, D = 40, 100, 4, 24
    pr = U.Pair([_text(rng, 4000, vocab)], vocab=vocab, D=D, n_slots=old + new, max_req_tokens=2400)
    every, a, b = list(range(old + new)), torch.cuda.Stream(), torch.cuda.Stream()
    first = [_text(rng, int(k), vocab) for k in rng.integers(5, 60, old + new)]
    pr.append(every, first)

    def build():
        prompts = [_text(rng, 1100 + 200 * k, vocab, 90) for k in range(new)]
        off, flat = U.ragged(prompts)
        flat = U.dev_i32(flat)
        torch.cuda.synchronize()

        def call():
            with torch.cuda.stream(a):
                pr.g.build_requests(np.arange(old, old + new), off, flat)
            torch.cuda.synchronize()
            for k in range(new):
                pr.o.slot_reset(old + k)
            pr.o.slot_append_batch(every[old:], prompts)
        return call

    for turn in range(8):
        pr.append([-1], [_text(rng, 300, vocab, 30)])            # the match nodes are stale
        lists = [_text(rng, 1 + (k + turn) % 7, vocab) for k in range(old)]
        off, flat = U.ragged(lists)
        args = (U.dev_i32(every[:old]), torch.as_tensor(off, device=U.DEV), U.dev_i32(flat))
        call = build()
        with torch.cuda.stream(b):
            pr.g.step(*args, 20, 2.0, 40)
        call()
        pr.o.slot_append_batch(every[:old], lists, n_threads=4)
        pr.check_speculate(every, 20, 2.0, 40)
        seqs = [_text(rng, 700, vocab, 50), _text(rng, 90, vocab)]
        off, flat = U.ragged(seqs)
        args = (U.dev_i32([-1, -1]), torch.as_tensor(off, device=U.DEV), U.dev_i32(flat))
        call = build()
        with torch.cuda.stream(b):
            pr.g.append(*args)
        call()
        for s in seqs:
            pr.o.global_insert(s)
        pr.check_speculate(every[::2], 20, 2.0, 40)
        pr.append([-1], [_text(rng, 80, vocab)])
        build()()                                                # leaves match nodes for all ...
        pr.append(every[:40], [_text(rng, 70, vocab) for _ in range(40)], reset=[1] * 40)       # ... of which some have another text now
        pr.append(every[30:60], [_text(rng, 3, vocab) for _ in range(30)])
        pr.check_speculate(every, 20, 2.0, 40)
    pr.check_tree(-1)
    pr.close()
