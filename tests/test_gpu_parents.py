"""GPU parity for parents that are not contiguous spans: the nearest-centre assignment that closes
Algorithm 3, Algorithm 2 on parents of any size with empty parents omitted, and a decode step over
records whose team count differs between the KV heads of a sequence. Integer results (labels, CSR
offsets, member order, representative rows, sampled teams) must match the fp64 oracle exactly.
"""
import numpy as np
import pytest
import torch

from oracle import santapp_oracle as orc
from paper_2609_35629_b200 import binding as sp
from paper_2609_35629_b200 import synth

import parity_util as pu
from test_gpu_parity import check_dense_step, check_sparse_step

pytestmark = pytest.mark.gpu


def _spec(prompt=(1536, 1000), n_sample=8, R=4, n_clusters=24):
    spec = synth.spec_small_gqa(n_seqs=len(prompt), prompt=prompt, n_sample=n_sample)
    spec.reps_per_parent = R
    spec.parent_size = 64
    spec.n_clusters = n_clusters
    return spec


def _centres_for(spec, data, n_centres):
    """fp32 centres per KV head and sequence: the generating centres of the synthetic keys, with
    traps: a repeated centre (an exact tie), a centre far from every key (an empty parent) and a
    centre that coincides with one key (a parent of very few tokens)."""
    rng = np.random.default_rng(99)
    out = np.zeros((spec.n_kv_heads, sum(n_centres), spec.head_dim), dtype=np.float32)
    off = 0
    row0 = 0
    for b, n in enumerate(n_centres):
        for j in range(spec.n_kv_heads):
            c = data.centres[j, rng.permutation(spec.n_clusters)[:n]].copy()
            if n >= 4:
                c[n - 1] = c[0]                                        # tie: never wins
                c[n - 2] = 100.0                                       # attracts nothing
                key = synth.bf16_to_f32(data.k_prompt[j, row0 + 7])
                c[n - 3] = key                                         # sits on token 7
            out[j, off:off + n] = c
        off += n
        row0 += spec.prompt_len[b]
    return out


def _labels_gpu(spec, data, n_centres, centres):
    geom = pu.geometry(spec)
    k = sp.bf16_bits_to_cuda(data.k_prompt)
    lab = sp.santapp_assign_parents(geom, spec.prompt_len, n_centres, k, torch.from_numpy(centres).cuda())
    torch.cuda.synchronize()
    return lab.cpu().numpy()


def test_assignment_matches_the_oracle_with_ties_and_empty_centres():
    spec = _spec()
    data = synth.make_layer(spec, layer=0, keep_centres=True)
    n_centres = [24, 9]
    centres = _centres_for(spec, data, n_centres)
    lab = _labels_gpu(spec, data, n_centres, centres)
    row0 = c0 = 0
    for b, n in enumerate(n_centres):
        N = spec.prompt_len[b]
        for j in range(spec.n_kv_heads):
            keys = synth.bf16_to_f64(data.k_prompt[j, row0:row0 + N])
            want, ps, _ = orc.nearest_centre_parents(keys, centres[j, c0:c0 + n].astype(np.float64))
            assert np.array_equal(lab[j, row0:row0 + N], want)
            assert not np.any(want == n - 1) and not np.any(want == n - 2)     # the traps stayed empty
            assert ps.shape[0] - 1 < n
        row0 += N
        c0 += n


def _check_records(layer, labels, n_parents):
    spec = layer.spec
    for b in range(spec.n_seqs):
        r0, r1 = int(layer.seq_row_off[b]), int(layer.seq_row_off[b + 1])
        N = r1 - r0
        slots = int(layer.seq_team_off[b + 1] - layer.seq_team_off[b])
        assert slots == min(N, n_parents[b] * spec.reps_per_parent)
        for j in range(spec.n_kv_heads):
            keys = synth.to_f64(layer.data.k_prompt[j, r0:r1], spec.elem)
            lab = np.clip(labels[j, r0:r1], 0, n_parents[b] - 1)
            kept = np.unique(lab)
            ps = np.concatenate([[0], np.cumsum([np.count_nonzero(lab == u) for u in kept])]).astype(np.int32)
            pm = np.concatenate([np.flatnonzero(lab == u) for u in kept]).astype(np.int32)
            ts_o, tm_o, rep_o = orc.build_teams(keys, ps, pm, spec.reps_per_parent)
            ts_g, tm_g, rep_g = layer.records(b, j)
            assert len(ts_g) == len(ts_o), "team count"
            assert np.array_equal(ts_g, ts_o)
            assert np.array_equal(tm_g, tm_o)
            assert np.array_equal(rep_g, keys[rep_o])
            assert np.array_equal(layer.k_packed_bits[j, r0:r1], layer.data.k_prompt[j, r0:r1][tm_g])
            assert np.array_equal(layer.v_packed_bits[j, r0:r1], layer.data.v_prompt[j, r0:r1][tm_g])
            # slots behind the last team are empty teams
            t0 = int(layer.seq_team_off[b])
            M = len(ts_o) - 1
            tail = layer.team_row_start[j, t0 + b + M: t0 + b + slots + 1]
            assert np.all(tail == N)
            assert not layer.rep_bits[j, t0 + M: t0 + slots].any()


def _layer_from_labels(spec, data, labels, n_parents):
    lab_dev = torch.from_numpy(np.ascontiguousarray(labels, dtype=np.int32)).cuda()

    def builder(geom, prompt_len, k, v):
        return sp.santapp_build_teams_parents(geom, prompt_len, n_parents, k, v, lab_dev)
    return pu.GpuLayer(spec, data, builder=builder)


def test_records_from_centre_parents_match_algorithm_2_of_the_oracle():
    spec = _spec()
    data = synth.make_layer(spec, layer=0, keep_centres=True)
    n_centres = [24, 9]
    labels = _labels_gpu(spec, data, n_centres, _centres_for(spec, data, n_centres))
    layer = _layer_from_labels(spec, data, labels, n_centres)
    _check_records(layer, labels, n_centres)
    for step in range(2):
        check_sparse_step(layer, step, spec.n_sample)
    check_dense_step(layer, 0)


def test_records_from_arbitrary_labels_large_and_single_token_parents():
    """Labels that no clustering would produce: one parent of 1200 tokens (more than any contiguous
    parent may hold), single-token parents, empty labels, labels outside the range (clamped), and
    a different partition for each KV head."""
    spec = _spec(prompt=(1536, 700), n_sample=6, R=8)
    data = synth.make_layer(spec, layer=0, keep_centres=True)
    rng = np.random.default_rng(4)
    n_parents = [40, 12]
    labels = np.zeros((spec.n_kv_heads, spec.rows_total), dtype=np.int32)
    for j in range(spec.n_kv_heads):
        a = rng.integers(2, 36, size=1536)
        a[rng.permutation(1536)[:1200]] = 1                            # the big parent, scattered
        a[5], a[900] = 37, 38                                          # singletons
        a[6] = -3                                                      # clamped to 0
        a[7] = 1000                                                    # clamped to 39
        bseq = rng.integers(0, 12 - j, size=700)                       # head j never uses its last labels
        labels[j] = np.concatenate([a, bseq])
    layer = _layer_from_labels(spec, data, labels, n_parents)
    _check_records(layer, labels, n_parents)
    check_sparse_step(layer, 0, spec.n_sample)
    check_dense_step(layer, 0)


def test_pair_with_fewer_teams_than_the_budget_reads_every_team():
    """One KV head of a sequence ends up with at most K teams while the others have more: that pair
    reads all its teams uncorrected (K = min(K, M) in Algorithm 1), the others sample."""
    spec = _spec(prompt=(600, 512), n_sample=8, R=4)
    data = synth.make_layer(spec, layer=0, keep_centres=True)
    rng = np.random.default_rng(8)
    n_parents = [16, 16]
    labels = np.zeros((spec.n_kv_heads, spec.rows_total), dtype=np.int32)
    for j in range(spec.n_kv_heads):
        labels[j, :600] = rng.integers(0, 16, size=600)
        labels[j, 600:] = rng.integers(0, 16, size=512)
    labels[1, :600] = rng.integers(3, 5, size=600)                     # two parents: 8 teams = K
    labels[2, 600:] = 9                                                # one parent: 4 teams < K
    layer = _layer_from_labels(spec, data, labels, n_parents)
    _check_records(layer, labels, n_parents)
    assert int(layer.team_count[1, 0]) == 8 and int(layer.team_count[2, 1]) == 4
    assert int(layer.team_count[0, 0]) == 64
    for step in range(2):
        check_sparse_step(layer, step, spec.n_sample)


def test_contiguous_builder_reports_every_slot_as_a_team():
    spec = synth.spec_small_gqa()
    layer = pu.GpuLayer(spec, synth.make_layer(spec, layer=0))
    want = np.diff(layer.seq_team_off).astype(np.int32)
    assert np.array_equal(layer.team_count, np.tile(want, (spec.n_kv_heads, 1)))


def _centre_layer(spec):
    """The configuration `bench.py --parents centres` times: as many of the generating centres as the
    first line of Algorithm 3 asks for, assignment and records built on the GPU."""
    data = synth.make_layer(spec, layer=0, keep_centres=True)
    n_cen = [min(sp.santapp_kmeans_parent_count(n, spec.parent_size), spec.n_clusters) for n in spec.prompt_len]
    cen = np.ascontiguousarray(np.concatenate([data.centres[:, :n] for n in n_cen], axis=1))
    labels = _labels_gpu(spec, data, n_cen, cen)
    return _layer_from_labels(spec, data, labels, n_cen), labels, n_cen, cen


def test_centre_parents_32k_full_size():
    """Config 2's shape with parents from centres instead of contiguous spans: labels and records of
    one KV head against the oracle, then decode steps of every head."""
    spec = synth.spec_qwen_b1()
    layer, labels, n_cen, cen = _centre_layer(spec)
    j = 1
    keys = synth.bf16_to_f64(layer.data.k_prompt[j])
    want, ps, pm = orc.nearest_centre_parents(keys, cen[j].astype(np.float64))
    assert np.array_equal(labels[j], want)
    ts_o, tm_o, rep_o = orc.build_teams(keys, ps, pm, spec.reps_per_parent)
    ts_g, tm_g, rep_g = layer.records(0, j)
    assert np.array_equal(ts_g, ts_o) and np.array_equal(tm_g, tm_o) and np.array_equal(rep_g, keys[rep_o])
    sizes = np.diff(ps)
    assert sizes.max() > spec.parent_size                      # parents larger than any contiguous one
    for step in (0, 255):
        check_sparse_step(layer, step, K=32)
    check_dense_step(layer, 3)


def test_centre_parents_paper_point_32k():
    """The paper's operating point (P = 16, R = 4, K = 31) on centre parents: 2048 parents of uneven
    size, a different team count for every KV head."""
    spec = synth.spec_paper_point()
    layer, _, _, _ = _centre_layer(spec)
    assert len({int(c) for c in layer.team_count[:, 0]}) > 1
    check_sparse_step(layer, 0, K=31)


def test_centroid_groups_on_centre_parents():
    """The paper's centroid-guided baseline on a clustering's groups (nominal group size 16): one
    group per non-empty parent routed by its mean key; records equal to the oracle's, decode as usual."""
    spec = _spec(prompt=(2048, 1100), n_sample=12, R=1, n_clusters=128)
    spec.parent_size = 16
    data = synth.make_layer(spec, layer=0, keep_centres=True)
    n_centres = [sp.santapp_kmeans_parent_count(n, spec.parent_size) for n in spec.prompt_len]     # 128, 68
    cen = np.ascontiguousarray(np.concatenate([data.centres[:, :n] for n in n_centres], axis=1))
    labels = _labels_gpu(spec, data, n_centres, cen)
    lab_dev = torch.from_numpy(labels).cuda()

    def builder(geom, prompt_len, k, v):
        return sp.santapp_build_groups_mean_parents(geom, prompt_len, n_centres, k, v, lab_dev)
    layer = pu.GpuLayer(spec, data, builder=builder)
    for b in range(spec.n_seqs):
        r0, r1 = int(layer.seq_row_off[b]), int(layer.seq_row_off[b + 1])
        for j in range(spec.n_kv_heads):
            keys = synth.bf16_to_f64(data.k_prompt[j, r0:r1])
            _, ps, pm = orc.nearest_centre_parents(keys, cen[j, sum(n_centres[:b]):sum(n_centres[:b + 1])].astype(np.float64))
            ts_o, tm_o, mean_o = orc.group_mean_keys_parents(keys, ps, pm)
            ts_g, tm_g, rep_g = layer.records(b, j)
            assert np.array_equal(ts_g, ts_o) and np.array_equal(tm_g, tm_o) and np.array_equal(rep_g, mean_o)
            assert np.array_equal(layer.k_packed_bits[j, r0:r1], data.k_prompt[j, r0:r1][tm_g])
    for step in range(2):
        check_sparse_step(layer, step, spec.n_sample)
    bad = pu.geometry(_spec(prompt=(2048, 1100), R=4))
    with pytest.raises(sp.SantappError):
        sp.santapp_build_groups_mean_parents(bad, spec.prompt_len, n_centres, layer.k_prompt, layer.v_prompt, lab_dev)


def test_null_team_count_means_every_slot_is_a_team():
    """Records of the contiguous builder fill every slot, so the decode must give the same bits with
    team_count left NULL (callers that built their records before the field existed)."""
    spec = synth.spec_small_gqa()
    layer = pu.GpuLayer(spec, synth.make_layer(spec, layer=0))
    q_bits = synth.make_queries(spec, layer.data, 0)
    sl = spec.suffix_len(0)
    out_a, dbg_a = pu.gpu_step(layer, q_bits, sl, spec.n_sample, 5, 0)
    saved = layer.teams.c.team_count
    layer.teams.c.team_count = None
    try:
        out_b, dbg_b = pu.gpu_step(layer, q_bits, sl, spec.n_sample, 5, 0)
        dense_b, _ = pu.gpu_step(layer, q_bits, sl, 0, 0, 0, dense=True)
    finally:
        layer.teams.c.team_count = saved
    dense_a, _ = pu.gpu_step(layer, q_bits, sl, 0, 0, 0, dense=True)
    assert np.array_equal(out_a, out_b) and np.array_equal(dense_a, dense_b)
    assert torch.equal(dbg_a.sel_idx, dbg_b.sel_idx)


@pytest.mark.parametrize("elem,far", [("fp16", 6000.0), ("fp16", 60000.0), ("bf16", 1e20), ("bf16", np.inf), ("bf16", np.nan)])
@pytest.mark.parametrize("at", [(0,), (40,), (97,), (150,), (299,), (5, 6, 33, 290)])
def test_assignment_with_centres_whose_norm_the_products_cannot_bound(elem, far, at):
    """Centres far outside the range of the bounds (squared norm beyond 4.2e9 for fp16 calls, 1e37 for bf16), or not
    numbers, among 300 ordinary ones, in every column half and tile of the scan: ordinary tokens still go to
    the nearest of all centres, exact ties to the smaller index (the last 30 ordinary centres repeat earlier ones)."""
    rng = np.random.default_rng([len(at), at[0]])
    N, k = 700, 300
    cen = rng.standard_normal((1, k, 128)).astype(np.float32)
    cen[0, 270:] = cen[0, rng.permutation(270)[:30]]
    keys = cen[0, rng.integers(0, k, size=N)] + 0.7 * rng.standard_normal((N, 128)).astype(np.float32)
    cen[0, list(at)] = np.float32(far)
    bits = synth.round_bits(keys[None], elem)
    geom = sp.Geometry(1, 1, 1, 128, 16, 4, sp.SANTAPP_FP16 if elem == "fp16" else sp.SANTAPP_BF16)
    lab = sp.santapp_assign_parents(geom, [N], [k], sp.bf16_bits_to_cuda(bits, dtype=geom.torch_dtype), torch.from_numpy(cen).cuda())
    want, _, _ = orc.nearest_centre_parents(synth.to_f64(bits[0], elem), cen[0].astype(np.float64))
    assert np.array_equal(lab[0].cpu().numpy(), want)
    assert len(set(want.tolist())) > 200 and not set(at) & set(want.tolist())


@pytest.mark.parametrize("size", [20, 100, 400, 700])
def test_records_of_parents_with_keys_that_are_not_numbers(size):
    """One key of a parent that is not a number makes its mean, and so every distance to it, not a number: the first
    representative is then the parent's first key, for parents of every kernel's sizes. The other parents'
    records are the oracle's."""
    rng = np.random.default_rng(size)
    N, n_parents, R = 3 * size, 3, 6
    labels = rng.permutation(np.repeat(np.arange(3), size)).astype(np.int32)
    bits = synth.round_bits(rng.standard_normal((1, N, 128)).astype(np.float32))
    bad = int(np.flatnonzero(labels == 1)[size // 2])
    bits[0, bad, 77] = 0x7FC0
    geom = sp.Geometry(1, 1, 1, 128, 3 * R, R)
    k = sp.bf16_bits_to_cuda(bits)
    t = sp.santapp_build_teams_parents(geom, [N], [n_parents], k, k, torch.from_numpy(labels[None]).cuda())
    csr, token = t.team_row_start[0, :3 * R + 1].cpu().numpy(), t.row_token[0].cpu().numpy()
    rep = t.rep_keys.view(torch.int16).cpu().numpy().view(np.uint16)[0]
    assert np.array_equal(np.sort(token), np.arange(N)) and np.all(np.diff(csr) >= 0)
    assert np.array_equal(rep[R], bits[0, np.flatnonzero(labels == 1)[0]])
    for u in (0, 2):
        rows = np.flatnonzero(labels == u).astype(np.int32)
        ts, tm, _ = orc.build_teams(synth.to_f64(bits[0]), np.array([0, size], dtype=np.int32), rows, R)
        assert np.array_equal(csr[u * R:u * R + R + 1] - u * size, ts) and np.array_equal(token[u * size:(u + 1) * size], tm[:size])


def _repeated(kind, n, rng):
    if kind == "few":                            # 40 distinct rows
        return rng.standard_normal((40, 128))[rng.integers(0, 40, size=n)]
    if kind == "same":
        return np.repeat(rng.standard_normal((1, 128)), n, axis=0)
    if kind == "padded":                         # half of them zero
        return rng.standard_normal((n, 128)) * (np.arange(n) < n // 2)[:, None]
    if kind == "some":                           # one in sixteen zero
        return rng.standard_normal((n, 128)) * (np.arange(n) % 16 > 0)[:, None]
    return rng.integers(-1, 2, size=(n, 128))    # "integer": many distinct rows at exactly equal distances


@pytest.mark.parametrize("kind", ["few", "same", "padded", "some", "integer"])
@pytest.mark.parametrize("elem,offset", [("bf16", 0), ("fp16", 1)])
def test_assignment_to_centres_that_repeat(kind, elem, offset):
    """Centres drawn from keys that repeat: the bounds leave every token, or few of a block, more candidates than are
    compared one by one. The centres' rows start at a 16-byte boundary and beside one."""
    rng = np.random.default_rng(len(kind))
    N, k = 900, 333
    bits = synth.round_bits(_repeated(kind, N, rng).astype(np.float32)[None], elem)
    keys = synth.to_f64(bits[0], elem)
    cen = keys[rng.integers(0, N, size=k)].astype(np.float32)
    cen[5] += 1e-6
    geom = sp.Geometry(1, 1, 1, 128, 16, 4, sp.SANTAPP_FP16 if elem == "fp16" else sp.SANTAPP_BF16)
    room = torch.zeros(k * 128 + 4, device="cuda")
    room[offset:offset + k * 128] = torch.from_numpy(cen.ravel())
    lab = sp.santapp_assign_parents(geom, [N], [k], sp.bf16_bits_to_cuda(bits, dtype=geom.torch_dtype),
                                    room[offset:offset + k * 128].view(1, k, 128))
    want, _, _ = orc.nearest_centre_parents(keys, cen.astype(np.float64))
    assert np.array_equal(lab[0].cpu().numpy(), want)


def test_tokens_that_the_bounds_leave_open_cost_their_fp64_distances_and_no_more():
    """512 centres of which eight and eight are equal, so that every token goes through all of them: about twelve times the
    usual call (the distances in fp64, which the call took for any centres before the bounds); 150 when each
    token's scan read its centres one lane each."""
    g = torch.Generator(device="cuda").manual_seed(3)
    N, k, geom = 8192, 512, sp.Geometry(1, 4, 4, 128, 16, 4)
    rows = torch.randn(4, N, 128, generator=g, device="cuda").to(torch.bfloat16)

    def microseconds(keys, cen):
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sp.santapp_assign_parents(geom, [N], [k], keys, cen)
            b.record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
        return best

    usual = microseconds(rows, rows[:, :k].float().contiguous())
    repeated = rows[:, :64].repeat(1, N // 64, 1)
    assert microseconds(repeated, repeated[:, :k].float().contiguous()) < 40 * usual


@pytest.mark.parametrize("n_centres", [[1, 2], [8, 3], [2, 9]])
@pytest.mark.parametrize("elem", ["bf16", "fp16"])
def test_assignment_to_few_centres(n_centres, elem):
    """Up to eight centres in every sequence, and one more in one: the two kernels of the assignment on ragged sequences."""
    rng = np.random.default_rng(n_centres)
    lens = [257, 130]
    bits = synth.round_bits(rng.standard_normal((2, sum(lens), 128)).astype(np.float32), elem)
    cen = rng.standard_normal((2, sum(n_centres), 128)).astype(np.float32)
    cen[0, -1] = cen[0, n_centres[0]]                                  # an exact tie, or the centre itself
    cen[1, 0] = np.nan if n_centres[0] > 1 else cen[1, 0]              # never the nearest
    geom = sp.Geometry(2, 2, 2, 128, 16, 4, sp.SANTAPP_FP16 if elem == "fp16" else sp.SANTAPP_BF16)
    lab = sp.santapp_assign_parents(geom, lens, n_centres, sp.bf16_bits_to_cuda(bits, dtype=geom.torch_dtype), torch.from_numpy(cen).cuda())
    for j in range(2):
        for r0, c0, n, k in ((0, 0, lens[0], n_centres[0]), (lens[0], n_centres[0], lens[1], n_centres[1])):
            want, _, _ = orc.nearest_centre_parents(synth.to_f64(bits[j, r0:r0 + n], elem), cen[j, c0:c0 + k].astype(np.float64))
            assert np.array_equal(lab[j, r0:r0 + n].cpu().numpy(), want)
