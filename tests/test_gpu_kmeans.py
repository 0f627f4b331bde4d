"""GPU parity for the minibatch k-means fit of Algorithm 3: the CUDA fit and the fp64 oracle take
the same random words and the same fp64 arithmetic in the same order, so centres (rounded to fp32)
and step counts must be equal, not merely close."""
import numpy as np
import pytest
import torch

from oracle import santapp_oracle as orc
from paper_2609_35629_b200 import binding as sp
from paper_2609_35629_b200 import synth

import parity_util as pu

pytestmark = pytest.mark.gpu


def _fit_both(spec, n_centres, **opts):
    data = synth.make_layer(spec, layer=0, keep_centres=True)
    geom = pu.geometry(spec)
    k = sp.bf16_bits_to_cuda(data.k_prompt, dtype=geom.torch_dtype)
    centres, steps = sp.santapp_kmeans_fit(geom, spec.prompt_len, n_centres, k, **opts)
    torch.cuda.synchronize()
    centres, steps = centres.cpu().numpy(), steps.cpu().numpy()
    base = opts.get("stream_base", 0)
    o = {kk: v for kk, v in opts.items() if kk not in ("stream_base", "no_host_poll")}
    o = {"batch": o.pop("batch_size", 4096), "ratio": o.pop("reassignment_ratio", 0.01), **o}
    row0 = c0 = 0
    for b, kc in enumerate(n_centres):
        N = spec.prompt_len[b]
        for j in range(spec.n_kv_heads):
            keys = synth.to_f64(data.k_prompt[j, row0:row0 + N], spec.elem)
            want, want_steps = orc.minibatch_kmeans(keys, kc, stream=base + b * spec.n_kv_heads + j, **o)
            assert int(steps[j, b]) == want_steps, f"steps of pair ({b}, {j})"
            assert np.array_equal(centres[j, c0:c0 + kc], want.astype(np.float32)), f"centres of pair ({b}, {j})"
        row0 += N
        c0 += kc
    return data, centres, steps


def test_fit_matches_the_oracle_on_two_ragged_sequences():
    spec = synth.spec_small_gqa(prompt=(1536, 1000))
    spec.n_clusters = 24
    n_centres = [24, 9]
    _, _, steps = _fit_both(spec, n_centres, batch_size=256, seed=3, stream_base=11)
    assert steps.min() >= 10


def test_fit_with_reassignment_every_period_and_short_patience():
    """A high ratio moves centres at every period, a patience of 2 stops early, k is not a multiple of
    the centres a block updates, and the sample is the whole sequence."""
    spec = synth.spec_small_gqa(prompt=(700,), n_seqs=1, suffix0=(0,))
    _fit_both(spec, [13], batch_size=512, reassignment_ratio=0.9, patience=2, max_iter=30, seed=1 << 40)
    _fit_both(spec, [13], batch_size=64, reassignment_ratio=0.0, patience=10 ** 6, max_iter=2)


def test_fit_without_host_polling_gives_the_same_centres():
    """With no_host_poll the call never waits for the stream: every step up to the limit is enqueued
    and the steps of a fit that has already stopped do nothing, so centres and step counts stay
    those of the oracle (two sequences whose fits stop at different steps)."""
    spec = synth.spec_small_gqa(prompt=(1536, 1000))
    spec.n_clusters = 24
    _, _, steps = _fit_both(spec, [24, 9], batch_size=256, seed=3, stream_base=11, max_iter=20, no_host_poll=True)
    assert len(set(steps.ravel().tolist())) > 1
    assert steps.max() < 20 * 6                                 # the fits stopped before the limit


def test_fit_without_host_polling_can_be_captured_in_a_cuda_graph():
    """With no_host_poll the call only enqueues work: captured in a CUDA graph on a side stream and
    replayed twice, it leaves the centres and step counts of the plain call (which the test above
    compares with the oracle)."""
    spec = synth.spec_small_gqa(prompt=(1536, 1000))
    spec.n_clusters = 24
    data = synth.make_layer(spec, layer=0, keep_centres=True)
    geom = pu.geometry(spec)
    k = sp.bf16_bits_to_cuda(data.k_prompt, dtype=geom.torch_dtype)
    opts = dict(batch_size=256, seed=3, stream_base=11, max_iter=20, no_host_poll=True)
    want_c, want_s = sp.santapp_kmeans_fit(geom, spec.prompt_len, [24, 9], k, **opts)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        got_c, got_s = sp.santapp_kmeans_fit(geom, spec.prompt_len, [24, 9], k, **opts)
    for _ in range(2):
        got_c.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(got_c, want_c) and torch.equal(got_s, want_s)


def test_fit_on_a_sequence_too_long_for_the_shared_memory_shuffle():
    """52000 keys beside 900: more indices than shared memory holds, of which the initialisation sample takes the head
    of a shuffle (entries found one by one, without the list), beside a sequence whose sample is all of it."""
    spec = synth.spec_small_gqa(prompt=(52000, 900), suffix0=(0, 0))
    spec.n_clusters = 16
    _fit_both(spec, [11, 6], batch_size=192, seed=5, max_iter=3, patience=4)


def test_fit_of_150_short_sequences_takes_its_tables_in_two_chunks():
    """More sequences than one kernel-argument chunk of the per-sequence tables holds (128)."""
    rng = np.random.default_rng(9)
    lens = tuple(int(x) for x in rng.integers(30, 70, size=150))
    spec = synth.spec_small_gqa(n_seqs=150, prompt=lens, suffix0=(0,) * 150)
    spec.n_clusters = 4
    _fit_both(spec, [2 + (i % 3) for i in range(150)], batch_size=16, seed=2, max_iter=2, patience=3)


def test_fit_fp16_inputs():
    spec = synth.spec_small_gqa(prompt=(900,), n_seqs=1, suffix0=(0,))
    spec.elem = "fp16"
    _fit_both(spec, [7], batch_size=128)


def test_fit_then_parents_then_decode():
    """Algorithm 3 end to end on the GPU (count, fit, assignment, omission of empty parents), then
    Algorithm 2 and a decode step on the result, each against the oracle."""
    from test_gpu_parents import _check_records, _layer_from_labels
    from test_gpu_parity import check_sparse_step
    spec = synth.spec_small_gqa(prompt=(2048, 1200))
    spec.parent_size, spec.reps_per_parent, spec.n_clusters = 64, 4, 32
    n_centres = [sp.santapp_kmeans_parent_count(n, spec.parent_size) for n in spec.prompt_len]
    assert n_centres == [32, 18]
    data, centres, _ = _fit_both(spec, n_centres, batch_size=512)
    geom = pu.geometry(spec)
    k = sp.bf16_bits_to_cuda(data.k_prompt)
    labels = sp.santapp_assign_parents(geom, spec.prompt_len, n_centres, k, torch.from_numpy(centres).cuda())
    torch.cuda.synchronize()
    labels = labels.cpu().numpy()
    keys = synth.bf16_to_f64(data.k_prompt[2, :2048])
    want, _, _ = orc.nearest_centre_parents(keys, centres[2, :32].astype(np.float64))
    assert np.array_equal(labels[2, :2048], want)
    layer = _layer_from_labels(spec, data, labels, n_centres)
    _check_records(layer, labels, n_centres)
    check_sparse_step(layer, 0, spec.n_sample)


def _one_pair_at_full_size(spec, j, **opts):
    """Fit every pair on the GPU, check one KV head against the oracle (the oracle takes seconds per pair)."""
    data = synth.make_layer(spec, layer=0)
    geom = pu.geometry(spec)
    n_centres = [sp.santapp_kmeans_parent_count(n, spec.parent_size) for n in spec.prompt_len]
    k = sp.bf16_bits_to_cuda(data.k_prompt)
    centres, steps = sp.santapp_kmeans_fit(geom, spec.prompt_len, n_centres, k, **opts)
    torch.cuda.synchronize()
    keys = synth.bf16_to_f64(data.k_prompt[j, :spec.prompt_len[0]])
    want, want_steps = orc.minibatch_kmeans(keys, n_centres[0], stream=j)
    assert int(steps[j, 0]) == want_steps
    assert np.array_equal(centres[j, :n_centres[0]].cpu().numpy(), want.astype(np.float32))
    return n_centres


def test_fit_config_2_full_size_paper_settings():
    """32K keys per KV head, 64 centres, the paper's settings (minibatch 4096, 100 iterations,
    patience 10, ratio 0.01, seed 0): the configuration `bench.py --parents kmeans` prepares."""
    assert _one_pair_at_full_size(synth.spec_qwen_b1(), j=1) == [64]


def test_fit_many_centres_paper_parent_size():
    """Parents of nominal size 16 (the paper's operating point) on 8K keys: 512 centres, 8 trials per
    centre, the initialisation sample is the whole sequence."""
    assert _one_pair_at_full_size(synth.spec_paper_point(prompt=8192), j=3) == [512]


@pytest.mark.parametrize("case", range(16))
def test_fit_random_small_configurations(case):
    rng = np.random.default_rng(500 + case)
    n_seqs = int(rng.integers(1, 4))
    prompt = tuple(int(rng.integers(2, 1500)) for _ in range(n_seqs))
    spec = synth.spec_small_gqa(n_seqs=n_seqs, prompt=prompt, suffix0=(0,) * n_seqs)
    spec.n_clusters = int(rng.integers(2, 30))
    spec.seed = case
    spec.elem = "fp16" if case % 2 else "bf16"
    n_centres = [int(rng.integers(1, min(n, 40) + 1)) for n in prompt]
    _fit_both(spec, n_centres, batch_size=int(rng.choice([16, 100, 512, 4096])), max_iter=int(rng.choice([1, 3, 100])),
              patience=int(rng.choice([1, 3, 10])), reassignment_ratio=float(rng.choice([0.0, 0.01, 0.5])),
              seed=int(rng.integers(1 << 62)), stream_base=int(rng.integers(1 << 30)))


@pytest.mark.parametrize("n", [300, 12800, 17000])
def test_fit_with_a_centre_per_key_returns_the_keys(n):
    """k = N on distinct points: every greedy pick is a point that is no centre yet, every minibatch point is
    its own centre, and with an inertia of zero the fit stops after one step and `patience` more. The sizes
    take the start in one kernel, the start for samples beyond shared memory, and labels beyond 14 bits."""
    bits = (np.arange(n)[:, None] >> np.arange(15)) & 1
    rows = np.zeros((1, n, 128), dtype=np.float32)
    rows[0, :, :15] = 3.0 * bits - 1.0
    geom = sp.Geometry(1, 1, 1, 128, 16, 4)
    k = torch.from_numpy(rows).cuda().to(torch.bfloat16)
    centres, steps = sp.santapp_kmeans_fit(geom, [n], [n], k, reassignment_ratio=0.0, patience=3)
    torch.cuda.synchronize()
    assert int(steps[0, 0]) == 4
    got = centres[0].cpu().numpy()
    order = (((got[:, :15] + 1.0) / 3.0) @ (2.0 ** np.arange(15))).astype(np.int64)
    assert np.array_equal(np.sort(order), np.arange(n))
    assert np.array_equal(got, rows[0][order])


def _fit_keys_both(keys, elem, k, **opts):
    """A fit of one sequence's keys [n_kv][N][128] on the GPU and by the oracle, pair by pair."""
    bits = synth.round_bits(keys, elem)
    n_kv, N = keys.shape[:2]
    geom = sp.Geometry(1, n_kv, n_kv, 128, 16, 4, sp.SANTAPP_FP16 if elem == "fp16" else sp.SANTAPP_BF16)
    centres, steps = sp.santapp_kmeans_fit(geom, [N], [k], sp.bf16_bits_to_cuda(bits, dtype=geom.torch_dtype), **opts)
    torch.cuda.synchronize()
    o = {"batch": opts["batch_size"], "max_iter": opts["max_iter"], "patience": opts["patience"], "seed": opts["seed"]}
    for j in range(n_kv):
        want, want_steps = orc.minibatch_kmeans(synth.to_f64(bits[j], elem), k, stream=j, ratio=opts["reassignment_ratio"], **o)
        assert int(steps[j, 0]) == want_steps, f"steps of pair {j}"
        assert np.array_equal(centres[j].cpu().numpy(), want.astype(np.float32)), f"centres of pair {j}"


@pytest.mark.parametrize("n", [100, 1153, 8200])
def test_start_in_clusters_with_blocks_without_keys(n):
    """1, 10 and 65 blocks of the sums: 15 of 16, 3 of 8 (nine pairs) and 3 of 16 thread blocks own none and take part in the messages
    all the same."""
    pairs = 9 if n == 1153 else 1
    keys = np.random.default_rng(47).standard_normal((pairs, n, 128))
    _fit_keys_both(keys.astype(np.float32), "bf16", 60, batch_size=4096, max_iter=1, patience=1, seed=14, reassignment_ratio=0.0)


@pytest.mark.parametrize("elem,far", [("fp16", 6000.0), ("fp16", 60000.0), ("bf16", 1e20)])
def test_fit_with_outlier_keys_beyond_the_range_of_the_bounds(elem, far):
    """Two keys so long that the greedy start makes them centres and no product bounds their distances
    (squared norm beyond 4.2e9 for fp16, 1e37 for bf16): the minibatch steps of the ordinary keys are the oracle's."""
    rng = np.random.default_rng(17)
    keys = rng.standard_normal((2, 900, 128)).astype(np.float32)
    for j, rows in enumerate([(3, 600), (450, 899)]):
        keys[j, rows[0]] = far
        keys[j, rows[1]] = -far
    _fit_keys_both(keys, elem, 200, batch_size=256, max_iter=3, patience=4, seed=2, reassignment_ratio=0.0)


@pytest.mark.parametrize("k,n", [(5, 900), (20, 900), (54, 900), (7, 2100), (54, 2100)])
def test_start_with_few_trials_beside_rows_without_a_bound(k, n):
    """Three to five trials a centre and four keys of different magnitudes whose squared norms fp32 does not hold: such a row is
    marked for every trial and for no column of the products beyond them, and where all trials drew one of these
    rows, which outweigh the rest, the centre is that row. 2100 keys are 17 blocks of the sums: a cluster of 16 has blocks without any."""
    rng = np.random.default_rng(41)
    keys = rng.standard_normal((2, n, 128)).astype(np.float32)
    for j in range(2):
        for row, far in zip(rng.choice(n, 4, replace=False), (2e18, 3e19, 5e20, -4e21)):
            keys[j, row] *= far
    _fit_keys_both(keys, "bf16", k, batch_size=700, max_iter=2, patience=4, seed=3, reassignment_ratio=0.0)


@pytest.mark.parametrize("n", [129, 2100])
def test_start_in_which_most_warps_send_nothing(n):
    """Two and 17 blocks of the sums on clusters of 16: a thread block has sums on none to two of its warps and sends gains from
    two or three; the others are held by barriers alone. Thirty runs with the oracle's centres."""
    keys = np.random.default_rng(43).standard_normal((2, n, 128))
    bits = synth.round_bits(keys.astype(np.float32))
    geom, k = sp.Geometry(1, 2, 2, 128, 16, 4), sp.bf16_bits_to_cuda(bits)
    want = np.stack([orc.minibatch_kmeans(synth.to_f64(bits[j], "bf16"), 100, batch=700, max_iter=1, patience=4, seed=12, stream=j)[0] for j in range(2)])
    for _ in range(30):
        centres, _ = sp.santapp_kmeans_fit(geom, [n], [100], k, batch_size=700, max_iter=1, patience=4, seed=12)
        assert np.array_equal(centres.cpu().numpy(), want.astype(np.float32))


def test_fits_that_stop_beside_their_own_sorting_blocks():
    """The stopping rule of a step is settled beside the ordering of the next minibatch, in other blocks of one launch.
    192 fits that stop at many different steps, every step enqueued: ten runs, each with the oracle's step counts
    and the first run's centres."""
    rng = np.random.default_rng(21)
    B, kv, k = 96, 2, 5
    lens = [int(x) for x in rng.integers(40, 90, size=B)]
    bits = synth.round_bits(rng.standard_normal((kv, sum(lens), 128)).astype(np.float32))
    geom, keys = sp.Geometry(B, kv, kv, 128, 16, 4), sp.bf16_bits_to_cuda(bits)
    opts = dict(batch_size=16, max_iter=12, patience=2, seed=6, no_host_poll=True)
    off = np.concatenate([[0], np.cumsum(lens)])
    want = [[orc.minibatch_kmeans(synth.to_f64(bits[j, off[b]:off[b + 1]]), k, batch=16, max_iter=12, patience=2, seed=6, stream=b * kv + j)[1]
             for b in range(B)] for j in range(kv)]
    first = None
    for _ in range(10):
        centres, steps = sp.santapp_kmeans_fit(geom, lens, [k] * B, keys, **opts)
        assert steps.cpu().tolist() == want
        first = centres if first is None else first
        assert torch.equal(centres, first)
    assert len(set(np.ravel(want).tolist())) > 8


@pytest.mark.parametrize("scale", [1e-18, 1e-20, 1e-21, 1e-22])
def test_fit_of_keys_whose_products_underflow(scale):
    keys = scale * np.random.default_rng(23).standard_normal((4, 800, 128))
    _fit_keys_both(keys.astype(np.float32), "bf16", 40, batch_size=128, max_iter=2, patience=4, seed=5, reassignment_ratio=0.01)


@pytest.mark.parametrize("elem,n,spread,tiny", [("bf16", 1000, 0, 0.0), ("bf16", 129, 14, 0.0), ("bf16", 1000, 14, 0.0), ("bf16", 900, 3, 1e-39),
                                                ("fp16", 1000, 0, 0.0), ("fp16", 700, 9, 0.0), ("fp16", 900, 2, 1e-7)])
def test_start_on_values_of_many_magnitudes(elem, n, spread, tiny):
    """A distance whose terms are multiples of one power of two, of which it has fewer than 2^53, is summed in any order,
    another in the defining one: keys of which all, some and hardly any distances are of the first kind, zeros
    and subnormal values among them."""
    rng = np.random.default_rng(29)
    keys = rng.standard_normal((2, n, 128)) * 2.0 ** -rng.integers(0, spread + 1, size=(2, n, 128))
    rows = rng.random((2, n)) < 0.5
    keys[rows] = np.where(rng.random((int(rows.sum()), 128)) < 0.05, tiny * rng.integers(-3, 4, size=(int(rows.sum()), 128)), keys[rows])
    _fit_keys_both(keys.astype(np.float32), elem, min(150, n // 2), batch_size=128, max_iter=1, patience=4, seed=4, reassignment_ratio=0.0)


@pytest.mark.parametrize("n", [8103, 8104, 12288])
def test_start_with_ten_and_eleven_trials_a_centre(n):
    """2 + floor(ln k) is 11 from k = 8104 on; samples of up to 12288 keys take the start in one kernel all the same."""
    test_fit_with_a_centre_per_key_returns_the_keys(n)


def test_start_with_eleven_trials_rows_without_a_bound_and_blocks_without_keys():
    """k = N = 8200: eleven trials, 65 blocks of the sums on a cluster of 16, three of whose blocks own none, and five keys
    whose squared norms fp32 does not hold. All keys differ, so every one becomes a centre."""
    n = 8200
    bits = (np.arange(n)[:, None] >> np.arange(15)) & 1
    rows = np.zeros((1, n, 128), dtype=np.float32)
    rows[0, :, :15] = 3.0 * bits - 1.0
    rows[0, [7, 1000, 4099, 8063, 8199]] *= np.float32([[2.0 ** 61], [2.0 ** 64], [-2.0 ** 66], [2.0 ** 70], [-2.0 ** 75]])
    geom = sp.Geometry(1, 1, 1, 128, 16, 4)
    k = torch.from_numpy(rows).cuda().to(torch.bfloat16)
    centres, steps = sp.santapp_kmeans_fit(geom, [n], [n], k, batch_size=256, reassignment_ratio=0.0, patience=3)
    torch.cuda.synchronize()
    assert int(steps[0, 0]) == 4
    assert np.array_equal(np.unique(centres[0].cpu().numpy(), axis=0), np.unique(rows[0], axis=0))


@pytest.mark.parametrize("batch,k", [(1, 2), (63, 7), (64, 8), (65, 9), (128, 16), (129, 16), (129, 17)])
def test_steps_at_the_edges_of_their_blocks_and_of_the_update_rule(batch, k):
    """64 points a block of the resolving kernel; fewer or more than eight points a centre in the update."""
    keys = np.random.default_rng(37).standard_normal((2, 400, 128))
    _fit_keys_both(keys.astype(np.float32), "bf16", k, batch_size=batch, max_iter=2, patience=30, seed=8, reassignment_ratio=0.01)


@pytest.mark.parametrize("kind", ["few", "same", "padded", "some", "integer"])
def test_fit_of_keys_that_repeat(kind):
    from test_gpu_parents import _repeated
    rng = np.random.default_rng(31)
    keys = np.stack([_repeated(kind, 1000, rng) for _ in range(2)])
    _fit_keys_both(keys.astype(np.float32), "bf16", 150, batch_size=256, max_iter=4, patience=5, seed=9, reassignment_ratio=0.3)
