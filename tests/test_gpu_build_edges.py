"""Contiguous records where the fp32 distances decide little or sit at the edges of their tiles: parents of
every kernel's smallest, largest and odd sizes, one team per key, keys repeated many times, keys whose squares
leave the range of fp32, and one key far larger than the rest; against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import santapp_oracle as orc
from paper_2609_35629_b200 import binding as sp
from paper_2609_35629_b200 import synth

pytestmark = pytest.mark.gpu


def _keys(kind, n, d, rng):
    x = rng.standard_normal((n, d)).astype(np.float32)
    if kind == "same":
        x[:] = x[:1]
    elif kind == "repeated":                     # few distinct rows: most distances are exactly zero or exactly tied
        x = x[rng.integers(0, 5, size=n)]
    elif kind == "zero":
        x[:] = 0.0
    elif kind == "huge":                         # squares overflow fp32 (fp64 decides)
        x *= np.float32(1e25)
    elif kind == "tiny":                         # squares underflow fp32
        x *= np.float32(1e-25)
    elif kind == "outlier":                      # one row a thousand times longer: its error bound dwarfs the others'
        x[n // 2] *= np.float32(1000.0)
    elif kind == "offset":                       # a common component much longer than the differences
        x += np.float32(30.0)
    elif kind == "integer":                      # exact ties at many distances
        x = rng.integers(-1, 2, size=(n, d)).astype(np.float32)
    return x


CASES = [(p, r) for p, r in [(1, 1), (5, 1), (8, 2), (16, 4), (16, 16), (17, 17), (24, 8), (32, 32), (33, 11), (64, 8), (65, 13),
                             (128, 8), (129, 43), (256, 16), (258, 258), (512, 32), (512, 512), (512, 1)]]


@pytest.mark.parametrize("P,R", CASES)
@pytest.mark.parametrize("kind,elem", [("plain", "bf16"), ("plain", "fp16"), ("repeated", "bf16"), ("integer", "fp16"),
                                       ("outlier", "bf16"), ("offset", "bf16")])
def test_records_at_every_parent_size(P, R, kind, elem):
    _check(P, R, kind, elem)


@pytest.mark.parametrize("P,R", [(16, 4), (32, 8), (64, 8), (512, 32)])
@pytest.mark.parametrize("kind", ["zero", "huge", "tiny"])
def test_records_outside_the_range_of_fp32_squares(P, R, kind):
    _check(P, R, kind, "bf16")


def _check(P, R, kind, elem):
    rng = np.random.default_rng([P, R, len(kind)])
    lens, kv = [2 * P + P // 2 + 1, P, max(1, P - 1)], 2
    n = sum(lens)
    k_bits = synth.round_bits(np.stack([_keys(kind, n, 128, rng) for _ in range(kv)]), elem)
    v_bits = synth.round_bits(rng.standard_normal((kv, n, 128)).astype(np.float32), elem)
    geom = sp.Geometry(len(lens), 2 * kv, kv, 128, P, R, sp.SANTAPP_FP16 if elem == "fp16" else sp.SANTAPP_BF16)
    t = sp.santapp_build_teams(geom, lens, sp.bf16_bits_to_cuda(k_bits, dtype=geom.torch_dtype), sp.bf16_bits_to_cuda(v_bits, dtype=geom.torch_dtype))
    torch.cuda.synchronize()
    csr, token = t.team_row_start.cpu().numpy(), t.row_token.cpu().numpy()
    kp, vp, rep = (x.view(torch.int16).cpu().numpy().view(np.uint16) for x in (t.k_packed, t.v_packed, t.rep_keys))
    toff, amax = t.seq_team_off.cpu().numpy(), t.rep_abs_max.cpu().numpy()
    off = np.concatenate([[0], np.cumsum(lens)])
    for j in range(kv):
        for b, N in enumerate(lens):
            rows = slice(off[b], off[b + 1])
            ts, tm, reps = orc.build_teams_contiguous(synth.to_f64(k_bits[j, rows], elem), P, R)
            t0, t1 = int(toff[b]), int(toff[b + 1])
            assert t.team_count[j, b].item() == t1 - t0 == len(reps)
            assert np.array_equal(csr[j, t0 + b:t1 + b + 1], ts)
            assert np.array_equal(token[j, rows], tm)
            assert np.array_equal(rep[j, t0:t1], k_bits[j, rows][reps])
            assert np.array_equal(kp[j, rows], k_bits[j, rows][tm]) and np.array_equal(vp[j, rows], v_bits[j, rows][tm])
            assert amax[j, b] == np.abs(synth.to_f32(k_bits[j, rows][reps], elem)).max()


@pytest.mark.parametrize("P,R", [(1, 1), (8, 2), (16, 4), (17, 17), (32, 8), (32, 32)])
@pytest.mark.parametrize("kind", ["plain", "repeated", "integer", "outlier", "huge", "zero"])
def test_shared_latent_records_at_every_parent_size(P, R, kind):
    rng = np.random.default_rng([P, R, len(kind), 1])
    lens = [3 * P + P // 2 + 1, P, max(1, P - 1)]
    off = np.concatenate([[0], np.cumsum(lens)])
    bits = synth.round_bits(_keys(kind, sum(lens), sp.LATENT_ROW, rng))
    t = sp.santapp_latent_build_teams(sp.LatentGeometry(len(lens), 16, P, R), lens, sp.bf16_bits_to_cuda(bits))
    torch.cuda.synchronize()
    csr, token, toff = t.team_row_start.cpu().numpy(), t.row_token.cpu().numpy(), t.seq_team_off.cpu().numpy()
    packed, rep = (x.view(torch.int16).cpu().numpy().view(np.uint16) for x in (t.rows_packed, t.rep_rows))
    for b in range(len(lens)):
        rows = bits[off[b]:off[b + 1]]
        ts, tm, reps = orc.shared_latent_records(synth.to_f64(rows), sp.LATENT_DIM, P, R)
        t0, t1 = int(toff[b]), int(toff[b + 1])
        assert np.array_equal(csr[t0 + b:t1 + b + 1], ts) and np.array_equal(token[off[b]:off[b + 1]], tm)
        assert np.array_equal(synth.to_f64(rep[t0:t1]), reps) and np.array_equal(packed[off[b]:off[b + 1]], rows[tm])
        assert t.rep_abs_max[b].item() == np.abs(synth.to_f32(rep[t0:t1])).max()


@pytest.mark.parametrize("P,R", [(16, 4), (32, 8), (64, 16), (128, 16), (256, 16), (512, 32)])
@pytest.mark.parametrize("scale", [1e-21, 1e-22, 3e-23])
def test_records_of_parents_with_one_ordinary_row_among_rows_whose_products_underflow(P, R, scale):
    """One row of every parent is of ordinary length, so that fp32 distances are used, and the products of the others are
    subnormal in fp32: their distances are decided by the fp64 sums."""
    rng = np.random.default_rng([P, R, int(1 / scale) & 0xFFFF])
    lens, kv = [4 * P], 2
    x = (scale * rng.standard_normal((kv, lens[0], 128))).astype(np.float32)
    x[:, P // 3::P] = rng.standard_normal((kv, 4, 128))
    k_bits = synth.round_bits(x)
    geom = sp.Geometry(1, kv, kv, 128, P, R)
    k = sp.bf16_bits_to_cuda(k_bits)
    t = sp.santapp_build_teams(geom, lens, k, k)
    csr, token = t.team_row_start.cpu().numpy(), t.row_token.cpu().numpy()
    for j in range(kv):
        ts, tm, _ = orc.build_teams_contiguous(synth.to_f64(k_bits[j]), P, R)
        assert np.array_equal(csr[j, :len(ts)], ts) and np.array_equal(token[j], tm)


@pytest.mark.parametrize("P,R", [(64, 8), (64, 32), (128, 64), (512, 256)])
@pytest.mark.parametrize("kind", ["same", "repeated", "integer"])
def test_records_of_rows_that_tie_at_many_choices(P, R, kind):
    """Distances known in fp64 are kept from choice to choice, and an open row is settled once."""
    _check(P, R, kind, "bf16")


@pytest.mark.parametrize("P,R", [(64, 8), (64, 32)])
def test_records_of_one_repeated_row_cost_little_more_than_others(P, R):
    """Every choice is a tie of all rows: 1.5 to 2 times the usual call; 22 and 61 times when 64 open rows, however
    many representatives they were compared with, were not enough to give up."""
    g = torch.Generator(device="cuda").manual_seed(5)
    geom, N = sp.Geometry(1, 4, 4, 128, P, R), 32768
    rows = torch.randn(4, N, 128, generator=g, device="cuda").to(torch.bfloat16)

    def microseconds(k):
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sp.santapp_build_teams(geom, [N], k, rows)
            b.record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
        return best

    assert microseconds(rows[:, :1].repeat(1, N, 1)) < 6 * microseconds(rows)


@pytest.mark.parametrize("P,R", [(8, 2), (16, 4), (17, 17), (32, 8), (32, 32)])
@pytest.mark.parametrize("kind", ["same", "repeated", "integer"])
def test_records_of_small_parents_whose_rows_tie(P, R, kind):
    _check(P, R, kind, "fp16")
    test_shared_latent_records_at_every_parent_size(P, R, kind)


def test_shared_latent_records_of_zero_rows_cost_a_few_times_the_usual():
    """About 3 times at 32 rows and 8 representatives (every comparison in fp64 once), 10 when each was made up to three
    times."""
    g = torch.Generator(device="cuda").manual_seed(6)
    geom, N = sp.LatentGeometry(1, 16, 32, 8), 1 << 18
    rows = torch.randn(N, sp.LATENT_ROW, generator=g, device="cuda").to(torch.bfloat16)

    def microseconds(x):
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sp.santapp_latent_build_teams(geom, [N], x)
            b.record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
        return best

    assert microseconds(torch.zeros_like(rows)) < 5.5 * microseconds(rows)


@pytest.mark.parametrize("kind", ["contiguous", "parents", "latent"])
def test_preparation_calls_can_be_captured_in_a_cuda_graph(kind):
    """The tables made from host arrays travel inside kernel arguments: a captured call, replayed on other keys after its
    host arrays are gone, leaves the records of a plain call on them."""
    g = torch.Generator(device="cuda").manual_seed(8)
    lens = [700, 333]
    first, second = (torch.randn(2, sum(lens), 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    k = first.clone()
    rows = torch.randn(sum(lens), sp.LATENT_ROW, generator=g, device="cuda").to(torch.bfloat16)
    cen = torch.randn(2, 30, 128, generator=g, device="cuda")
    geom = sp.Geometry(2, 4, 2, 128, 64, 8)

    def call():
        if kind == "contiguous":
            t = sp.santapp_build_teams(geom, list(lens), k, k)
        elif kind == "parents":
            t = sp.santapp_build_teams_parents(geom, list(lens), [20, 10], k, k, sp.santapp_assign_parents(geom, list(lens), [20, 10], k, cen))
        else:
            t = sp.santapp_latent_build_teams(sp.LatentGeometry(2, 16, 16, 4), list(lens), rows)
            return t, [t.rows_packed, t.rep_rows, t.team_row_start, t.row_token, t.seq_row_off, t.seq_team_off, t.rep_abs_max]
        return t, [t.k_packed, t.rep_keys, t.team_row_start, t.row_token, t.seq_row_off, t.seq_team_off, t.rep_abs_max, t.team_count]

    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        kept, got = call()
    for other in (second, first):
        k.copy_(other)
        rows.mul_(-0.5)
        graph.replay()
        want = call()[1]
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
