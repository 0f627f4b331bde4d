"""Performance cases of the library: what a decode loop and its preparation ask of it.

A case is a dict of plain values with a `kind`:

  token         one generated token through `layers` layers: santapp_decode_attn per layer
  dense         the same token with full attention: santapp_dense_decode_attn per layer
  build         the records of one layer after prefill, contiguous parents: santapp_build_teams
  kmeans        the same with k-means parents: santapp_kmeans_fit, santapp_assign_parents,
                santapp_build_teams_parents
  latent_token, latent_dense, latent_build   the three operations on shared-latent rows

Inputs follow the recipe of `paper_2609_35629_b200.synth`, drawn on the GPU: rows scattered around
cluster centres (sigma 0.3), clusters drawn row by row ("iid") or in runs of neighbouring rows ("runs"),
four sink rows per sequence scaled by 4, queries that are noisy copies of prompt rows. Output buffers and
workspaces of the per-token calls are kept by the caller, as a serving loop does; the builders make
their own.
"""
import math
import random

import torch

from paper_2609_35629_b200 import binding as sp

D = 128                                    # head_dim of the K/V path
ROW = sp.LATENT_ROW                        # values of a shared-latent row
LATENT_SCALE = 1.0 / math.sqrt(192.0)      # 128 content + 64 rotary query values before absorption


def _token(name, n_seqs, lo, hi, layers, q_heads, kv_heads, parent, reps, sample, suffix_lo, suffix_cap, elem, layout,
           clusters, kind="token"):
    return dict(name=name, kind=kind, n_seqs=n_seqs, lo=lo, hi=hi, layers=layers, q_heads=q_heads, kv_heads=kv_heads,
                parent=parent, reps=reps, sample=sample, suffix_lo=suffix_lo, suffix_cap=suffix_cap, elem=elem,
                layout=layout, clusters=clusters, shape_seed=0)


def _latent(name, kind, n_seqs, lo, hi, heads, parent, reps, sample, suffix_lo, suffix_cap):
    return dict(name=name, kind=kind, n_seqs=n_seqs, lo=lo, hi=hi, heads=heads, parent=parent, reps=reps, sample=sample,
                suffix_lo=suffix_lo, suffix_cap=suffix_cap, layout="iid", clusters=512, shape_seed=0)


def listed():
    return [
        # The smallest call: one layer of a one-head model with 4096 keys. Launches and host time.
        _token("tiny_4k", 1, 4096, 4096, 1, 1, 1, 256, 16, 16, 16, 16, "bf16", "iid", 64),
        # A single user's token at 32K through all 28 layers: the benchmark's default step.
        _token("token_b1_32k", 1, 32768, 32768, 28, 28, 4, 512, 32, 32, 128, 256, "bf16", "iid", 2048),
        # The same token at the paper's operating point: small teams, fp16, no suffix yet.
        _token("token_b1_32k_fine_fp16", 1, 32768, 32768, 28, 28, 4, 16, 4, 31, 0, 16, "fp16", "runs", 2048),
        # A small serving batch of long chats with a generous budget.
        _token("token_b8_32k", 8, 32768, 32768, 1, 28, 4, 512, 32, 64, 0, 16, "bf16", "iid", 2048),
        # A full serving batch: prompts of every (odd) length, suffixes of every length.
        _token("token_b32_ragged", 32, 8192, 65536, 1, 28, 4, 512, 32, 31, 1, 1024, "bf16", "iid", 2048),
        # Long documents, where sampling saves most.
        _token("token_b4_128k", 4, 131072, 131072, 1, 28, 4, 512, 32, 32, 0, 16, "bf16", "runs", 2048),
        # Full attention over the same records: the layers that a model keeps dense.
        _token("dense_b1_32k", 1, 32768, 32768, 28, 28, 4, 512, 32, 32, 128, 256, "bf16", "iid", 2048, kind="dense"),
        # After prefill: one layer's records on contiguous parents.
        _token("build_32k", 1, 32768, 32768, 1, 28, 4, 512, 32, 32, 0, 16, "bf16", "iid", 2048, kind="build"),
        # After prefill with k-means parents at the paper's settings (2048 centres per KV head).
        _token("kmeans_32k", 1, 32768, 32768, 1, 28, 4, 16, 4, 31, 0, 16, "bf16", "iid", 2048, kind="kmeans"),
        # Rows shared by 16 heads, 32 sequences of 8K: a sampled token, a dense token, the records.
        _latent("latent_token_b32_8k", "latent_token", 32, 8192, 8192, 16, 16, 4, 128, 8, 16),
        _latent("latent_dense_b32_8k", "latent_dense", 32, 8192, 8192, 16, 16, 4, 128, 8, 16),
        _latent("latent_build_b32_8k", "latent_build", 32, 8192, 8192, 16, 16, 4, 128, 8, 16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same calls at other sizes, head layouts, team shapes, budgets and types."""
    kind = rng.choice(["token"] * 5 + ["dense", "build", "kmeans", "latent_token", "latent_token", "latent_dense",
                                       "latent_build"])
    shape_seed = rng.randrange(1 << 20)
    layout = rng.choice(["iid", "runs"])
    if kind.startswith("latent"):
        n_seqs = _log_int(rng, 1, 32)
        hi = _log_int(rng, 512, 8192)
        parent, reps = rng.choice([(16, 4), (16, 4), (32, 8), (8, 2)])
        cap = rng.choice([0, 16, 64])
        return dict(kind=kind, n_seqs=n_seqs, lo=rng.choice([hi, max(256, hi // 4)]), hi=hi, heads=rng.choice([16, 16, 12, 8]),
                    parent=parent, reps=reps, sample=rng.choice([32, 64, 128, 256, _log_int(rng, 16, 256)]),
                    suffix_lo=rng.randint(0, cap), suffix_cap=cap, layout=layout, clusters=512, shape_seed=shape_seed)
    q_heads, kv_heads = rng.choice([(28, 4), (28, 4), (32, 8), (16, 2), (12, 4), (8, 8)])
    elem = rng.choice(["bf16", "bf16", "fp16"])
    if kind == "kmeans":
        n_seqs, kv_heads, q_heads = 1, 4, 28
        hi = _log_int(rng, 2048, 32000)
        parent, reps = rng.choice([(16, 4), (32, 4), (64, 8), (128, 8), (256, 16), (512, 32)])
        lo, layers = hi, 1
    else:
        n_seqs = _log_int(rng, 1, 32)
        most = min(131072, (1 << 20) // n_seqs)
        hi = _log_int(rng, 1024, most)
        lo = rng.choice([hi, max(512, hi // 8)])
        parent, reps = rng.choice([(512, 32), (512, 32), (256, 16), (128, 8), (64, 8), (16, 4)])
        layers = max(1, min(rng.choice([1, 4, 28]), (1 << 20) // (hi * n_seqs)))
        if kind == "build":
            layers = 1
    cap = rng.choice([0, 16, 256, 1024])
    group = q_heads // kv_heads
    sample = min(rng.choice([16, 31, 32, 64, _log_int(rng, 8, 128)]), 1024 // group)
    return dict(kind=kind, n_seqs=n_seqs, lo=lo, hi=hi, layers=layers, q_heads=q_heads, kv_heads=kv_heads, parent=parent,
                reps=reps, sample=sample, suffix_lo=rng.randint(0, cap), suffix_cap=cap, elem=elem, layout=layout,
                clusters=2048, shape_seed=shape_seed)


# ---- shapes ----------------------------------------------------------------------------------------
def _prompt_len(case):
    rng = random.Random(case["shape_seed"])
    return [rng.randint(case["lo"], case["hi"]) for _ in range(case["n_seqs"])]


def _suffix_len(case):
    rng = random.Random(case["shape_seed"] + 1)
    if case["lo"] == case["hi"]:
        return [case["suffix_lo"]] * case["n_seqs"]
    return [rng.randint(case["suffix_lo"], case["suffix_cap"]) for _ in range(case["n_seqs"])]


def _n_teams(case, n):
    full, rest = divmod(n, case["parent"])
    return full * case["reps"] + min(rest, case["reps"])


# ---- inputs ----------------------------------------------------------------------------------------
def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda")


def _clustered(gen, centres, n, layout, mean_run):
    k = centres.shape[0]
    if layout == "runs":
        new_run = torch.rand(n, generator=gen, device="cuda") * mean_run < 1.0
        ids = torch.randint(k, (n,), generator=gen, device="cuda")
        which = ids[torch.cumsum(new_run, 0).clamp_(max=n - 1)]
    else:
        which = torch.randint(k, (n,), generator=gen, device="cuda")
    return centres[which] + 0.3 * _normal(gen, n, centres.shape[1])


def _sinks(x, offsets):
    for o in offsets:
        x[o:o + 4] *= 4.0


def _kv_layer(case, gen, dtype, lens, offsets):
    """K and V of one layer's prompts, the suffix rows, and one query per head."""
    n, kv, cap = sum(lens), case["kv_heads"], case["suffix_cap"]
    n_seqs, group = case["n_seqs"], case["q_heads"] // case["kv_heads"]
    k = torch.empty(kv, n, D, dtype=dtype, device="cuda")
    v = torch.empty_like(k)
    k_suffix = torch.empty(n_seqs, kv, cap, D, dtype=dtype, device="cuda")
    v_suffix = torch.empty_like(k_suffix)
    q = torch.empty(n_seqs, kv, group, D, dtype=dtype, device="cuda")
    first = torch.tensor(offsets, device="cuda").view(-1, 1)
    length = torch.tensor(lens, device="cuda").view(-1, 1)
    for j in range(kv):
        centres = _normal(gen, case["clusters"], D)
        x = _clustered(gen, centres, n, case["layout"], max(1.0, case["hi"] / case["clusters"]))
        _sinks(x, offsets)
        k[j] = x
        v[j] = _normal(gen, n, D)
        rows = first + (torch.rand(n_seqs, group, generator=gen, device="cuda") * length).long()
        q[:, j] = 2.0 * (k[j][rows].float() + 0.5 * _normal(gen, n_seqs, group, D))
        if cap:
            k_suffix[:, j] = _clustered(gen, centres, n_seqs * cap, "iid", 1.0).view(n_seqs, cap, D)
            v_suffix[:, j] = _normal(gen, n_seqs, cap, D)
    return k, v, k_suffix, v_suffix, q.view(n_seqs, case["q_heads"], D)


def _latent_layer(case, gen, lens, offsets):
    n, cap, n_seqs, heads = sum(lens), case["suffix_cap"], case["n_seqs"], case["heads"]
    centres = _normal(gen, case["clusters"], sp.LATENT_DIM)

    def some(m, layout):
        x = torch.empty(m, ROW, device="cuda")
        x[:, :sp.LATENT_DIM] = _clustered(gen, centres, m, layout, max(1.0, case["hi"] / case["clusters"]))
        x[:, sp.LATENT_DIM:] = _normal(gen, m, sp.LATENT_ROPE_DIM)
        return x

    x = some(n, case["layout"])
    _sinks(x, offsets)
    rows = x.to(torch.bfloat16)
    suffix = some(n_seqs * cap, "iid").to(torch.bfloat16).view(n_seqs, cap, ROW) if cap else None
    first = torch.tensor(offsets, device="cuda").view(-1, 1)
    length = torch.tensor(lens, device="cuda").view(-1, 1)
    picked = first + (torch.rand(n_seqs, heads, generator=gen, device="cuda") * length).long()
    q = 0.55 * (rows[picked].float() + 0.5 * _normal(gen, n_seqs, heads, ROW))
    return rows, suffix, q.to(torch.bfloat16)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    lens = _prompt_len(case)
    offsets = [sum(lens[:b]) for b in range(len(lens))]
    state = dict(kind=case["kind"], lens=lens, sample=case["sample"], seed=seed, step=seed % 977)
    suffix_len = torch.tensor(_suffix_len(case), dtype=torch.int32, device="cuda")
    if case["kind"].startswith("latent"):
        geom = sp.LatentGeometry(case["n_seqs"], case["heads"], case["parent"], case["reps"])
        rows, suffix, q = _latent_layer(case, gen, lens, offsets)
        state.update(geom=geom, rows=rows)
        if case["kind"] != "latent_build":
            teams = sp.santapp_latent_build_teams(geom, lens, rows)
            n = (sp.santapp_latent_dense_workspace_bytes(geom, teams) if case["kind"] == "latent_dense" else
                 sp.santapp_latent_decode_workspace_bytes(geom, teams, case["sample"], case["suffix_cap"]))
            state.update(teams=teams, q=q, suffix=suffix, suffix_len=suffix_len,
                         out=torch.empty(case["n_seqs"], case["heads"], sp.LATENT_DIM, device="cuda"),
                         workspace=torch.empty(n, dtype=torch.uint8, device="cuda"))
            del state["rows"]
        return state
    geom = sp.Geometry(case["n_seqs"], case["q_heads"], case["kv_heads"], D, case["parent"], case["reps"],
                       sp.SANTAPP_FP16 if case["elem"] == "fp16" else sp.SANTAPP_BF16)
    state.update(geom=geom, layers=[], suffix_len=suffix_len)
    if case["kind"] == "kmeans":
        state["n_centres"] = [sp.santapp_kmeans_parent_count(n, case["parent"]) for n in lens]
    for _ in range(case["layers"]):
        k, v, k_suffix, v_suffix, q = _kv_layer(case, gen, geom.torch_dtype, lens, offsets)
        if case["kind"] in ("build", "kmeans"):
            state.update(k=k, v=v)
            return state
        teams = sp.santapp_build_teams(geom, lens, k, v)
        if "workspace" not in state:      # the layers follow one another on one stream: one workspace serves them all
            n = (sp.santapp_dense_workspace_bytes(geom, teams) if case["kind"] == "dense" else
                 sp.santapp_decode_workspace_bytes(geom, teams, case["sample"]))
            state["workspace"] = torch.empty(n, dtype=torch.uint8, device="cuda")
        if not case["suffix_cap"]:
            k_suffix = v_suffix = None
        out = torch.empty(case["n_seqs"], case["q_heads"], D, device="cuda")
        state["layers"].append((teams, q, k_suffix, v_suffix, out))
    return state


# ---- one pass --------------------------------------------------------------------------------------
def _records(t):
    return [t.k_packed, t.v_packed, t.rep_keys, t.team_row_start, t.row_token, t.seq_row_off, t.seq_team_off,
            t.rep_abs_max, t.team_count]


def run(state):
    kind, geom = state["kind"], state["geom"]
    if kind == "token":
        n = geom.n_seqs
        for i, (teams, q, k_suffix, v_suffix, out) in enumerate(state["layers"]):
            sp.santapp_decode_attn(geom, teams, q, k_suffix, v_suffix, state["suffix_len"], state["sample"], state["seed"],
                                   state["step"], stream_base=i * n, out=out, workspace=state["workspace"])
        return [layer[4] for layer in state["layers"]]
    if kind == "dense":
        for teams, q, k_suffix, v_suffix, out in state["layers"]:
            sp.santapp_dense_decode_attn(geom, teams, q, k_suffix, v_suffix, state["suffix_len"], out=out,
                                         workspace=state["workspace"])
        return [layer[4] for layer in state["layers"]]
    if kind == "build":
        return _records(sp.santapp_build_teams(geom, state["lens"], state["k"], state["v"]))
    if kind == "kmeans":
        lens, n_centres, k = state["lens"], state["n_centres"], state["k"]
        centres, steps = sp.santapp_kmeans_fit(geom, lens, n_centres, k)
        parent_of = sp.santapp_assign_parents(geom, lens, n_centres, k, centres)
        return [centres, steps, parent_of] + _records(
            sp.santapp_build_teams_parents(geom, lens, n_centres, k, state["v"], parent_of))
    if kind == "latent_token":
        return sp.santapp_latent_decode_attn(geom, state["teams"], state["q"], state["suffix"], state["suffix_len"],
                                             state["sample"], state["seed"], state["step"], LATENT_SCALE,
                                             out=state["out"], workspace=state["workspace"])
    if kind == "latent_dense":
        return sp.santapp_latent_dense_decode_attn(geom, state["teams"], state["q"], state["suffix"], state["suffix_len"],
                                                   LATENT_SCALE, out=state["out"], workspace=state["workspace"])
    t = sp.santapp_latent_build_teams(geom, state["lens"], state["rows"])
    return [t.rows_packed, t.rep_rows, t.team_row_start, t.row_token, t.seq_row_off, t.seq_team_off, t.rep_abs_max]


def work(case):
    """Bytes and operations of one pass. The rows a sampled token reads depend on the draw: counted are
    the rows of the expected number of distinct teams of equal size (larger teams are drawn more often,
    so the true figure is higher)."""
    kind, lens = case["kind"], _prompt_len(case)
    latent = kind.startswith("latent")
    width = ROW if latent else D
    per_row = 2 * ROW if latent else 4 * D           # stored bytes of a token's row
    heads = case["heads"] if latent else case["q_heads"]
    kv = 1 if latent else case["kv_heads"]
    group = heads // kv
    n_bytes = flops = 0
    if kind.endswith("token") or kind.endswith("dense"):
        values = sp.LATENT_DIM if latent else D
        for n, t in zip(lens, _suffix_len(case)):
            rows, m = n, _n_teams(case, n)
            if kind.endswith("token"):
                n_bytes += kv * (m * width * 2 + (m + 1) * 4)
                flops += 2 * heads * m * width
                rows = n * (1.0 - (1.0 - min(case["sample"], m) / m) ** group)
            n_bytes += kv * (rows + t) * per_row + heads * (2 * width + 4 * values)
            flops += 2 * heads * (rows + t) * (width + values)
        layers = 1 if latent else case["layers"]
        return {"bytes": layers * n_bytes, "flops": layers * flops}
    # records: rows in and out, representatives, CSR and token tables; a distance is 3 operations per value
    dims = sp.LATENT_DIM if latent else D
    for n in lens:
        m = _n_teams(case, n)
        n_bytes += kv * (2 * n * per_row + 2 * width * m + 4 * (m + n))
        flops += kv * 3 * dims * n * case["reps"]
        if kind == "kmeans":
            k = max(2, n // case["parent"])
            first = min(n, max(3 * 4096, 3 * k))     # the initialisation sample
            trials = 2 + int(math.log(k))
            flops += kv * 3 * dims * k * (n + first * trials + 10 * 4096)
            n_bytes += kv * (n * dims * 2 + 4 * n + k * dims * 4)
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    """Records, labels and centres follow from fp64 arithmetic in a fixed order: the same values
    everywhere. Attention outputs are fp32 sums over exact 16-bit inputs, whose logits reach a few
    tens (2^-24 of that is what a weight may be off by), with the weights carried to 16 bits or more."""
    if case["kind"] in ("build", "kmeans", "latent_build"):
        return "exact"
    return {"rel": 2e-5}
