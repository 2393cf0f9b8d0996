"""The work that users of this library have it do, as cases that can be timed.

A case names a transformer's cached attention (layers, images, heads, data type), the token-map schedule of an image as text
("1x1,2x2,..": height x width of every scale) and how the library is driven:

  kind "step"    one scalekv_step per layer and scale: append, attend, compress with the paper's rule
       "rule"    one scalekv_step_ex per layer and scale, with the selection options that `rule` names
       "calls"   scalekv_append, scalekv_attend and scalekv_compress(_ex) one by one, as an engine does that computes
                 something between them
       "stats"   the offline calibration: a full cache, scalekv_layer_stats_ex per layer and scale

  rule "paper"   window = the 16 patch centroids of the map, importance per head
       "snapkv"  window = the last 16 rows of the map, importance pooled over 7 keys
       "sinks"   positional: 4 attention sinks and the most recent entries
       "shared"  the paper's window, one importance for all heads of an image

Budgets are fractions of the tokens that are ever cached: `drafter` for every fourth layer, `refiner` for the others.  `graph`:
the pass is captured into a CUDA graph when the buffers are set up and replayed.  `lse`: the log-sum-exp of every row too.
"""
import numpy as np
import torch

from paper_2505_19602_b200 import binding, synth

WINDOW = 16
TOPK_PRIME = 16
DISTINCT = 8          # layers with inputs of their own; layer l takes those of layer l mod DISTINCT


def _text(sides):
    return ",".join(f"{h}x{w}" for h, w in sides)


def _square(sides):
    return _text([(s, s) for s in sides])


def _sides(case):
    return [tuple(int(x) for x in s.split("x")) for s in case["sides"].split(",")]


def _case(name, kind, sides, layers, batch, heads, drafter=0.30, refiner=0.03, dtype="bf16", rule="paper", graph=False, page=0,
          lse=False):
    return {"name": name, "kind": kind, "sides": sides, "layers": layers, "batch": batch, "heads": heads, "drafter": drafter,
            "refiner": refiner, "dtype": dtype, "rule": rule, "graph": graph, "page": page, "lse": lse}


def listed():
    s13, s16, s19 = synth.SIDES_13, synth.SIDES_16, synth.SIDES_19
    return [
        # one small image (up to 16 x 16 tokens) through a few layers: nothing but call, launch and kernel latency
        _case("small_image", "step", _square(s13[:7]), 4, 1, 16),
        # one user, one 1024 x 1024 image, all 32 layers, called layer by layer
        _case("one_image", "step", _square(s13), 32, 1, 16),
        # the same image from an engine that replays its captured pass: what the GPU alone takes for one user
        _case("one_image_graph", "step", _square(s13), 32, 1, 16, graph=True),
        # the headline: a batch of 8 images, 32 layers, 13 scales
        _case("batch_8", "step", _square(s13), 32, 8, 16, graph=True),
        # one layer of it at a uniform budget: every step waits for the compress of the scale before
        _case("one_layer", "step", _square(s13), 1, 8, 16, 0.10, 0.10, lse=True),
        # a larger model: 32 heads, 8 images, four of its layers
        _case("wide_model", "step", _square(s13), 4, 8, 32, graph=True),
        # 2048 x 2048 images: 16 scales, 4 images, four layers at 10 % overall
        _case("hires", "step", _square(s16), 4, 4, 16, 0.30770, 0.03077),
        # a 4K-class image: 19 scales, a drafter and a refiner layer
        _case("uhd", "step", _square(s19), 2, 1, 16, 0.30770, 0.03077),
        # rectangular maps of odd sizes, the SnapKV-like rule at a uniform budget, small pages
        _case("snapkv_wide_format", "rule", "1x1,2x3,3x5,5x8,7x12,10x17,14x24,19x33,25x44,33x57,43x75", 8, 2, 16, 0.10, 0.10,
              rule="snapkv", page=32),
        # sinks and recent entries through the three calls, tall maps
        _case("sinks_tall_format", "calls", "1x1,3x2,5x3,8x5,13x8,19x12,27x17,37x23,50x31,67x42", 6, 3, 12, 0.12, 0.12, rule="sinks",
              lse=True),
        # single precision
        _case("single_precision", "step", _square(s13[:11]), 4, 2, 8, dtype="f32", lse=True),
        # calibration of one image's layers on the full cache
        _case("calibration", "stats", _square(s13), 4, 1, 16),
    ]


def draw(rng):
    """One more case: another schedule (prefixes of the ones above, stretched and of any aspect), another model, another way in."""
    biggest = {"bf16": 4.0e13, "f32": 2.0e11, "stats": 1.5e11}
    while True:
        kind = rng.choice(["step", "step", "step", "rule", "calls", "stats"])
        dtype = "f32" if kind != "stats" and rng.random() < 0.15 else "bf16"
        stretch, aspect = rng.uniform(0.75, 1.25), rng.choice([1.0, 1.0, rng.uniform(0.5, 2.0)])
        sides = []
        for s in synth.SIDES_19[: rng.randint(6, 17)]:
            hw = (max(1, round(s * stretch * aspect ** 0.5)), max(1, round(s * stretch / aspect ** 0.5)))
            if not sides or hw[0] * hw[1] > sides[-1][0] * sides[-1][1]:
                sides.append(hw)
        refiner = round(10 ** rng.uniform(-2.0, -0.5), 5)
        drafter = round(min(0.6, refiner * rng.choice([1, 3, 10])), 5)
        rule = {"step": "paper", "stats": "paper"}.get(kind) or rng.choice(["paper", "snapkv", "sinks", "shared"])
        case = {"kind": kind, "sides": _text(sides), "layers": round(2 ** rng.uniform(0, 5)), "batch": round(2 ** rng.uniform(0, 3)),
                "heads": rng.choice([4, 8, 12, 16, 20, 32]), "drafter": drafter, "refiner": refiner, "dtype": dtype, "rule": rule,
                "graph": kind != "stats" and rng.random() < 0.4, "page": rng.choice([0, 0, 0, 32, 64]), "lse": rng.random() < 0.3}
        if kind == "stats":
            case["batch"] = 1
        elements = sum(h * w for h, w in sides) * case["batch"] * case["heads"] * (128 if dtype == "bf16" else 64)
        held = elements * (4 * min(case["layers"], DISTINCT) + case["layers"]) * (2 if dtype == "bf16" else 4)
        if 1e6 < work(case)["flops"] <= biggest["stats" if kind == "stats" else dtype] and held < 2.5e10:
            return case


# ---- what a case does -----------------------------------------------------------------------------------------------------------
def _dim(case):
    return 128 if case["dtype"] == "bf16" else 64


def _is_drafter(layer):
    return layer % 4 == 0


def _budgets(case):
    sides = _sides(case)
    if case["kind"] == "stats":
        return [[binding.KEEP_ALL] * len(sides) for _ in range(case["layers"])]
    h, w = [s[0] for s in sides], [s[1] for s in sides]
    b = {role: binding.scalekv_budget_tokens(case["drafter" if role else "refiner"], h, w) for role in (True, False)}
    return [[b[_is_drafter(l)]] * len(sides) for l in range(case["layers"])]


def _windows(case):
    pick = binding.scalekv_window_last if case["rule"] == "snapkv" else binding.scalekv_window_centroids
    return [pick(h, w, WINDOW) for h, w in _sides(case)]


def _options(case):
    return {"paper": {}, "snapkv": {"pool_kernel": 7}, "sinks": {"policy": "recent", "n_sink": 4}, "shared": {"head_shared": True}}[case["rule"]]


def _stride(n):
    return max(1, min(16, n // 16))      # query rows sampled by the calibration


def _mix(*xs):
    h = 0x9E3779B97F4A7C15
    for x in xs:
        h = ((h ^ (int(x) + 0x7F4A7C15)) * 0xBF58476D1CE4E5B9) & 0xFFFFFFFFFFFFFFFF
        h ^= h >> 29
    return h & 0x7FFFFFFFFFFFFFFF


def _inputs(case, seed):
    """Queries, keys and values of every (distinct layer, scale): keys of a scale share an offset, four sink keys per head are
    four times as long, refiner layers look at their own scale and drafter layers at everything (see synth.py)."""
    sides, d, dev = _sides(case), _dim(case), torch.device("cuda")
    dt = synth.torch_dtype(case["dtype"])
    B, H = case["batch"], case["heads"]
    n = [h * w for h, w in sides]
    t_c = max(sum(n[:-1]), 1)
    data = {}
    for l in range(min(case["layers"], DISTINCT)):
        g = torch.Generator(device=dev)
        g.manual_seed(_mix(seed, l))
        sinks = torch.randint(0, t_c, (B, H, 4), generator=g, device=dev)
        sinks[:, :, 0] = 0
        base = 0
        for k, nk in enumerate(n):
            Q, K, V = (torch.randn(B, H, nk, d, generator=g, device=dev) for _ in range(3))
            mu = 0.5 * torch.randn(B, H, 1, d, generator=g, device=dev)
            K += mu
            if _is_drafter(l):
                Q *= 0.25
            else:
                Q += mu
            at = sinks - base
            inside = (at >= 0) & (at < nk)
            gain = torch.ones(B, H, nk, device=dev)
            gain.scatter_reduce_(2, at.clamp(0, nk - 1), torch.where(inside, 4.0, 1.0), "amax")
            K *= gain.unsqueeze(-1)
            data[l, k] = tuple(t.to(dt) for t in (Q, K, V))
            base += nk
    return data


def prepare(case, seed):
    sides = _sides(case)
    s = {"case": case, "n": [h * w for h, w in sides], "windows": _windows(case), "options": _options(case), "inputs": _inputs(case, seed)}
    kv = s["kv"] = binding.ScaleKV(case["layers"], case["batch"], case["heads"], _dim(case), case["dtype"], [a for a, _ in sides],
                                   [b for _, b in sides], _budgets(case), max_window=WINDOW, page_tokens=case["page"],
                                   window_kind="last" if case["rule"] == "snapkv" else "centroids")
    s["arrays"] = [kv.window_array(w) for w in s["windows"]]
    if case["kind"] != "stats":
        shape, dt = (case["layers"], case["batch"], case["heads"]), synth.torch_dtype(case["dtype"])
        s["O"] = [torch.zeros(*shape, n, _dim(case), dtype=dt, device="cuda") for n in s["n"]]
        s["lse"] = [torch.zeros(*shape, n, device="cuda") for n in s["n"]] if case["lse"] else None
    torch.cuda.synchronize()
    if case["graph"]:
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], stream=kv.stream_main, capture_error_mode="thread_local"):
            _pass(s)
    return s


def _pass(s):
    case, kv, options = s["case"], s["kv"], s["options"]
    kind, last = case["kind"], len(s["n"]) - 1
    kv.scalekv_reset()
    for k in range(len(s["n"])):
        window, array = s["windows"][k], s["arrays"][k]
        for l in range(case["layers"]):
            Q, K, V = s["inputs"][l % DISTINCT, k]
            O = s["O"][k][l]
            lse = s["lse"][k][l] if s["lse"] is not None else None
            if kind == "step":
                kv.scalekv_step(l, k, Q, K, V, O, window_pos=array if k < last else None, lse=lse)
            elif kind == "rule":
                kv.scalekv_step_ex(l, k, Q, K, V, O, compress=k < last, window_pos=array, lse=lse, **options)
            else:
                kv.scalekv_append(l, k, K, V)
                kv.scalekv_attend(l, Q, O, lse=lse)
                if k < last and options:
                    kv.scalekv_compress_ex(l, Q, window, qw_is_full_map=True, **options)
                elif k < last:
                    kv.scalekv_compress(l, Q, window, qw_is_full_map=True)
    kv.scalekv_join()


def run(s):
    kv, here = s["kv"], torch.cuda.current_stream()
    kv.stream_main.wait_stream(here)           # the model's own kernels come before and after the pass
    if s["case"]["kind"] == "stats":
        kv.scalekv_reset()
        out = []
        for k, n in enumerate(s["n"]):
            for l in range(s["case"]["layers"]):
                Q, K, V = s["inputs"][l % DISTINCT, k]
                kv.scalekv_append(l, k, K, V)
                car, htk, cars, htks, ncas = kv.scalekv_layer_stats_ex(l, Q, TOPK_PRIME, _stride(n))
                out.append([[car, htk, 0.0]] + [list(x) for x in zip(cars[0], htks[0], ncas[0])])
        return np.array(out)
    if s["case"]["graph"]:
        with torch.cuda.stream(kv.stream_main):
            s["graph"].replay()
    else:
        _pass(s)
    here.wait_stream(kv.stream_main)
    return {"O": s["O"], "lse": s["lse"]}


def work(case):
    """Attention flops; queries, keys and values in, outputs out, the cached rows read once per step, the rows the cache grows by
    written (an evicting step has to move at least those)."""
    n, d = [h * w for h, w in _sides(case)], _dim(case)
    slices, size = case["batch"] * case["heads"], 2 if case["dtype"] == "bf16" else 4
    flops = moved = 0
    for role in (True, False):
        layers = sum(_is_drafter(l) == role for l in range(case["layers"]))
        budget = int(case["drafter" if role else "refiner"] * sum(n[:-1]) + 0.5)
        hist = 0
        for k, nk in enumerate(n):
            length = hist + nk
            rows = -(-nk // _stride(nk)) if case["kind"] == "stats" else nk
            flops += layers * (2 if case["kind"] == "stats" else 4) * rows * length * d * slices
            window = 0 if case["rule"] == "sinks" else min(WINDOW, nk)
            kept = length if case["kind"] == "stats" else min(length, budget + window)
            grown = max(kept - hist, 0) if k + 1 < len(n) else 0
            if case["kind"] == "stats":
                moved += layers * slices * size * d * (rows + hist + 4 * nk)
            else:
                moved += layers * slices * (size * d * (4 * nk + 2 * hist + 2 * grown) + (4 * nk if case["lse"] else 0))
            hist = kept
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    # Against the same pass in 64 bits: calibration 3e-8 (largest 1e-7), single precision 1.1e-6 (1.5e-5), bf16 2.4e-3 (0.018 with
    # the same entries kept; where two entries whose importances agree to six digits change places, rows of that head move by up
    # to 0.33 of the root mean square).
    if case["kind"] == "stats":
        return {"rel": 1e-6, "max": 1e-5}
    if case["dtype"] == "f32":
        return {"rel": 5e-6, "max": 1e-4}
    return {"rel": 1e-2, "max": 0.5}
