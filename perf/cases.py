"""The work that users of this library have it do, as cases for timing.

A denoising loop calls `heart_step` once per layer and step, with the TMR state of the layer carried
along; its first steps run dense (`HEART_FORCE_DENSE`), and the backbone may bring the strided
antidiagonal estimator (`HEART_ESTIMATOR_ANTIDIAG`).  A program with block lists of its own calls
`heart_block_sparse_attn`.  The offline calibration reads realised sparsities (drift and masks, no
attention) and band errors, and the mask-reuse study reads full-token drifts and mask IoUs.

A case is a dict of plain values; `do` says which of these it is.  Shapes and thresholds are those of
`paper_2605_14513_b200.inputs`, of the benchmark and of the tests; the tensors come from
`inputs.Sequence` (random values plus a positional term, so that attention is local), and a state has
its anchors and masks from the step before the one that is timed.
"""
import math

import numpy as np
import torch

from paper_2605_14513_b200 import heart, inputs

D = 128


def _case(name, do, B, H, grid, block, tau, density, gain=2.6, refresh=1.0, gate=False, layout="bhnd", lse=False):
    return {"name": name, "do": do, "B": B, "H": H, "T": grid[0], "Y": grid[1], "X": grid[2], "block": block,
            "tau_lo": tau[0], "tau_hi": tau[1], "density": density, "gain": gain, "refresh": refresh, "gate": gate,
            "layout": layout, "lse": lse}


def listed():
    """density: share of the block pairs that these thresholds retain, measured; only work() reads it."""
    return [
        # A layer of a toy model or of a unit test: two heads, everything in L2, latency and launches.
        _case("step_2x2k_b64", "step", 1, 2, (2, 32, 32), 64, (0.90, 0.95), 0.477, gain=2.5, refresh=0.5),
        # A short clip with guidance (two batch entries), [B, N, H, D] tensors as projections leave them, a
        # token count that no tile divides, the layer gate on, log-sum-exp wanted.
        _case("step_2x12x2465_b64_gate", "step", 2, 12, (5, 17, 29), 64, (0.85, 0.97), 0.348, refresh=0.5, gate=True,
              layout="bnhd", lse=True),
        # Wan2.1-1.3B at 480P: the usual step, about a third of the heads refresh their masks.
        _case("step_12x33k_b64", "step", 1, 12, (21, 30, 52), 64, (0.85, 0.98), 0.150, refresh=0.3),
        # Wan2.1-14B at 480P: 40 heads, half of them refreshing.
        _case("step_40x33k_b64", "step", 1, 40, (21, 30, 52), 64, (0.85, 0.98), 0.101, refresh=0.5),
        # Wan2.1-14B at 720P: the largest step, 128-token blocks, a fifth of the heads refreshing.
        _case("step_40x76k_b128", "step", 1, 40, (21, 45, 80), 128, (0.92, 0.98), 0.128, refresh=0.2),
        # HunyuanVideo at 720P: the longest sequence, every head refreshing.
        _case("step_24x119k_b128", "step", 1, 24, (33, 45, 80), 128, (0.80, 0.97), 0.070, refresh=1.0),
        # The warm-up steps of a sweep: attention over all blocks.
        _case("dense_12x33k_b64", "dense", 1, 12, (21, 30, 52), 64, (0.9, 0.9), 1.0),
        # The antidiagonal estimator as its backbone is configured (stride 16, 128-token blocks).
        _case("antidiag_12x33k_b128", "antidiag", 1, 12, (21, 30, 52), 128, (0.85, 0.95), 0.131),
        # Calibration, realised sparsity of a threshold: drift and masks of every head, no attention.
        _case("masks_24x119k_b128", "masks", 1, 24, (33, 45, 80), 128, (0.80, 0.97), 0.070),
        # A program with lists of its own: attention alone, odd sizes, strided tensors, log-sum-exp.
        _case("attend_16x8k_b128", "attend", 1, 16, (7, 27, 43), 128, (0.85, 0.95), 0.237, layout="bnhd", lse=True),
        # The mask-reuse study: full-token drift and mask IoU between two steps.
        _case("study_12x33k_b64", "study", 1, 12, (21, 30, 52), 64, (0.85, 0.98), 0.150),
        # Calibration, frequency-aware error of one probe: a 480P latent (16 channels).
        {"name": "band_error_480p", "do": "band_error", "C": 16, "T": 21, "Y": 60, "X": 104},
    ]


def _density(n_blocks, tau_lo, tau_hi, gain):
    """Rough share of retained pairs of such inputs, a fit to measurements (work() of drawn cases only)."""
    d = 0.357 * n_blocks ** -0.33 * (1.0 - 0.5 * (tau_lo + tau_hi)) ** -0.48 * (2.6 / gain) ** 3.6
    return min(1.0, d)


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    do = rng.choice(["step"] * 9 + ["antidiag"] * 2 + ["attend"] * 2 + ["dense", "masks", "study", "band_error"])
    if do == "band_error":
        return {"do": do, "C": rng.choice([4, 16]), "T": rng.randint(5, 33), "Y": rng.randint(30, 96), "X": rng.randint(40, 170)}
    tokens = _log_uniform(rng, 400, 118800)
    T = max(1, min(33, round(_log_uniform(rng, 1, 33)), int(tokens / 64)))
    Y = max(4, round(math.sqrt(tokens / T * rng.uniform(0.4, 0.9))))
    X = max(8, round(tokens / (T * Y)))
    while T * Y * X > 118800:
        X -= 1
    N = T * Y * X
    block = rng.choice([64, 128]) if N <= 45000 else 128
    nb = -(-N // block)
    lo = rng.uniform(0.80, 0.92)
    hi = rng.uniform(lo + 0.02, 0.98)
    gain = rng.uniform(2.4, 2.8)
    density = 1.0 if do == "dense" else _density(nb, lo, hi, gain)
    # no more tokens in all and no more attention than the largest listed case
    most = min(3.0e6 / N, 2.6e10 / (float(N) * N * density))
    if do == "antidiag":
        most = min(most, 3.0e10 / (float(N) * N))
    heads = max(1, min(int(most), round(_log_uniform(rng, 1, 48))))
    B = 2 if heads % 2 == 0 and rng.random() < 0.3 else 1
    return {"do": do, "B": B, "H": heads // B, "T": T, "Y": Y, "X": X, "block": block, "tau_lo": round(lo, 3),
            "tau_hi": round(hi, 3), "density": round(density, 4), "gain": round(gain, 3),
            "refresh": rng.choice([0.0, 0.2, 0.5, 1.0]) if do == "step" else 1.0, "gate": do == "step" and rng.random() < 0.2,
            "layout": rng.choice(["bhnd", "bnhd"]), "lse": rng.random() < 0.3}


def _workload(case, seed):
    R = case["B"] * case["H"]
    rs = np.random.RandomState(seed % (1 << 31))
    tau = np.linspace(case["tau_lo"], case["tau_hi"], R)[rs.permutation(R)]
    # heads that refresh: a negative threshold always does; the others: a threshold that is never reached
    n_ref = round(case["refresh"] * R)
    delta = np.where(rs.permutation(R) < n_ref, -1.0, 1e6)
    return inputs.Workload("case", case["H"], (case["T"], case["Y"], case["X"]), case["block"], tau, delta, np.full(R, 0.05),
                           np.full(R, case["gain"]), seed=seed, steps=2, B=case["B"])


def _tensors(seq, layout):
    out = seq.bf16()
    if layout == "bnhd":
        out = tuple(x.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for x in out)
    return out


def prepare(case, seed):
    if case["do"] == "band_error":
        g = torch.Generator("cuda").manual_seed(seed)
        shape = (case["C"], case["T"], case["Y"], case["X"])
        dense = torch.randn(shape, generator=g, device="cuda")
        return {"do": "band_error", "dense": dense, "sparse": dense + 0.05 * torch.randn(shape, generator=g, device="cuda")}
    do, layout = case["do"], case["layout"]
    wl = _workload(case, seed)
    seq = inputs.Sequence(wl, "cuda")
    Q, K, V = _tensors(seq, layout)
    flags = {"dense": heart.FORCE_DENSE, "antidiag": heart.ESTIMATOR_ANTIDIAG}.get(do, 0)
    gate = (0.4, 0.8) if case["gate"] else (0.0, 1.0)
    cfg = heart.config_for(Q, case["block"], gate_lo=gate[0], gate_hi=gate[1], flags=flags)
    st, ws = heart.State(cfg), heart.new_workspace(cfg)
    s = {"do": do, "cfg": cfg, "st": st, "ws": ws, "O": torch.empty_like(Q),
         "tau": torch.tensor(wl.tau, dtype=torch.float64, device="cuda"),
         "delta": torch.tensor(wl.delta, dtype=torch.float64, device="cuda"),
         "drift": torch.empty(wl.R, dtype=torch.float64, device="cuda"),
         "refresh": torch.empty(wl.R, dtype=torch.uint8, device="cuda"),
         "lse": torch.empty((wl.R, wl.N), dtype=torch.float32, device="cuda") if case["lse"] else None}
    if do != "dense":  # the step before: anchors and masks
        heart.heart_drift(cfg, Q, K, s["delta"], st, ws)
        heart.heart_predict_mask(cfg, Q, K, s["tau"], st, ws)
    if do == "study":
        s["Qa"], s["Ka"], s["mask_a"] = Q, K, st.mask_bits.clone()
    if do != "attend":
        seq.advance()
        Q, K, V = _tensors(seq, layout)
    if do == "study":
        heart.heart_predict_mask(cfg, Q, K, s["tau"], st, ws)
        s["iou"] = torch.empty(wl.R, dtype=torch.float64, device="cuda")
        s["counts"] = torch.empty((wl.R, 2), dtype=torch.int64, device="cuda")
    s["Q"], s["K"], s["V"] = Q, K, V
    return s


def run(s):
    do = s["do"]
    if do == "band_error":
        return heart.heart_band_error(s["sparse"], s["dense"])
    cfg, st, ws = s["cfg"], s["st"], s["ws"]
    if do == "study":
        heart.heart_full_token_drift(cfg, s["Qa"], s["Ka"], s["Q"], s["K"], s["drift"], ws)
        heart.heart_mask_iou(cfg, s["mask_a"], st.mask_bits, s["iou"], s["counts"])
        return s["drift"], s["iou"], s["counts"]
    if do == "attend":
        heart.heart_block_sparse_attn(cfg, s["Q"], s["K"], s["V"], st.kv_idx, st.kv_cnt, s["O"], ws, lse=s["lse"])
        return s["O"], s["lse"]
    if do == "masks":
        heart.heart_drift(cfg, s["Q"], s["K"], s["delta"], st, ws, drift_out=s["drift"], refresh_out=s["refresh"])
        heart.heart_predict_mask(cfg, s["Q"], s["K"], s["tau"], st, ws, refresh=s["refresh"], means_valid=True)
        return s["drift"], s["refresh"], st.tensors()
    heart.heart_step(cfg, s["Q"], s["K"], s["V"], s["delta"], s["tau"], st, s["O"], ws, lse=s["lse"], drift_out=s["drift"],
                     refresh_out=s["refresh"])
    if do == "dense":
        return s["O"], s["lse"]
    return s["O"], s["lse"], s["drift"], s["refresh"], st.tensors()


def work(case):
    if case["do"] == "band_error":
        n, points = case["C"] * case["T"] * case["Y"] * case["X"], case["T"] * case["Y"] * case["X"]
        return {"bytes": 8.0 * n, "flops": 2.5 * n * math.log2(points) + 12.0 * n}  # one real transform, the sums
    do, block = case["do"], case["block"]
    R, N = case["B"] * case["H"], case["T"] * case["Y"] * case["X"]
    nb = -(-N // block)
    tensor, pairs = 2.0 * R * N * D, R * float(nb) * nb
    lists = (4.0 * case["density"] + 0.125) * pairs
    if do == "study":
        return {"bytes": 4 * tensor + 0.25 * pairs, "flops": 6.0 * R * N * D + 3.0 * pairs}
    attention = 4.0 * D * R * float(N) * N * case["density"]
    if do in ("attend", "dense"):
        return {"bytes": 4 * tensor + (lists if do == "attend" else 0.0), "flops": attention}
    refreshed = round(case["refresh"] * R) / R
    scores = 2.0 * pairs * D if do != "antidiag" else 2.0 * R * float(N // 16) ** 2 * 16 * D
    flops = 2.0 * R * N * D + refreshed * scores
    if do == "masks":
        return {"bytes": 2 * tensor + lists, "flops": flops}
    return {"bytes": 4 * tensor + lists, "flops": flops + attention}


def tolerance(case):
    """About four times what the paths differ by from themselves in 64 bits (sampled rows of every listed case)."""
    do = case["do"]
    if do == "band_error":
        return {"rel": 1e-14}  # fp64 throughout: 9e-16 against a direct transform
    if do == "study":
        return {"rel": 2e-12}  # 3e-13
    if do == "masks":
        return {"rel": 3e-9}  # drift 7e-10; masks equal
    if do == "antidiag":  # importances from bf16 products with fp32 sums: a row in some hundred may cut elsewhere
        return {"rel": 7e-3, "max": 2.5e-2, "differ": 4e-4}
    return {"rel": 7e-3, "max": 2.5e-2}  # bf16 weights and outputs: 1.7e-3, largest 6e-3
