"""Performance cases: what a user of the framework has it do, with the inputs and the work of each.

Three kinds of case, all through the public binding (paper_1901_08924_b200.lpc):

  "round"  one communication round on gradient vectors that the user's own model produced: quantize and pack N worker
           vectors, count their coded size if asked, pass them through the chosen scheme of the paper (broadcast, or a
           server that sums or re-quantizes), decode, average, proximal step.
  "train"  a training job on a linear model from a given iterate: `epochs` times a snapshot pass and `m` inner steps of
           Algorithm 1 ("lpc") or of Algorithms 2/3 ("alpc"), with the objective at the end if asked.
  "host"   the same job for a user whose data lie in host memory.
"""
import math
import random

import torch

from paper_1901_08924_b200 import lpc, synth

CLIPS = {"none": lpc.CLIP_NONE, "lambda": lpc.CLIP_LAMBDA, "std": lpc.CLIP_STD}
LOSSES = {"logistic": lpc.LOGISTIC, "least_squares": lpc.LEAST_SQUARES}


def _round(name, N, length, b, clip="std", clip_value=2.0, dist="gauss", tensors="one", sub=False, scheme="broadcast",
           count=False):
    return dict(name=name, kind="round", N=N, length=length, b=b, clip=clip, clip_value=clip_value, dist=dist,
                tensors=tensors, sub=sub, scheme=scheme, count=count)


def _train(name, method, loss, n, d, N, B, b, m, epochs=1, clip="std", clip_value=2.0, objective=False):
    return dict(name=name, kind="train", method=method, loss=loss, n=n, d=d, N=N, B=B, b=b, m=m, epochs=epochs, clip=clip,
                clip_value=clip_value, objective=objective)


def listed():
    return [
        # a small linear model's gradient (1,000 features, as the small logistic workload): latency is all there is
        _round("round_1k", 4, 1000, 2, clip_value=2.5),
        # the shortest vector of the quantizer sweep: a small network's gradient
        _round("round_64k", 8, 1 << 16, 4),
        # a vector of odd length with the paper's three levels and Eq. 2's lambda
        _round("round_1m_odd", 8, 1000003, 3, clip="lambda", clip_value=0.5),
        # layer-wise use: the 62 tensors of an 18-layer residual network, current minus snapshot gradient formed in the call
        _round("round_layers", 16, synth.segment_offsets(synth.resnet18_shapes())[-1], 4, clip_value=2.5,
               tensors="resnet18", sub=True),
        # 8-bit codes of heavy-tailed gradients without clipping, with the entropy-coded size of every message counted
        _round("round_16m_counted", 8, 1 << 24, 8, clip="none", clip_value=1.0, dist="student_t3", count=True),
        # a parameter server that adds the codes on a common grid (scheme (b))
        _round("round_4m_server", 8, 1 << 22, 4, scheme="sum"),
        # a large model's gradient, the middle of the sweep's long end
        _round("round_64m", 8, 1 << 26, 4),
        # the small logistic workload, with the objective that the user watches
        _train("train_tiny_logistic", "lpc", "logistic", 4000, 1000, 4, 1, 2, 1000, clip_value=2.5, objective=True),
        # the benchmark's workload: one epoch
        _train("train_least_squares", "lpc", "least_squares", 131072, 4096, 16, 8, 4, 1024, clip_value=3.0),
        # the accelerated method on the wide logistic workload: one epoch
        _train("train_alpc_logistic", "alpc", "logistic", 262144, 8192, 32, 16, 2, 512),
        # large minibatches, whose rows stream through the worker kernel
        _train("train_large_batch", "lpc", "logistic", 65536, 8192, 32, 256, 2, 64),
        # a job on host data: two epochs on a matrix of 268 MB in pinned memory
        dict(name="host_job", kind="host", loss="least_squares", n=32768, d=2048, N=8, B=8, b=4, m=512, epochs=2, clip="std",
             clip_value=3.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_clip(rng):
    clip = rng.choice(["std", "std", "std", "lambda", "none"])
    return clip, {"std": rng.choice([1.0, 2.0, 2.5, 3.0, 4.0]), "lambda": rng.choice([0.25, 0.5, 0.9]), "none": 1.0}[clip]


def _draw_round(rng):
    N = rng.choice([1, 2, 3, 4, 8, 8, 16, 16, 32])
    b = rng.choice([1, 2, 2, 3, 3, 4, 4, 4, 4, 6, 8, 8, 16, 32])
    clip, value = _draw_clip(rng)
    sub = rng.random() < 0.3
    length = _log(rng, 500, min(1 << 26, (1 << (28 if sub else 29)) // N))
    tensors = rng.choice(["one", "one", "one", "resnet18", "cut"])
    if tensors == "resnet18":
        length = synth.segment_offsets(synth.resnet18_shapes())[-1]
    scheme, count = "broadcast", False
    if 2 <= b <= 8 and rng.random() < 0.3:
        scheme = rng.choice(["sum", "requantize"])
    elif b <= 8 and rng.random() < 0.25:
        count = True
    case = _round("", N, length, b, clip, value, rng.choice(["gauss", "gauss", "student_t3"]), tensors, sub, scheme, count)
    del case["name"]
    return case


def _draw_train(rng):
    method = rng.choice(["lpc", "lpc", "alpc"])
    N, B = rng.choice([2, 4, 5, 8, 16, 16, 32]), rng.choice([1, 2, 4, 8, 8, 16, 16, 32, 100, 256])
    d = 4 * _log(rng, 16, 4096)
    n = max(1, _log(rng, 2000, max(4000, (1 << 29) // d)) // N) * N
    m = max(16, min(_log(rng, 64, 1024), (1 << 31) // (N * B * d)))
    clip, value = _draw_clip(rng)
    case = _train("", method, rng.choice(["logistic", "least_squares"]), n, d, N, B, rng.choice([1, 2, 3, 4, 4, 8, 32]), m,
                  rng.choice([1, 1, 2]), clip, value, rng.random() < 0.3)
    del case["name"]
    return case


def draw(rng):
    """One more case: gradient rounds of 500 to 2^26 values per worker, training on 2,000 rows of 64 to 16,384 features up
    to 2 GiB, every clip rule, the code widths in use, ragged sizes; now and then a job on host data."""
    u = rng.random()
    if u < 0.6:
        return _draw_round(rng)
    if u < 0.93:
        return _draw_train(rng)
    N, d = rng.choice([2, 4, 8, 16]), 4 * _log(rng, 64, 2048)
    clip, value = _draw_clip(rng)
    return dict(kind="host", loss=rng.choice(["logistic", "least_squares"]), n=max(1, _log(rng, 2000, (1 << 26) // d) // N) * N, d=d,
                N=N, B=rng.choice([1, 4, 8]), b=rng.choice([2, 4, 8]), m=_log(rng, 100, 512), epochs=rng.choice([1, 2, 3]),
                clip=clip, clip_value=value)


def _offsets(case):
    """Element offsets of the tensors that make up the vector, or None for a single one."""
    if case["tensors"] == "one":
        return None
    if case["tensors"] == "resnet18":
        return synth.segment_offsets(synth.resnet18_shapes())
    rng = random.Random(case["length"])  # "cut": a parameter list of matrices and vectors, sizes over three decades
    sizes = [math.exp(rng.uniform(0.0, math.log(1000.0))) for _ in range(max(2, min(40, case["length"] // 100)))]
    total, offs = sum(sizes), [0]
    for s in sizes[:-1]:
        offs.append(min(case["length"], offs[-1] + max(1, int(case["length"] * s / total))))
    return offs + [case["length"]]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _gradients(case, g, offs):
    """N gradient vectors, each starting on a 16-byte boundary; the scale differs from tensor to tensor as in a network."""
    N, length = case["N"], case["length"]
    base = torch.empty((N, (length + 3) // 4 * 4), device="cuda")
    base.normal_(generator=g)
    if case["dist"] == "student_t3":
        for i in range(N):
            c = torch.zeros(base.shape[1], device="cuda")
            for _ in range(3):
                c += torch.randn(base.shape[1], generator=g, device="cuda").square_()
            base[i] /= c.div_(3.0).sqrt_()
    if offs is not None:
        rng = random.Random(len(offs))
        for a, e in zip(offs, offs[1:]):
            base[:, a:e] *= 10.0 ** rng.uniform(-4.0, -1.0)
    return base[:, :length]


def _prepare_round(case, seed):
    N, length, b = case["N"], case["length"], case["b"]
    g, offs = _generator(seed), _offsets(case)
    nseg = 1 if offs is None else len(offs) - 1
    st = dict(kind="round", k=0, length=length, offs=offs, scheme=case["scheme"], count=case["count"])
    st["U"] = _gradients(case, g, offs)
    st["sub"] = _gradients(case, g, offs) if case["sub"] else None
    st["mu"] = torch.randn(length, generator=g, device="cuda") * 0.01 if case["sub"] else None
    st["x"] = torch.randn(length, generator=g, device="cuda")
    ctx = lpc.Context(None, None, lpc.LOGISTIC, 0.0, N, 1, b, CLIPS[case["clip"]], case["clip_value"], seed)
    st["ctx"] = st["decoder"] = ctx
    # the buffers that a training loop keeps from round to round
    stride = lpc.packed_layout(length, b, offs)[1]
    st["codes"] = torch.zeros((N, stride), dtype=torch.int32, device="cuda")
    st["delta"] = torch.zeros((N, nseg), device="cuda")
    st["clipped"] = torch.zeros((N, nseg), dtype=torch.int32, device="cuda")
    if case["count"]:
        st["hist"] = torch.zeros((N, nseg, 1 << b), dtype=torch.int64, device="cuda")
    if case["scheme"] != "broadcast":
        ctx.set_option(lpc.OPT_SHARED_SCALE, 1)
        st["server"] = lpc.SCHEME_SERVER_SUM if case["scheme"] == "sum" else lpc.SCHEME_SERVER_REQUANTIZE
        bits = lpc.sum_bits(b, N) if case["scheme"] == "sum" else b
        st["reduced"] = torch.zeros((1, lpc.packed_layout(length, bits, offs)[1]), dtype=torch.int32, device="cuda")
        st["decoder"] = lpc.Context(None, None, lpc.LOGISTIC, 0.0, 1, 1, bits, lpc.CLIP_NONE, 1.0, seed)
        if case["scheme"] == "sum":
            st["decoder"].set_option(lpc.OPT_AVERAGE_DIVISOR, N)
    return st


def _problem(case, seed):
    """X with independent N(0, 1/d) entries, labels from a planted sparse model, and the Lipschitz constant."""
    n, d = case["n"], case["d"]
    g = _generator(seed)
    X = torch.empty((n, d), device="cuda")
    X.normal_(std=1.0 / math.sqrt(d), generator=g)
    w = torch.randn(d, generator=g, device="cuda") * (torch.rand(d, generator=g, device="cuda") < 0.1)
    t = X @ w + 0.1 * torch.randn(n, generator=g, device="cuda")
    y = t if case["loss"] == "least_squares" else torch.where(t >= 0, 1.0, -1.0)
    L = float(torch.linalg.vector_norm(X, dim=1).max()) ** 2 * (1.0 if case["loss"] == "least_squares" else 0.25)
    return X, y, L, 0.1 * torch.randn(d, generator=g, device="cuda")


def prepare(case, seed):
    if case["kind"] == "round":
        return _prepare_round(case, seed)
    X, y, L, x0 = _problem(case, seed)
    st = dict(case, seed=seed, k=0, L=L)
    if case["kind"] == "host":
        st["X"], st["y"] = (torch.empty(t.shape, pin_memory=True).copy_(t) for t in (X, y))
        st["x0"] = x0.cpu()
        return st
    st["x0"] = x0
    st["mu"] = torch.zeros(case["d"], device="cuda")
    st["ctx"] = lpc.Context(X, y, LOSSES[case["loss"]], 1e-4, case["N"], case["B"], case["b"], CLIPS[case["clip"]],
                            case["clip_value"], seed)
    return st


def _run_round(st):
    ctx, k, length, offs = st["ctx"], st["k"], st["length"], st["offs"]
    st["k"] += 1
    codes, delta, clipped = ctx.quantize_pack(st["U"], k, U_sub=st["sub"], seg_offsets=offs, codes_out=st["codes"],
                                              delta_out=st["delta"], clipped_out=st["clipped"])
    out = dict(codes=codes, delta=delta, clipped=clipped)
    if st["count"]:
        out["hist"], out["entropy"], out["huffman"] = ctx.message_entropy(codes, length, seg_offsets=offs, hist_out=st["hist"])
    if st["scheme"] != "broadcast":
        codes, _ = ctx.server_reduce(codes, length, st["server"], k, seg_offsets=offs, codes_out=st["reduced"])
        out["reduced"] = codes
    out["x"] = st["decoder"].unpack_average_prox(codes, delta, length, st["x"], 0.01, 1e-4, mu=st["mu"], seg_offsets=offs)
    return out


def _run_train(st):
    ctx, m, L = st["ctx"], st["m"], st["L"]
    ctx.set_iterate(st["x0"])
    if st["method"] == "alpc":
        ctx.alpc_begin()
    for s in range(st["epochs"]):
        ctx.snapshot_full_grad(mu_out=st["mu"])
        if st["method"] == "lpc":
            ctx.inner_steps(1.0 / (6.0 * L), st["k"], m)
        else:  # Algorithm 3's parameters
            tau1 = 2.0 / (s + 4)
            ctx.alpc_double_sample_steps(tau1, 0.5, 1.0 / (6.0 * L * tau1), 1.0 / (4.0 * L), st["k"], m)
            ctx.alpc_end_epoch(m)
        st["k"] += m
    out = dict(x=ctx.get_iterate(), mu=st["mu"])
    if st["method"] == "alpc":
        out["y"], out["z"] = ctx.get_buffer(lpc.BUF_Y), ctx.get_buffer(lpc.BUF_Z)
    if st["objective"]:
        out["objective"] = ctx.objective()
    return out


def run(st):
    if st["kind"] == "round":
        return _run_round(st)
    if st["kind"] == "train":
        return _run_train(st)
    x, objective, _ = lpc.svrg_run_host(st["X"], st["y"], LOSSES[st["loss"]], 1e-4, st["N"], st["B"], st["b"],
                                        CLIPS[st["clip"]], st["clip_value"], st["seed"], st["epochs"], st["m"],
                                        1.0 / (6.0 * st["L"]), st["x0"])
    return dict(x=x, objective=objective)


def work(case):
    if case["kind"] == "round":
        N, length, b = case["N"], case["length"], case["b"]
        # the vectors once, the messages once, the iterate read and written; per value: magnitude, two sums, scale, round
        out = 0.0
        if case["scheme"] != "broadcast":
            out = length * (b + (math.ceil(math.log2(N)) if case["scheme"] == "sum" else 0)) / 8.0
        return dict(bytes=N * length * (4.0 * (2 if case["sub"] else 1) + b / 8.0) + length * (12.0 if case["sub"] else 8.0) + out,
                    flops=10.0 * N * length)
    n, d, N, B, m, epochs = (float(case[k]) for k in ("n", "d", "N", "B", "m", "epochs"))
    passes = epochs + (1 if case["kind"] == "host" or case.get("objective") else 0)
    rows = (N + (1 if case.get("method") == "alpc" else 0)) * B * m * epochs
    # X and the labels once per pass over the data, the sampled rows, their labels and margins
    return dict(bytes=passes * 4.0 * n * (d + 1) + rows * 4.0 * (d + 2), flops=4.0 * n * d * epochs + 2.0 * n * d * (passes - epochs) + 4.0 * rows * d)


def tolerance(case):
    if case["kind"] == "round":
        # codes, scales and decoded vectors are defined to the bit; the coded sizes are sums in double precision
        return {"rel": 1e-12, "max": 1e-10} if case["count"] else "exact"
    # full gradients are 32-bit sums whose order is free; a trajectory amplifies their last bits where a code flips
    return {"rel": 3e-5, "max": 1e-3}
