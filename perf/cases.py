"""Performance cases of the library: products and training steps as programs
call them, over the range of sizes, kinds and options in use.

listed() gives the named cases, draw(rng) one more of the same ranges,
prepare(case, seed) the inputs a program holds before the call, run(state) one
pass through the public entry points, work(case) the bytes and operations a
pass cannot do without, and exact(case, seed) the outputs in plain binary64.

Three families:
  gemm   hs.gemm on device tensors (binary64, int8 or bf16 slices; the caller's
         grid or the automatic configuration; both grid layouts);
  host   hs.gemm_host on pinned host tensors (copies in, product, copy out);
  train  one step of the cost model's training: the backward pass of
         hsumma_mlp_backward and the update of hsumma_mlp_adam.
"""
import math

import torch

import paper_1306_4161_gb300 as hs

AUTO = dict(P=0, Q=0, G=0, b=0, Bouter=0)
TILE = {"fp64": (128, 128, 32), "int8": (128, 128, 128), "bf16": (128, 256, 64)}
TRAIN_STEP = 1000          # the Adam step number a pass stands at


def _gemm(name, M, N, K, kind="fp64", slices=0, layout="block", dist="uniform", family="gemm",
          **cfg):
    return dict(name=name, family=family, M=M, N=N, K=K, kind=kind, slices=slices,
                layout=layout, dist=dist, **(cfg or AUTO))


def listed():
    return [
        # the smallest workload of the library: 512^3 on a 4 x 4 grid in 2 x 2 groups
        _gemm("fp64_512_grid4x4", 512, 512, 512, P=4, Q=4, G=4, b=32, Bouter=64),
        # a product of no round size handed over without a configuration; its
        # odd rows are not 16-byte aligned
        _gemm("fp64_ragged_auto", 1500, 1301, 1201),
        # the G sweep's shape at G = sqrt(p): a 16 x 16 grid of 256 x 256 blocks
        # in groups of 4 x 4
        _gemm("fp64_4096_grid16x16", 4096, 4096, 4096, P=16, Q=16, G=16, b=64, Bouter=128),
        # the rectangular workload's proportions and 12 x 16 grid, an eighth of
        # its sizes, dealt block-cyclically
        _gemm("fp64_rect_cyclic", 3072, 2048, 4096, dist="normal_spiked", layout="cyclic",
              P=12, Q=16, G=48, b=32, Bouter=128),
        # a small split product, where launches and latency count
        _gemm("bf16_512_s4", 512, 512, 512, "bf16", 4, P=4, Q=2, G=4, b=64, Bouter=128),
        # an ordinary split product of odd sizes, configuration left to the library
        _gemm("bf16_ragged_auto_s5", 3001, 2047, 2500, "bf16", 5, dist="wide"),
        # the benchmark's product and launch
        _gemm("bf16_16384_s4", 16384, 16384, 16384, "bf16", 4, P=128, Q=64, G=4096, b=64,
              Bouter=512),
        # the rectangular workload at full size: 1 % of A's columns scaled by 1e6
        _gemm("bf16_rect_s5", 24576, 16384, 32768, "bf16", 5, dist="normal_spiked", P=192, Q=64,
              G=6144, b=64, Bouter=512),
        # int8 slices on a flat grid, six of them for binary64 accuracy
        _gemm("int8_4096_s6", 4096, 4096, 4096, "int8", 6, P=32, Q=32, G=1, b=128, Bouter=2048),
        # wide-range inputs with every int8 slice, odd sizes, left to the library
        _gemm("int8_ragged_auto_s8", 1153, 1700, 1301, "int8", 8, dist="wide"),
        # a product that starts and ends in host memory
        _gemm("host_bf16_4096_s4", 4096, 4096, 4096, "bf16", 4, family="host", P=32, Q=16, G=256,
              b=64, Bouter=256),
        # one training step of the cost model on a full batch of its samples
        dict(name="train_2400", family="train", batch=2400),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))))


def _flops(c):
    pairs = c["slices"] * (c["slices"] + 1) // 2 if c["kind"] != "fp64" else 1
    return 2.0 * c["M"] * c["N"] * c["K"] * pairs


def draw(rng):
    if rng.random() < 0.1:
        return dict(family="train", batch=_log_int(rng, 64, 4096))
    family = "host" if rng.random() < 0.12 else "gemm"
    kind = rng.choice(("fp64", "bf16", "bf16", "int8"))
    hi, most = {"fp64": (4096, 1.0e11), "int8": (6144, 6e12), "bf16": (16384, 2e14)}[kind]
    if family == "host":
        hi, most = min(hi, 6144), min(most, 2e13)
    slices = {"fp64": 0, "int8": rng.randint(3, 8), "bf16": rng.randint(3, 6)}[kind]
    while True:
        M, N, K = (_log_int(rng, 256, hi) for _ in range(3))
        if rng.random() < 0.5:                       # half of them round sizes
            M, N, K = (max(256, 128 * round(v / 128)) for v in (M, N, K))
        c = dict(family=family, M=M, N=N, K=K, kind=kind, slices=slices,
                 layout=rng.choice(("block", "block", "block", "cyclic")),
                 dist=rng.choice(("uniform", "wide", "normal_spiked")))
        if _flops(c) <= most:
            break
    if family == "gemm" and rng.random() < 0.4:
        c.update(AUTO)
        return c
    # a grid of one or two sub-tiles per block, with an even number of rows;
    # groups of one, of 2 x 1 or of 2 x 2 processors
    tm, tn, b = TILE[kind]
    fm, fn = rng.randint(1, 2), rng.randint(1, 2)
    P, Q = -(-M // (fm * tm)), -(-N // (fn * tn))
    P += P % 2
    Q += Q % 2
    G = rng.choice((P * Q, P * Q // 2, P * Q // 4))
    c.update(P=P, Q=Q, G=G, b=b, Bouter=b * rng.choice((4, 16)))
    return c


def _matrix(rows, cols, gen, dist):
    u = torch.empty((rows, cols), dtype=torch.float64, device="cuda")
    if dist == "normal_spiked":
        u.normal_(generator=gen)
        n = int(round(0.01 * cols))
        if n:
            u[:, torch.randperm(cols, generator=gen, device="cuda")[:n]] *= 1e6
        return u
    u.uniform_(-1.0, 1.0, generator=gen)
    if dist == "wide":
        e = torch.randint(-20, 21, (rows, cols), generator=gen, device="cuda")
        u = torch.ldexp(u, e)
    return u


def _operands(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    A = _matrix(case["M"], case["K"], gen, case["dist"])
    B = _matrix(case["K"], case["N"], gen,
                "uniform" if case["dist"] == "normal_spiked" else case["dist"])
    return A, B


def _training(case, seed):
    """Standardised features and targets, weights of a network part-way through
    its training and the moments that go with them (binary32)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = case["batch"]
    X = torch.randn((n, 10), generator=gen, device="cuda")
    y = torch.randn(n, generator=gen, device="cuda")
    parts = []
    for fan_in, fan_out in ((10, 64), (64, 64), (64, 64), (64, 1)):
        lim = math.sqrt(6.0 / (fan_in + fan_out))
        parts.append(torch.empty(fan_in * fan_out, device="cuda").uniform_(-lim, lim,
                                                                           generator=gen))
        parts.append(torch.empty(fan_out, device="cuda").uniform_(-0.1, 0.1, generator=gen))
    theta = torch.cat(parts)
    m = torch.randn(theta.numel(), generator=gen, device="cuda") * 1e-3
    v = torch.rand(theta.numel(), generator=gen, device="cuda") * 1e-4 + 1e-4
    return X, y, theta, m, v


def prepare(case, seed):
    hs.init(0)
    if case["family"] == "train":
        X, y, theta, m, v = _training(case, seed)
        return dict(case=case, X=X, y=y, theta=theta, m=m, v=v, grad=torch.empty_like(theta),
                    loss=torch.empty(1, device="cuda"))
    A, B = _operands(case, seed)
    state = dict(case=case, kw={k: case[k] for k in
                                ("P", "Q", "G", "b", "Bouter", "kind", "slices", "layout")})
    if case["family"] == "host":
        state["A"] = A.cpu().pin_memory()
        state["B"] = B.cpu().pin_memory()
        state["C"] = torch.empty((case["M"], case["N"]), dtype=torch.float64).pin_memory()
    else:
        state["A"], state["B"] = A, B
        state["C"] = torch.empty((case["M"], case["N"]), dtype=torch.float64, device="cuda")
    return state


def run(state):
    case = state["case"]
    if case["family"] == "train":
        s, lib = state, hs.lib()
        stream = torch.cuda.current_stream().cuda_stream
        st = lib.hsumma_mlp_backward(case["batch"], s["theta"].data_ptr(), s["X"].data_ptr(),
                                     s["y"].data_ptr(), s["grad"].data_ptr(),
                                     s["loss"].data_ptr(), stream)
        if st == 0:
            st = lib.hsumma_mlp_adam(hs.N_MLP_PARAMS, s["theta"].data_ptr(),
                                     s["grad"].data_ptr(), s["m"].data_ptr(), s["v"].data_ptr(),
                                     TRAIN_STEP, 1e-3, 0.9, 0.999, 1e-8, stream)
        if st != 0:
            raise RuntimeError(hs.last_error())
        return dict(grad=s["grad"], loss=s["loss"], theta=s["theta"], m=s["m"], v=s["v"])
    if case["family"] == "host":
        return hs.gemm_host(state["A"], state["B"], state["C"], **state["kw"])
    return hs.gemm(state["A"], state["B"], out=state["C"], **state["kw"])


def work(case):
    if case["family"] == "train":
        n, p = case["batch"], hs.N_MLP_PARAMS
        # forward, and the two products per layer of the backward pass; samples
        # and targets read, parameters and both moments read and written
        return {"bytes": 4.0 * (11 * n + 7 * p + 1), "flops": 6.0 * n * p}
    M, N, K = case["M"], case["N"], case["K"]
    return {"bytes": 8.0 * (M * K + K * N + M * N), "flops": _flops(case)}


def _exact_training(case, seed):
    X, y, theta, m, v = (t.double() for t in _training(case, seed))
    theta = theta.requires_grad_(True)
    h, o = X, 0
    for layer, (fi, fo) in enumerate(((10, 64), (64, 64), (64, 64), (64, 1))):
        h = h @ theta[o:o + fi * fo].view(fo, fi).T + theta[o + fi * fo:o + fi * fo + fo]
        o += fi * fo + fo
        if layer < 3:
            h = torch.nn.functional.gelu(h)
    loss = ((h[:, 0] - y) ** 2).mean()
    (g,) = torch.autograd.grad(loss, theta)
    lr, b1, b2, eps = (float(torch.tensor(x, dtype=torch.float32))
                       for x in (1e-3, 0.9, 0.999, 1e-8))
    m = b1 * m + (1 - b1) * g
    v = b2 * v + (1 - b2) * g * g
    step = lr * (m / (1 - b1 ** TRAIN_STEP)) / ((v / (1 - b2 ** TRAIN_STEP)).sqrt() + eps)
    return dict(grad=g, loss=loss.detach().view(1), theta=(theta - step).detach(), m=m, v=v)


def exact(case, seed):
    if case["family"] == "train":
        return _exact_training(case, seed)
    if 2.0 * case["M"] * case["N"] * case["K"] > 1e13:   # about ten seconds in binary64
        return None
    A, B = _operands(case, seed)
    return A @ B
