"""Timing cases of the codec: what a training program has it do, through its public entry points.

A case is a dict of plain values. `op` says which calls make up one pass:

  encode  one worker encodes its gradient (qsgd_encode)
  hook    the same for one layer's gradient, without a workspace (qsgd_encode_elias_static)
  decode  K received messages are decoded, summed and applied to the parameters in one call
          (qsgd_decode_sgd_step_packed: nothing is read back to the host between Encode and Decode)
  apart   the same as two calls (qsgd_decode_accumulate_packed, then qsgd_sgd_step)
  worker  one data-parallel iteration of one GPU: encode the own gradient, decode it and K - 1 others
  step    one iteration of K workers played by one GPU: K encodes, one decode
  policy  `worker` under the per-tensor policy (small tensors raw, buckets cut to the tensors)
  qsvrg   one iteration of the variance-reduced variant: K one-bucket vectors encoded, the offset tables
          built from the sizes on the device, one decode and step

Messages and parameters are compared bit for bit: every sum has a stated order.
"""
import math

import numpy as np
import torch

import paper_1610_02132_b200 as Q
from paper_1610_02132_b200 import inputs as I

NORM = {"l2": Q.NORM_L2, "max": Q.NORM_MAX}
CODE = {"fixed": Q.CODE_FIXED, "elias": Q.CODE_ELIAS, "dense": Q.CODE_ELIAS_DENSE}
SHAPES = {"alexnet": I.alexnet_shapes, "resnet152": I.resnet152_shapes}
ETA, PHILOX_SEED, ITERATION = 0.05, 7, 3


def listed():
    resnet = I.numel(I.resnet152_shapes())
    case = lambda name, op, n, d, s, norm, code, K, grad, **more: dict(
        name=name, op=op, n=n, d=d, s=s, norm=norm, code=code, K=K, grad=grad, **more)
    return [
        # the smallest calls: 16 KB vectors, eight encodes and a decode an iteration
        case("qsvrg_n4096_k8", "qsvrg", 4096, 4096, 64, "l2", "dense", 8, "gauss"),
        # a small layer group: a few messages of half a megabyte
        case("tiny_fixed_k4", "step", 2 ** 20, 512, 15, "l2", "fixed", 4, "gauss"),
        # a 512 x 512 x 3 x 3 convolution's gradient leaving from a gradient hook, 2-bit levels
        case("hook_conv512_2bit", "hook", 512 * 512 * 9, 128, 3, "l2", "elias", 1, "mixture"),
        # odd length, a bucket size that is no power of two, 8-bit levels, sum and step apart
        case("ragged_elias_8bit_k5", "apart", 1000003, 96, 255, "l2", "elias", 5, "gauss"),
        # the sparse regime (s = 1, long buckets): eight workers on one GPU
        case("sparse_elias_k8", "step", 2 ** 24, 4096, 1, "l2", "elias", 8, "laplace"),
        # the dense code at s = sqrt(d)
        case("dense_elias_k8", "worker", 2 ** 24, 4096, 64, "l2", "dense", 8, "gauss"),
        # a ResNet-152-shaped gradient with 4-bit levels, each direction and each code
        case("encode_fixed_resnet152", "encode", resnet, 512, 15, "l2", "fixed", 1, "mixture"),
        case("decode_fixed_resnet152_k16", "decode", resnet, 512, 15, "l2", "fixed", 16, "mixture"),
        case("encode_elias_resnet152", "encode", resnet, 512, 15, "l2", "elias", 1, "mixture"),
        case("decode_elias_resnet152_k16", "decode", resnet, 512, 15, "l2", "elias", 16, "mixture"),
        # AlexNet-shaped, 8-bit levels with max-norm scales, small tensors raw
        case("policy_alexnet_8bit_k16", "policy", I.numel(I.alexnet_shapes()), 512, 255, "max", "fixed", 16, "gauss",
             model="alexnet"),
        # the largest: a gibibyte of gradient from sixteen workers
        case("sweep_elias_2e28_k16", "apart", 2 ** 28, 512, 15, "l2", "elias", 16, "gauss"),
    ]


def draw(rng):
    op = rng.choice(["encode", "encode", "hook", "decode", "decode", "apart", "worker", "worker", "step", "policy", "qsvrg"])
    K = 1 if op in ("encode", "hook") else rng.choice([2, 3, 4, 5, 8, 8, 16, 16, 32])
    if op == "qsvrg":
        n = 32 * rng.randint(8, 128)
        return dict(op=op, n=n, d=n, s=min(math.isqrt(n), 255), norm="l2", code=rng.choice(["dense", "dense", "elias", "fixed"]),
                    K=min(K, 8), grad="gauss")
    most = min(2.0 ** 26, 2.0 ** 28 / K)
    n = int(math.exp(rng.uniform(math.log(2.0 ** 13), math.log(most))))
    d = rng.choice([64, 128, 128, 256, 512, 512, 512, 1024, 4096, 32 * rng.randint(1, 128)])
    n -= rng.choice([0, n % d, n % 4, n % 4096])            # odd lengths, whole buckets, whole tiles
    s = rng.choice([1, 3, 3, 7, 15, 15, 15, 255, 255, min(math.isqrt(d), 255)])
    case = dict(op=op, n=max(n, 1), d=d, s=s, norm=rng.choice(["l2", "max"]), K=K,
                code="elias" if op == "hook" else rng.choice(["fixed", "fixed", "fixed", "elias", "elias", "elias", "dense"]),
                grad=rng.choice(["gauss", "mixture", "laplace"]))
    if op == "hook":
        case["n"] = min(case["n"], 2 ** 23 - n % 32)         # what the built-in scratch holds at every bucket size
    if op == "step":
        case["K"] = min(K, 16)                               # one GPU plays no more workers than that
    if op == "policy":
        case["model"] = rng.choice(["alexnet", "resnet152"])
        case["n"] = I.numel(SHAPES[case["model"]]())
        case["K"] = min(K, 4)
        if case["d"] % 128:
            case["d"] = 512
    return case


# ------------------------------------ what a program has in hand ------------------------------------
def gradient(case, seed):
    if case["grad"] == "laplace":
        return I.sparse_laplace_device(case["n"], 1e-3, 0.3, seed=seed)
    if case["grad"] == "mixture":
        return I.gaussian_mixture_device(case["n"], seed=seed)
    return I.gaussian_device(case["n"], 0.01, seed=seed)


def plan_of(case):
    if case["op"] != "policy":
        return None
    return Q.Policy([math.prod(t) for t in SHAPES[case["model"]]()], case["d"])


def buffers(case, plan):
    """Message, info words and workspace of one sender. Messages are compared whole, so the bytes behind
    a message shorter than its buffer start out as zeros."""
    n, d, s, code = case["n"], case["d"], case["s"], CODE[case["code"]]
    cap = Q.qsgd_policy_message_capacity(plan, s, code) if plan else Q.qsgd_message_capacity(n, d, s, code)
    scratch = Q.qsgd_policy_workspace_bytes(plan, s, code) if plan else Q.qsgd_workspace_bytes(n, d, s, code)
    if case["op"] == "hook":
        scratch = 0
    return {"out": torch.zeros(cap, dtype=torch.uint8, device="cuda"),
            "info": torch.zeros(4, dtype=torch.int64, device="cuda"),
            "ws": torch.empty(max(scratch, 16), dtype=torch.uint8, device="cuda")}


def encode(case, plan, g, buf, worker, status):
    d, s, norm, code = case["d"], case["s"], NORM[case["norm"]], CODE[case["code"]]
    if plan:
        Q.qsgd_policy_encode(g, plan, s, norm, code, PHILOX_SEED, ITERATION, worker, buf["out"], buf["info"], buf["ws"], status)
    elif case["op"] == "hook":
        Q.qsgd_encode_elias_static(g, d, s, norm, code, PHILOX_SEED, ITERATION, worker, buf["out"], buf["info"], status)
    else:
        Q.qsgd_encode(g, d, s, norm, code, PHILOX_SEED, ITERATION, worker, buf["out"], buf["info"], buf["ws"], status)


def received(case, plan, seed, workers, status):
    """The messages of other workers as an exchange delivers them: cut to their length."""
    msgs, infos, tables = [], [], []
    buf = buffers(case, plan)
    B = plan.n_buckets if plan else -(-case["n"] // case["d"])
    for w in workers:
        encode(case, plan, gradient(case, 1000 * seed + w), buf, w, status)
        info = [int(v) for v in buf["info"].tolist()]
        m = torch.zeros(info[2] + 16, dtype=torch.uint8, device="cuda")
        m[: info[2]] = buf["out"][: info[2]]
        msgs.append(m)
        infos.append(buf["info"].clone())
        if info[1]:
            tables.append(m[info[1]: info[1] + 8 * (B + 1)].view(torch.int64))
    return msgs, infos, tables or None


def prepare(case, seed):
    op, K, n = case["op"], case["K"], case["n"]
    plan, status = plan_of(case), Q.new_status()
    st = {"case": case, "plan": plan, "status": status}
    sent = {"step": K, "qsvrg": K, "decode": 0, "apart": 0}.get(op, 1)       # gradients that this GPU encodes in a pass
    st["grads"] = [gradient(case, 1000 * seed + w) for w in range(sent)]
    st["own"] = [buffers(case, plan) for _ in range(sent)]
    if op in ("step", "qsvrg"):
        for b in st["own"]:
            b["ws"] = st["own"][0]["ws"]                     # one after the other on one stream: one workspace
    if op == "qsvrg":
        st["info"] = torch.zeros(K, 4, dtype=torch.int64, device="cuda")
        for b, row in zip(st["own"], st["info"]):
            b["info"] = row
        st["tables"] = torch.zeros(K, 2, dtype=torch.int64, device="cuda")
    if op in ("decode", "apart", "policy"):
        st["msgs"], st["infos"], st["offsets"] = received(case, plan, seed, range(K), status)
    elif op == "worker":
        msgs, infos, _ = received(case, plan, seed, range(1, K), status)
        st["msgs"], st["infos"] = [st["own"][0]["out"]] + msgs, [st["own"][0]["info"]] + infos
    elif op == "step":
        st["msgs"], st["infos"] = [b["out"] for b in st["own"]], [b["info"] for b in st["own"]]
    elif op == "qsvrg":
        st["msgs"] = [b["out"] for b in st["own"]]
    if op not in ("encode", "hook"):
        st["x"] = I.gaussian_device(n, 1.0, seed=1000 * seed + 999)
    if op == "apart":
        st["acc"] = torch.zeros(n, dtype=torch.float32, device="cuda")
    return st


# ---------------------------------------- one pass ---------------------------------------------------
def run(st):
    case, plan, status = st["case"], st["plan"], st["status"]
    op, n, d, s, K, code = case["op"], case["n"], case["d"], case["s"], case["K"], CODE[case["code"]]
    for w, (g, buf) in enumerate(zip(st["grads"], st["own"])):
        encode(case, plan, g, buf, w, status)
    out = {"messages": [b["out"] for b in st["own"]], "infos": [b["info"] for b in st["own"]], "status": status}
    if op in ("decode", "worker", "step"):
        Q.qsgd_decode_sgd_step_packed(st["msgs"], st["infos"], n, d, s, code, st["x"], ETA, status)
    elif op == "apart":
        Q.qsgd_decode_accumulate_packed(st["msgs"], st["infos"], n, d, s, code, st["acc"], status)
        Q.qsgd_sgd_step(st["x"], st["acc"], ETA, K)
        out["acc"] = st["acc"]
    elif op == "policy":
        Q.qsgd_policy_decode_sgd_step(st["msgs"], st["offsets"], plan, s, code, st["x"], ETA, status)
    elif op == "qsvrg":
        tables = None
        if code != Q.CODE_FIXED:
            st["tables"][:, 1] = st["info"][:, 0]
            tables = [st["tables"][w] for w in range(K)]
        Q.qsgd_decode_sgd_step(st["msgs"], tables, n, d, s, code, st["x"], ETA, status)
    if "x" in st:
        out["x"] = st["x"]
    return out


# ---------------------------------------- what it needs ----------------------------------------------
def elias_len(k):
    bits = 1
    while k > 1:
        bits += k.bit_length()
        k = k.bit_length() - 1
    return bits


def message_bytes(case):
    """Expected bytes of one message: exact for the fixed-width code, the mean over a few drawn buckets
    for the Elias codes."""
    n, d, s = case["n"], case["d"], case["s"]
    B = -(-n // d)
    if case["code"] == "fixed":
        return Q.qsgd_fixed_layout(n, d, s)[2]
    r = np.random.default_rng(1)
    lens = [elias_len(k) if k else 0 for k in range(max(d, 256) + 2)]
    bits, buckets = 0, 8
    for _ in range(buckets):
        v = r.standard_normal(d)
        if case["grad"] == "mixture":
            v *= np.where(r.random(d) < 0.9, 1e-2, 1.0)
        elif case["grad"] == "laplace":
            v = r.laplace(0.0, 1.0, d) * (r.random(d) >= 0.3)
        a = np.linalg.norm(v) if case["norm"] == "l2" else np.abs(v).max()
        level = np.minimum(np.floor(s * np.abs(v) / a + r.random(d)), s).astype(int)
        if case["code"] == "dense":
            bits += sum(1 + lens[k + 1] for k in level)
        else:
            at = np.flatnonzero(level)
            bits += sum(lens[k] for k in np.diff(at, prepend=-1)) + sum(1 + lens[k] for k in level[at])
    return int((32 * B + bits / buckets / d * n) / 8) + 8 * (B + 1)


def work(case):
    """Each gradient, message and parameter read once, each message and parameter written once."""
    op, n, K, m = case["op"], case["n"], case["K"], message_bytes(case)
    sent = {"step": K, "qsvrg": K, "decode": 0, "apart": 0}.get(op, 1)
    total = sent * (4 * n + m)
    if op not in ("encode", "hook"):
        total += K * m + 8 * n
    if op == "apart":
        total += 8 * n                                       # the sum is asked for by itself: written, then read
    return {"bytes": total, "flops": 0}


def tolerance(case):
    return "exact"
