"""The work that users of this library have it do, as timed cases.

Five kinds, all through the package's public entry points (``NitiTrainer`` and the layer calls of ``Niti``):

``train``  one integer training step of a network: weights restored from their snapshot, forward, integer loss,
           backward with the weight update; captured into a CUDA graph (``NitiTrainer.capture``) or launched eagerly.
``gemm``   the fused multiply of one fully connected layer: forward, with ``both`` its backward call too.
``head``   a classification head: forward, integer cross-entropy, backward.
``conv``   one convolution layer: forward and weight gradient, and the error below it unless it is a first layer.

Every output is whole numbers, so results have to be equal.  ``listed()`` holds the networks and the layers of the
paper's workloads plus ragged ones; ``draw()`` gives more of the same ranges."""
import math

import torch

from paper_2009_13108_b200 import Niti, NitiTrainer
from synth.workloads import Net, config_net, he_like_exponent


def listed():
    return [
        # The MNIST-shaped MLP 784-256-256-10 at batch 64: the smallest step, launches and latency.
        {"name": "mlp_784_256_256_10_b64", "kind": "train", "net": "mlp", "batch": 64, "inp": 784, "hidden": 256,
         "depth": 2, "classes": 10, "round_mode": 0, "m_u": 5, "graph": True},
        # The MNIST-shaped CNN at batch 256, launched call by call as a first training loop does it.
        {"name": "mnist_cnn_b256_eager", "kind": "train", "net": "mnist", "batch": 256, "round_mode": 0, "m_u": 5,
         "graph": False},
        # The CIFAR-shaped VGG-11 at batch 256.
        {"name": "cifar_vgg11_b256", "kind": "train", "net": "vgg11", "batch": 256, "round_mode": 0, "m_u": 5,
         "graph": True},
        # The ImageNet-shaped VGG-16 at batch 64, 224 x 224: the largest step (the default benchmark).
        {"name": "imagenet_vgg16_b64", "kind": "train", "net": "vgg16", "batch": 64, "round_mode": 0, "m_u": 5,
         "graph": True},
        # A user's own CNN: batch, image side, channel counts and classes that are no powers of two, with
        # round-to-nearest and 3-bit gradients, the setting of the paper's accuracy runs.
        {"name": "cnn_ragged_b100_nearest", "kind": "train", "net": "cnn", "batch": 100, "side": 36, "cin": 3,
         "c1": 48, "c2": 96, "c3": 160, "fc": 200, "classes": 100, "round_mode": 1, "m_u": 3, "graph": True},
        # The fused multiply alone: the smallest point of the benchmark's sweep (one call, latency) ...
        {"name": "gemm_256", "kind": "gemm", "m": 256, "n": 256, "k": 256, "relu": False, "round_mode": 0, "m_u": 5,
         "both": False},
        # ... and the largest, in both directions.
        {"name": "gemm_8192_both", "kind": "gemm", "m": 8192, "n": 8192, "k": 8192, "relu": True, "round_mode": 0,
         "m_u": 5, "both": True},
        # A classification head over a large batch with 1000 classes.
        {"name": "head_4096x1000x512", "kind": "head", "batch": 4096, "classes": 1000, "k": 512, "round_mode": 0,
         "m_u": 5},
        # The paper's timed layer (batch 64, 64 -> 128 channels, 3 x 3) at a middle size of its table.
        {"name": "conv3x3_64to128_56_b64", "kind": "conv", "batch": 64, "side": 56, "cin": 64, "cout": 128, "r": 3,
         "pad": 1, "stride": 1, "first": False, "round_mode": 0, "m_u": 5},
        # The first layer of the paper's AlexNet: 11 x 11, stride 4, on RGB images.
        {"name": "conv11x11s4_rgb_224_b64", "kind": "conv", "batch": 64, "side": 224, "cin": 3, "cout": 96, "r": 11,
         "pad": 2, "stride": 4, "first": True, "round_mode": 0, "m_u": 5},
        # A 5 x 5 layer of such a network: odd image side, channel counts that are not powers of two.
        {"name": "conv5x5_96to256_27_b128", "kind": "conv", "batch": 128, "side": 27, "cin": 96, "cout": 256, "r": 5,
         "pad": 2, "stride": 1, "first": False, "round_mode": 0, "m_u": 5},
        # A downsampling 3 x 3 layer with stride 2, as networks without pooling use it.
        {"name": "conv3x3s2_128to256_56_b64", "kind": "conv", "batch": 64, "side": 56, "cin": 128, "cout": 256, "r": 3,
         "pad": 1, "stride": 2, "first": False, "round_mode": 0, "m_u": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes spread over the logarithm of their range; a case above the bound is drawn again."""
    kind = rng.choice(["mlp", "cnn", "gemm", "head", "conv", "conv"])
    opt = {"round_mode": rng.choice([0, 0, 1]), "m_u": rng.choice([5, 5, 4, 3])}
    while True:
        if kind == "mlp":
            case = {"kind": "train", "net": "mlp", "batch": _log_int(rng, 16, 1024), "inp": _log_int(rng, 64, 3072),
                    "hidden": _log_int(rng, 64, 2048), "depth": rng.choice([1, 2, 2, 3]),
                    "classes": rng.choice([10, 10, 37, 100, 1000]), "graph": rng.random() < 0.7}
        elif kind == "cnn":
            c1 = rng.choice([16, 24, 32, 48, 64])
            case = {"kind": "train", "net": "cnn", "batch": _log_int(rng, 16, 256), "side": rng.choice([28, 32, 36, 40, 48, 64]),
                    "cin": rng.choice([1, 3]), "c1": c1, "c2": rng.choice([32, 64, 72, 96, 128]),
                    "c3": rng.choice([64, 96, 128, 160, 256]), "fc": _log_int(rng, 64, 1024),
                    "classes": rng.choice([10, 10, 100, 1000]), "graph": rng.random() < 0.7}
        elif kind == "gemm":
            case = {"kind": "gemm", "m": _log_int(rng, 64, 8192), "n": _log_int(rng, 64, 8192), "k": _log_int(rng, 64, 8192),
                    "relu": rng.random() < 0.5, "both": rng.random() < 0.5}
            if rng.random() < 0.5:                    # half of them at the multiples of 64 that layer widths usually are
                for d in ("m", "n", "k"):
                    case[d] = (case[d] + 63) // 64 * 64
        elif kind == "head":
            case = {"kind": "head", "batch": _log_int(rng, 64, 8192), "classes": rng.choice([10, 100, 257, 1000, 2000]),
                    "k": _log_int(rng, 64, 4096)}
        else:
            first = rng.random() < 0.25
            if first:                                 # image networks' first layers
                cin, (r, pad, stride) = rng.choice([1, 3, 3]), rng.choice([(3, 1, 1), (5, 2, 1), (5, 0, 1), (7, 3, 2), (11, 2, 4)])
                side = _log_int(rng, 28, 224 if stride > 1 else 160)
            else:
                cin, (r, pad, stride) = rng.choice([16, 32, 48, 64, 96, 128, 192, 256, 384, 512]), rng.choice(
                    [(3, 1, 1), (3, 1, 1), (3, 1, 2), (5, 2, 1), (1, 0, 1), (1, 0, 2)])
                side = _log_int(rng, 7, 112)
            case = {"kind": "conv", "batch": _log_int(rng, 8, 128), "side": side, "cin": cin,
                    "cout": rng.choice([16, 32, 48, 64, 96, 128, 192, 256, 384, 512]), "r": r, "pad": pad,
                    "stride": stride, "first": first}
        case.update(opt)
        w = work(case)
        if w["bytes"] <= 400e6 and w["flops"] <= (1.1e12 if kind in ("gemm", "head") else 0.3e12):
            return case


def _net(case):
    """The network of a ``train`` case: the repository's configurations, or one of the same make with other sizes."""
    kind, batch = case["net"], case["batch"]
    if kind in ("mnist", "vgg11", "vgg16"):
        net = config_net({"mnist": 2, "vgg11": 3, "vgg16": 4}[kind], batch=batch)
    elif kind == "mlp":
        sizes = [case["inp"]] + [case["hidden"]] * case["depth"] + [case["classes"]]
        net = Net("mlp", batch, (sizes[0],), case["classes"], -7, 0)
        net.layers = [{"op": "fc", "k": k, "n": n, "relu": i < case["depth"], "s_w": he_like_exponent(k)}
                      for i, (k, n) in enumerate(zip(sizes, sizes[1:]))]
    else:
        side, c = case["side"], [case["cin"], case["c1"], case["c2"], case["c3"]]
        net = Net("cnn", batch, (side, side, c[0]), case["classes"], -7, 0)
        conv = lambda i: {"op": "conv", "cin": c[i], "cout": c[i + 1], "relu": True,  # noqa: E731
                          "s_w": he_like_exponent(9 * c[i])}
        k = (side // 4) * (side // 4) * c[3]
        net.layers = [conv(0), conv(1), {"op": "pool"}, conv(2), {"op": "pool"},
                      {"op": "fc", "k": k, "n": case["fc"], "relu": True, "s_w": he_like_exponent(k)},
                      {"op": "fc", "k": case["fc"], "n": case["classes"], "relu": False, "s_w": he_like_exponent(case["fc"])}]
    net.m_u = case["m_u"]
    return net


class _Make:
    """Seeded int8 tensors on the GPU with the values the path meets."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def uniform(self, *shape):                        # images and weights: uniform over [-127, 127]
        return torch.randint(-127, 128, shape, generator=self.g, dtype=torch.int8, device="cuda")

    def error(self, *shape):                          # errors: bell-shaped, sigma about 32
        return (torch.randn(shape, generator=self.g, device="cuda") * 32).round_().clamp_(-127, 127).to(torch.int8)

    def act(self, *shape):                            # activations behind a ReLU: half of them zero
        return self.error(*shape).clamp_(min=0)

    def labels(self, n, classes):
        return torch.randint(0, classes, (n,), generator=self.g, dtype=torch.int32, device="cuda")


def _conv_out(case):
    return (case["side"] + 2 * case["pad"] - case["r"]) // case["stride"] + 1


def prepare(case, seed):
    mk, n = _Make(seed), Niti(0)
    st = {"case": case, "n": n}
    i8 = lambda *shape: torch.empty(shape, dtype=torch.int8, device="cuda")  # noqa: E731
    if case["kind"] == "train":
        net = _net(case)
        weights = []
        for L in net.layers:
            if L["op"] == "conv":
                weights.append(mk.uniform(L["cout"], 3, 3, L["cin"]))
            elif L["op"] == "fc":
                weights.append(mk.uniform(L["n"], L["k"]))
        tr = NitiTrainer(n, net, weights, round_mode=case["round_mode"])
        tr.load_batch(mk.uniform(net.batch, *net.in_shape), mk.labels(net.batch, net.n_classes))
        tr.snapshot_weights()
        st["tr"] = tr
        if case["graph"]:
            tr.step()                                 # sizes the workspace and the kernels' attributes
            st["replay"] = tr.capture(with_reset=True)
        return st
    if case["kind"] == "conv":
        B, S, Ci, Co, So = case["batch"], case["side"], case["cin"], case["cout"], _conv_out(case)
        st["x"] = mk.uniform(B, S, S, Ci) if case["first"] else mk.act(B, S, S, Ci)
        st["w"] = mk.uniform(Co, case["r"], case["r"], Ci)
        st["e"] = mk.error(B, So, So, Co)
        st["y"], st["g"] = i8(B, So, So, Co), i8(Co, case["r"], case["r"], Ci)
        st["ep"] = None if case["first"] else i8(B, S, S, Ci)
        K = case["r"] * case["r"] * Ci
    else:
        head = case["kind"] == "head"
        M, K, N = (case["batch"], case["k"], case["classes"]) if head else (case["m"], case["k"], case["n"])
        st["x"], st["w"] = mk.act(M, K), mk.uniform(N, K)
        st["y"] = i8(M, N)
        if head:
            st["labels"], st["e"] = mk.labels(M, N), i8(M, N)
        elif case["both"]:
            st["e"] = mk.error(M, N)
        if head or case["both"]:
            st["ep"], st["g"] = i8(M, K), i8(N, K)
    st["s_x"], st["s_w"] = n.scalar(-7), n.scalar(he_like_exponent(K))
    st["s_y"], st["b_y"], st["b_e"], st["b_g"] = n.scalar(), n.scalar(), n.scalar(), n.scalar()
    st["b_loss"], st["hits"] = n.scalar(), n.scalar()
    return st


def run(st):
    case, n = st["case"], st["n"]
    mode, m_u = case["round_mode"], case["m_u"]
    if case["kind"] == "train":
        tr = st["tr"]
        if case["graph"]:
            st["replay"]()
        else:
            tr.reset_weights()
            tr.step()
        return {"weights": tr.weights, "logits": tr.acts[-1], "s_logits": tr.s_act[-1], "hits": tr.n_correct,
                "b_loss": tr.b_loss}
    if case["kind"] == "conv":
        pad, stride, x, e, w = case["pad"], case["stride"], st["x"], st["e"], st["w"]
        n.conv_fwd(x, st["s_x"], w, st["s_w"], y=st["y"], s_y=st["s_y"], b_y=st["b_y"], pad=pad, relu=True,
                   round_mode=mode, stride=stride)
        if not case["first"]:
            n.conv_dgrad(e, w, (case["side"], case["side"]), e_prev=st["ep"], relu_mask_src=x, b_e=st["b_e"], pad=pad,
                         round_mode=mode, stride=stride)
        n.conv_wgrad(x, e, (case["r"], case["r"]), g=st["g"], b_g=st["b_g"], pad=pad, m_u=m_u, round_mode=mode,
                     stride=stride)
        return {"y": st["y"], "s_y": st["s_y"], "b_y": st["b_y"], "e_prev": st["ep"], "b_e": st["b_e"], "g": st["g"],
                "b_g": st["b_g"]}
    head = case["kind"] == "head"
    n.linear_fwd(st["x"], st["s_x"], st["w"], st["s_w"], out=st["y"], s_out=st["s_y"], b_out=st["b_y"],
                 relu=not head and case["relu"], round_mode=mode)
    out = {"y": st["y"], "s_y": st["s_y"], "b_y": st["b_y"]}
    if head:
        n.int_xent(st["y"], st["s_y"], st["labels"], e=st["e"], b_e=st["b_loss"], n_correct=st["hits"], round_mode=mode)
        out.update(e=st["e"], b_loss=st["b_loss"], hits=st["hits"])
    if head or case["both"]:
        n.linear_bwd(st["x"], st["e"], st["w"], relu_mask_src=st["x"], e_prev=st["ep"], g=st["g"], b_e=st["b_e"],
                     b_g=st["b_g"], m_u=m_u, round_mode=mode)
        out.update(e_prev=st["ep"], b_e=st["b_e"], g=st["g"], b_g=st["b_g"])
    return out


def work(case):
    """Inputs read once, outputs written once; 2 int8 operations per multiply-accumulate."""
    if case["kind"] == "train":
        net = _net(case)
        inputs = net.batch * (math.prod(net.in_shape) + 4)
        return {"bytes": inputs + 2 * net.n_weights() + net.batch * net.n_classes, "flops": net.int8_ops_per_step()}
    if case["kind"] == "conv":
        B, S, Ci, Co, So, R = case["batch"], case["side"], case["cin"], case["cout"], _conv_out(case), case["r"]
        x, w, y = B * S * S * Ci, Co * R * R * Ci, B * So * So * Co
        passes = 2 if case["first"] else 3
        # x, w, e in; y, g and (unless a first layer) the error below out
        return {"bytes": x + w + y + y + w + (0 if case["first"] else x), "flops": passes * 2 * y * R * R * Ci}
    head = case["kind"] == "head"
    M, K, N = (case["batch"], case["k"], case["classes"]) if head else (case["m"], case["k"], case["n"])
    both = head or case["both"]
    moved = M * K + N * K + M * N                     # forward: a, w in, output out
    if head:
        moved += 4 * M + M * N                        # labels in, loss gradient out
    elif both:
        moved += M * N                                # error in
    if both:
        moved += M * K + N * K                        # error below and gradient out
    return {"bytes": moved, "flops": (3 if both else 1) * 2 * M * N * K}


def tolerance(case):
    return "exact"
