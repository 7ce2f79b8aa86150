"""The work that users have this library do, as cases that can be timed and compared.

A case is a dict of plain values.  Its "path" names the public entry points that it goes through:

  step        one train step on device buffers (revnet_train_step)
  step_host   one train step fed from pinned host memory, loss read back (revnet_train_step_host)
  block_fwd   inference through one reversible block: weights packed once, float state (revnet_block_fwd)
  block_train one block in training: weight packs, forward in place, reconstructing backward in place
              (revnet_pack_weights, revnet_block_fwd, revnet_block_bwd)
  transition  one stored BN-ReLU-conv layer, forward and backward (revnet_transition_fwd / _bwd)

Networks are those of paper_1707_04585_b200.synthetic; inputs have the distributions described there
(images and activations ~N(0,1), labels uniform, Kaiming-normal weights, gamma ~N(1,0.1), beta ~N(0,0.1),
the last BN of a residual branch scaled down), drawn on the GPU from the seed.
"""
import math
from dataclasses import replace

import torch

from paper_1707_04585_b200 import binding as B
from paper_1707_04585_b200 import runner as R
from paper_1707_04585_b200 import synthetic as syn

CIFAR_NETS = ("revnet38", "revnet110", "revnet164", "paper_revnet38", "paper_revnet110", "paper_revnet164")

# Scale of the last BN of every residual function: branches small beside their skip paths, as in trained residual networks
# and after the customary small initialisation of that gamma.  (With all gammas at 1 a deep stack at random weights amplifies
# the last bit of any sum to per cents of its logits, and two correct implementations could not be told from a wrong one.)
GAMMA_LAST = 0.1
LR = 0.01          # the warm-up rate customary for the deep CIFAR networks

_ctx = None


def context():
    """One library context per process, as a program keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = B.Context(0)
    return _ctx


# ------------------------------------------------------------------ the cases
def _step(name, net, batch, img, mode=0, stored=False, path="step"):
    return dict(name=name, path=path, net=net, batch=batch, img=img, mode=mode, stored=stored)


def _block(name, path, kind, n, h, w, c, width, mode=0):
    return dict(name=name, path=path, kind=kind, n=n, h=h, w=w, c=c, width=width, mode=mode)


def _trans(name, n, h, cin, cout, k, stride, split, mode=0):
    return dict(name=name, path="transition", n=n, h=h, cin=cin, cout=cout, k=k, stride=stride, split=split, mode=mode)


def listed():
    return [
        # the smallest call: one layer per function on a few pixels, as in unit-level inference; launches and host work count
        _block("block_fwd_tiny", "block_fwd", "single", 4, 8, 8, 8, 0),
        # a first-stage unit of the large-image network at its training batch, forward only
        _block("block_fwd_image", "block_fwd", "bottleneck", 64, 56, 56, 512, 128),
        # a first-stage unit of the CIFAR-sized networks, driven by a user's own training loop
        _block("block_train_cifar", "block_train", "basic", 128, 32, 32, 16, 0),
        # the same on a ragged shape: odd batch, rows that do not divide the pixel tiles
        _block("block_train_odd", "block_train", "basic", 37, 15, 21, 24, 0),
        # a stored down-sampling layer of the large-image network, reduced batch
        _trans("transition_image", 48, 28, 2048, 4096, 3, 2, True),
        # the train step of the four networks at their training batch
        _step("step_revnet38", "revnet38", 128, 32),
        _step("step_revnet110", "revnet110", 128, 32),
        _step("step_revnet164", "revnet164", 128, 32),
        _step("step_revnet104", "revnet104", 64, 224),
        # fed from the host with the last, smaller batch of an epoch (50000 mod 128), paper-shaped network
        _step("step_host_paper38", "paper_revnet38", 80, 32, path="step_host"),
        # single-precision training of the smallest network
        _step("step_revnet38_fp32", "revnet38", 128, 32, mode=1),
        # activations kept (ordinary backprop), smaller images, odd batch
        _step("step_revnet104_stored", "revnet104", 23, 160, stored=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(case):
    """Seconds a pass may take at worst: keeps drawn cases below the largest listed one."""
    w = work(case)
    return w["flops"] / (3e12 if case["mode"] == 1 else 2e14) + w["bytes"] / 1e12


def draw(rng):
    limit = 0.3 * _cost(_step("", "revnet104", 64, 224))
    while True:
        c = _draw(rng)
        if _cost(c) <= limit:
            return c


def _draw(rng):
    path = rng.choice(("step", "step", "step", "step_host", "block_fwd", "block_fwd", "block_train", "block_train", "transition"))
    mode = 1 if rng.random() < 0.15 else 0
    if path in ("step", "step_host"):
        if mode == 0 and rng.random() < 0.3:
            net, batch, img = "revnet104", _log_int(rng, 8, 64), 32 * rng.randint(4, 7)
        else:
            net, batch, img = rng.choice(CIFAR_NETS), _log_int(rng, 16, 256), 32
        c = _step("", net, batch, img, mode, path == "step" and rng.random() < 0.25, path)
    elif path == "block_fwd":
        kind = rng.choice(("single", "basic", "bottleneck"))
        n, h, w = _log_int(rng, 1, 128), rng.randint(4, 56), rng.randint(4, 56)
        width = 8 * _log_int(rng, 2, 64) if kind == "bottleneck" else 0
        c = _block("", path, kind, n, h, w, 4 * width if width else 8 * _log_int(rng, 1, 16), width, mode)
    elif path == "block_train":
        n, h, w = _log_int(rng, 8, 128), rng.randint(7, 32), rng.randint(7, 32)
        c = _block("", path, rng.choice(("single", "basic")), n, h, w, 8 * rng.randint(1, 8), 0, mode)
    else:
        stride = rng.choice((1, 2, 2))
        c = _trans("", _log_int(rng, 4, 128), 2 * rng.randint(3, 28), 16 * _log_int(rng, 2, 128), 16 * _log_int(rng, 4, 256),
                   3, stride, stride == 2, mode)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs and what a program keeps
class _Draws:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda")

    def labels(self, n, classes):
        return torch.randint(0, classes, (n,), generator=self.g, device="cuda", dtype=torch.int32)


def _config(case):
    return replace(syn.stack_config(case["net"]), N=case["batch"], img=case["img"], lr=LR)


def _role_scale(shape, role):
    """(standard deviation, mean) of a parameter tensor."""
    if role == "convw":
        return math.sqrt(2.0 / (shape[1] * shape[2] * shape[3])), 0.0
    if role == "fcw":
        return math.sqrt(2.0 / shape[1]), 0.0
    return {"gamma": (0.1, 1.0), "beta": (0.1, 0.0), "fcb": (0.0, 0.0)}[role]


def _branch_end(name, cfg):
    """Whether a parameter belongs to the last layer of a residual function of a reversible unit (a down-sampling unit's
    functions are the only source of its new channels and keep their scale)."""
    part = name.split(".")
    return len(part) == 5 and part[1] != "d" and part[3] == {"single": "l0", "basic": "l1", "bottleneck": "l2"}[cfg.stages[int(part[0][1:])].kind]


def _fn_params(d, kind, c, width):
    out = []
    for cin, cout, k in syn.fn_layers(kind, c, width):
        out.append(dict(W=d.normal(cout, k, k, cin) * math.sqrt(2.0 / (cin * k * k)),
                        gamma=1.0 + 0.1 * d.normal(cin), beta=0.1 * d.normal(cin)))
    out[-1]["gamma"] *= GAMMA_LAST
    out[-1]["beta"] *= GAMMA_LAST
    return out


def _grad_like(layers):
    return [{k: torch.zeros_like(v) for k, v in l.items()} for l in layers]


def _prepare_step(case, d):
    cfg = _config(case)
    r = R.StackRunner(context(), cfg, case["mode"], store_activations=case["stored"])
    r.params.normal_(generator=d.g)
    at = 0
    for name, shape, role in r.specs:
        n = math.prod(shape)
        std, mean = _role_scale(shape, role)
        if role in ("gamma", "beta") and _branch_end(name, cfg):
            std, mean = std * GAMMA_LAST, mean * GAMMA_LAST
        r.params[at:at + n].mul_(std).add_(mean)
        at += n
    r.images.normal_(generator=d.g)
    r.labels.copy_(d.labels(cfg.N, cfg.n_classes))
    s = dict(case=case, run=r)
    if case["path"] == "step_host":
        s["images_host"] = r.images.cpu().pin_memory()
        s["labels_host"] = r.labels.cpu().pin_memory()
        s["loss_host"] = torch.zeros(1).pin_memory()
        s["pred_host"] = torch.zeros(cfg.N, dtype=torch.int32).pin_memory()
    return s


def _prepare_block(case, d):
    ctx = context()
    train = case["path"] == "block_train"
    # training runs on the mode's own state format (fixed point in the bf16 mode); inference needs no reversal: float state
    frac = R.DEFAULT_FRAC_BITS[case["mode"]] if train else 0
    b = syn.BlockCfg(case["n"], case["h"], case["w"], case["c"], case["width"], case["kind"], seed=0)
    desc = B.block_desc(b, case["mode"], frac)
    fwd, bwd = B.revnet_block_workspace_bytes(ctx, desc)
    shape = (b.N, b.H, b.W, b.c)
    s = dict(case=case, desc=desc, F=_fn_params(d, b.kind, b.c, b.w), G=_fn_params(d, b.kind, b.c, b.w),
             x1=d.normal(*shape), x2=d.normal(*shape),
             packs=torch.empty(max(B.revnet_block_pack_bytes(ctx, desc), 256), dtype=torch.uint8, device="cuda"),
             ws=torch.empty(max(fwd, bwd if train else 0), dtype=torch.uint8, device="cuda"))
    if train:
        if frac:
            s["x1"], s["x2"] = (torch.round(x * 2.0 ** frac).to(torch.int32) for x in (s["x1"], s["x2"]))
        s["dy1"], s["dy2"] = d.normal(*shape), d.normal(*shape)
        s["dx1"], s["dx2"] = torch.empty_like(s["dy1"]), torch.empty_like(s["dy2"])
        s["gF"], s["gG"] = _grad_like(s["F"]), _grad_like(s["G"])
    else:
        s["y1"], s["y2"] = torch.empty_like(s["x1"]), torch.empty_like(s["x2"])
        B.revnet_pack_weights(ctx, desc, s["F"], s["G"], s["packs"])
    return s


def _prepare_transition(case, d):
    ctx = context()
    n, h, cin, cout, k, stride = (case[f] for f in ("n", "h", "cin", "cout", "k", "stride"))
    desc = B.TransitionDesc(n, h, h, cin, cout, k, stride, int(case["split"]), 1e-5, case["mode"], 0)
    ws = max(B.revnet_transition_workspace_bytes(ctx, desc))
    parts = 2 if case["split"] else 1
    ho = h // stride
    ins = [d.normal(n, h, h, cin // parts) for _ in range(parts)]
    douts = [d.normal(n, ho, ho, cout // 2) for _ in range(2)]
    W = d.normal(cout, k, k, cin) * math.sqrt(2.0 / (cin * k * k))
    gamma, beta = 1.0 + 0.1 * d.normal(cin), 0.1 * d.normal(cin)
    return dict(case=case, desc=desc, ins=ins, douts=douts, W=W, gamma=gamma, beta=beta,
                outs=[torch.empty_like(t) for t in douts], dins=[torch.empty_like(t) for t in ins],
                dW=torch.empty_like(W), dgamma=torch.empty_like(gamma), dbeta=torch.empty_like(beta),
                ws=torch.empty(ws, dtype=torch.uint8, device="cuda"))


def prepare(case, seed):
    d = _Draws(seed)
    if case["path"] in ("step", "step_host"):
        return _prepare_step(case, d)
    return _prepare_transition(case, d) if case["path"] == "transition" else _prepare_block(case, d)


# ------------------------------------------------------------------ one pass
def run(s):
    path, ctx = s["case"]["path"], context()
    if path == "step":
        r = s["run"]
        r.step()
        return dict(loss=r.loss, logits=r.logits, params=r.params)
    if path == "step_host":
        # (the arg-max predictions come back too; ties between bf16-accurate logits make them no output to compare)
        r = s["run"]
        B.revnet_train_step_host(ctx, r.plan, s["images_host"], s["labels_host"], r.images, r.labels, r.params, r.grads, r.momentum,
                                 r.act, r.ws, r.loss, r.pred, s["loss_host"], s["pred_host"])
        return dict(loss=s["loss_host"], params=r.params)
    if path == "block_fwd":
        B.revnet_block_fwd(ctx, s["desc"], s["x1"], s["x2"], s["F"], s["G"], s["y1"], s["y2"], s["ws"])
        return dict(y1=s["y1"], y2=s["y2"])
    if path == "block_train":
        # the weights of a training loop change from step to step, so the packs are made in every pass; the state is
        # overwritten by the block's output and comes back from the reversal
        B.revnet_pack_weights(ctx, s["desc"], s["F"], s["G"], s["packs"])
        B.revnet_block_fwd(ctx, s["desc"], s["x1"], s["x2"], s["F"], s["G"], s["x1"], s["x2"], s["ws"])
        B.revnet_block_bwd(ctx, s["desc"], s["x1"], s["x2"], s["dy1"], s["dy2"], s["F"], s["G"], s["x1"], s["x2"], s["dx1"], s["dx2"],
                           s["gF"], s["gG"], s["ws"])
        return dict(x1=s["x1"], x2=s["x2"], dx1=s["dx1"], dx2=s["dx2"], gF=s["gF"], gG=s["gG"])
    ins, outs, douts, dins = ((t + [None])[:2] for t in (s["ins"], s["outs"], s["douts"], s["dins"]))
    B.revnet_transition_fwd(ctx, s["desc"], *ins, s["W"], s["gamma"], s["beta"], *outs, s["ws"])
    B.revnet_transition_bwd(ctx, s["desc"], *ins, *douts, s["W"], s["gamma"], s["beta"], *dins, s["dW"], s["dgamma"], s["dbeta"], s["ws"])
    return dict(outs=s["outs"], dins=s["dins"], dW=s["dW"], dgamma=s["dgamma"], dbeta=s["dbeta"])


# ------------------------------------------------------------------ what a pass cannot do without
def _net_flops(cfg, stored):
    """Multiply-adds of the convolutions and the classifier of one train step, times two.  A layer runs forward, data
    gradient and weight gradient; one of a reversible unit also runs once more in the reversal (unless activations are kept)."""
    total = 0.0
    h = cfg.img // cfg.stem_stride
    total += 2 * 2.0 * cfg.N * h * h * cfg.stem_k ** 2 * cfg.in_ch * cfg.stem_cout            # no data gradient
    if cfg.maxpool:
        h //= 2
    cprev = cfg.stem_cout
    for s in cfg.stages:
        if s.trans_k:
            h //= s.trans_stride
            total += 3 * 2.0 * cfg.N * h * h * s.trans_k ** 2 * cprev * 2 * s.c
        elif s.down:
            at = h
            h //= 2
            for cin, cout, k, stride in syn.down_fn_layers(s.kind, cprev // 2, s.c, s.w):
                at //= stride
                total += 3 * 2.0 * cfg.N * at * at * k * k * cin * cout
            total += 3 * sum(2.0 * cfg.N * h * h * k * k * cin * cout for cin, cout, k in syn.fn_layers(s.kind, s.c, s.w))
        fn = sum(2.0 * cfg.N * h * h * k * k * cin * cout for cin, cout, k in syn.fn_layers(s.kind, s.c, s.w))
        total += (3 if stored else 4) * 2 * fn * syn.reversible_units(s)
        cprev = 2 * s.c
    return total + 3 * 2.0 * cfg.N * cprev * cfg.n_classes


def work(case):
    if case["path"] in ("step", "step_host"):
        cfg = _config(case)
        n = sum(math.prod(shape) for _, shape, _ in syn.param_specs(cfg))
        # images in; parameters and momentum in and out, gradients out; logits out
        return dict(bytes=4.0 * (cfg.N * cfg.img ** 2 * cfg.in_ch + 5 * n + cfg.N * cfg.n_classes), flops=_net_flops(cfg, case["stored"]))
    if case["path"] == "transition":
        p_in, p_out = case["n"] * case["h"] ** 2, case["n"] * (case["h"] // case["stride"]) ** 2
        nw = case["cout"] * case["k"] ** 2 * case["cin"]
        # forward: input, weights, output; backward: input, upstream gradient, weights, input gradient, weight gradient
        return dict(bytes=4.0 * (3 * p_in * case["cin"] + 2 * p_out * case["cout"] + 3 * nw), flops=3 * 2.0 * p_out * nw)
    p = case["n"] * case["h"] * case["w"]
    nw = 2 * sum(cin * cout * k * k for cin, cout, k in syn.fn_layers(case["kind"], case["c"], case["width"]))
    if case["path"] == "block_fwd":
        return dict(bytes=4.0 * (4 * p * case["c"] + nw), flops=2.0 * p * nw)
    # forward: the pair in and out; backward: the pair and its gradient in and out; weights twice in, their gradients out
    return dict(bytes=4.0 * (12 * p * case["c"] + 3 * nw), flops=4 * 2.0 * p * nw)


def tolerance(case):
    """About four times what one unit in the last place of the batch statistics changes.  Gradients are discontinuous at the
    ReLU's zero: a decision that falls the other way moves single elements of dx by up to their own size (max)."""
    if case["mode"] == 1:
        return {"step": {"rel": 1e-4}, "step_host": {"rel": 1e-4}, "block_fwd": {"rel": 1e-5},
                "block_train": {"rel": 4e-3, "max": 0.9}, "transition": {"rel": 1e-3, "max": 0.9}}[case["path"]]
    if case["path"] in ("step", "step_host"):
        # logits after two steps: 5e-4 .. 2e-3, 9e-3 on the deepest network whose down-sampling units keep their scale
        return {"rel": 2e-2 if case["net"] == "paper_revnet164" else 1e-2}
    return {"block_fwd": {"rel": 4e-3}, "block_train": {"rel": 1e-2, "max": 0.9}, "transition": {"rel": 3e-3, "max": 0.9}}[case["path"]]
