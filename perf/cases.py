"""The work that users of libslim have it do, as cases that can be timed.

A case is a problem (batch B, heads H, length L, head width d, features M, slice
C, dtype, feature map) and a `kind`, the call a program makes on it:

  train   one causal layer forward and backward into kept buffers, as a training
          step does it: slim.forward_into (with the state's residuals) and
          slim.backward_into.
  infer   the causal forward alone (scoring, prefill): slim.forward_into.
  stream  a few new tokens appended to a running state, as generation does it:
          slim.forward_into with S_init / z_init.
  bidir   the non-causal form forward and backward (encoders).
  stack   a stack of residual layers forward and backward (slim.stack_forward /
          slim.stack_backward), slices outer and layers inner.

Sizes and distributions are those of paper_2012_11346_gb300/workloads.py and of
the tests, or generic ones.
"""
import math

import torch

from paper_2012_11346_gb300 import slim
from paper_2012_11346_gb300.workloads import orthogonal_gaussian

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(kind, B, H, L, d, M, C, dtype, feature, layers=1):
    return {"kind": kind, "B": B, "H": H, "L": L, "d": d, "M": M, "C": C, "dtype": dtype,
            "feature": feature, "layers": layers}


def listed():
    cases = [
        # one new token for each of 64 sequence-heads: generation, the smallest call
        ("stream_L1_bf16", _case("stream", 8, 8, 1, 64, 256, 64, "bf16", "exp")),
        # the smallest training step: one chain of four slices, where launches count
        ("train_tiny_f32", _case("train", 1, 1, 256, 16, 32, 64, "f32", "exp")),
        # a medium fp32 layer with sizes that fit no tile: ragged rows, slices and features
        ("train_ragged_f32", _case("train", 3, 5, 1777, 32, 112, 200, "f32", "exp")),
        # prefill / scoring of a batch of odd length, forward only
        ("infer_L4001_bf16", _case("infer", 8, 8, 4001, 64, 256, 1024, "bf16", "exp")),
        # the benchmark's training step
        ("train_L4096_bf16", _case("train", 8, 8, 4096, 64, 256, 1024, "bf16", "exp")),
        # long sequences with small slices: the low-memory end of the slice sweep
        ("train_L32768_C64_bf16", _case("train", 2, 8, 32768, 64, 256, 64, "bf16", "exp")),
        # generalized ReLU features in fp32
        ("train_L8192_relu_f32", _case("train", 4, 12, 8192, 64, 128, 512, "f32", "relu")),
        # wide heads with tiny slices: the near-O(1)-memory extreme
        ("train_L65536_C16_bf16", _case("train", 1, 4, 65536, 128, 256, 16, "bf16", "exp")),
        # the paper's elementwise quadratic map on the benchmark's shape
        ("train_L4096_square_bf16", _case("train", 8, 8, 4096, 64, 64, 1024, "bf16", "square")),
        # an encoder layer on the benchmark's shape
        ("bidir_L4096_bf16", _case("bidir", 8, 8, 4096, 64, 256, 1024, "bf16", "exp")),
        # a three-layer model on the benchmark's shape
        ("stack3_L4096_bf16", _case("stack", 8, 8, 4096, 64, 256, 1024, "bf16", "exp", 3)),
    ]
    return [dict(c, name=n) for n, c in cases]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind, then sizes spread over the range its listed cases
    stand for (B H L up to 262,144 rows, d 16 to 128, M 16 to 256, C from 16)."""
    kind = rng.choice(["stream", "train", "train", "train", "train", "infer", "bidir", "stack"])
    B, H = _log(rng, 1, 8), rng.choice([1, 2, 4, 5, 8, 12])
    if kind == "stream":
        return _case(kind, B, H, _log(rng, 1, 48), rng.choice([64, 128]),
                     rng.choice([128, 256]), 64, rng.choice(["f32", "bf16"]),
                     rng.choice(["exp", "relu"]))
    dtype, feature = rng.choice([("bf16", "exp"), ("bf16", "exp"), ("f32", "exp"),
                                 ("f32", "relu"), ("bf16", "square")])
    d = rng.choice([64, 64, 128, 32, 16])
    if feature == "square":
        M = d
    elif d == 64 and dtype == "bf16":
        M = rng.choice([128, 256])
    else:
        M = 16 * _log(rng, 2, 16)
    if kind == "stack":
        dtype, feature, d, M = "bf16", "exp", 64, rng.choice([128, 256])
    # rows in all: as many as the largest listed case of the kind, fewer where a row is wider
    most = {"train": 262144, "infer": 262144, "bidir": 262144, "stack": 131072}[kind]
    if d * M > 64 * 256 or dtype == "f32":
        most //= 2
    L = max(65, _log(rng, 256, most) // (B * H))
    # slices: of 64 rows and more down to one per 64 slices, or the shortest ones
    if kind in ("train", "infer") and d != 64 and rng.random() < 0.25:
        C = rng.choice([16, 32, 48])
    else:
        C = min(L, max(64, _log(rng, max(64, L // 64), max(65, L))))
    return _case(kind, B, H, L, d, M, C, dtype, feature, _log(rng, 1, 6) if kind == "stack" else 1)


# ------------------------------------------------------------------ inputs
def _inputs(case, seed):
    """q, k, v ~ N(0, 1) / d^(1/4) (U(-1, 1) with ReLU features), Omega
    orthogonal Gaussian for bf16 and iid Gaussian for fp32, dout ~ N(0, 1); for
    stream also the state of an earlier 512-row segment."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    B, H, L, d, M = (case[n] for n in ("B", "H", "L", "d", "M"))
    dt = DTYPES[case["dtype"]]

    def rows(n):
        if case["feature"] == "relu":
            return (torch.rand(B, H, n, d, generator=g, device=dev) * 2.0 - 1.0).to(dt)
        return (torch.randn(B, H, n, d, generator=g, device=dev) / d ** 0.25).to(dt)

    def omega():
        if case["feature"] == "square":
            return None
        if case["dtype"] == "bf16":
            cg = torch.Generator().manual_seed(int(torch.randint(1 << 40, (1,), generator=g,
                                                                 device=dev)))
            return orthogonal_gaussian(M, d, cg).to(dev).contiguous()
        return torch.randn(M, d, generator=g, device=dev)

    x = {}
    if case["kind"] == "stack":
        x["x"] = rows(L)
        oms = [omega() for _ in range(case["layers"])]
        x["omegas"] = None if oms[0] is None else torch.stack(oms).contiguous()
        x["dy"] = torch.randn(B, H, L, d, generator=g, device=dev).to(dt)
        return x
    x["q"], x["k"], x["v"], x["omega"] = rows(L), rows(L), rows(L), omega()
    if case["kind"] in ("train", "bidir"):
        x["dout"] = torch.randn(B, H, L, d, generator=g, device=dev).to(dt)
    if case["kind"] == "stream":
        # the state after 512 earlier rows, summed here in double precision
        k, v = rows(512), rows(512)
        phi = _phi(k, x["omega"], case["feature"])
        x["S0"] = (phi.transpose(-1, -2) @ v.double()).float().contiguous()
        x["z0"] = phi.sum(-2).float().contiguous()
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    B, H, L, d, M, C = (case[n] for n in ("B", "H", "L", "d", "M", "C"))
    dt, ft, kind = DTYPES[case["dtype"]], case["feature"], case["kind"]
    dev = torch.device("cuda")

    def ws(n):
        return torch.empty(max(n, 256), dtype=torch.uint8, device=dev)

    st = {"case": case, "x": x}
    if kind == "stack":
        for name, bwd in (("wf", False), ("wb", True)):
            st[name] = ws(slim.stack_workspace_size(B, H, L, d, M, C, case["layers"], dt, ft, bwd))
        return st
    size = slim.bidir_workspace_size if kind == "bidir" else slim.workspace_size
    st["wf"] = ws(size(B, H, L, d, M, C, dt, ft, False))
    st["out"] = torch.empty_like(x["q"])
    st["S"] = torch.empty(B, H, M, d, device=dev)
    st["z"] = torch.empty(B, H, M, device=dev)
    if kind == "train":
        st["S_lo"], st["z_lo"] = torch.empty_like(st["S"]), torch.empty_like(st["z"])
    if kind in ("train", "bidir"):
        st["wb"] = ws(size(B, H, L, d, M, C, dt, ft, True))
        for n in ("dq", "dk", "dv"):
            st[n] = torch.empty_like(x["q"])
        st["domega"] = None if x["omega"] is None else torch.empty(M, d, device=dev)
    return st


def run(st):
    case, x = st["case"], st["x"]
    C, ft, kind = case["C"], case["feature"], case["kind"]
    if kind == "stack":
        y, S, z, S_lo, z_lo = slim.stack_forward(x["x"], x["omegas"], C, ft,
                                                 layers=case["layers"], workspace=st["wf"])
        dx, dom = slim.stack_backward(x["x"], x["omegas"], x["dy"], S, z, C, ft, S_lo=S_lo,
                                      z_lo=z_lo, workspace=st["wb"])
        return {"y": y, "S": S, "z": z, "dx": dx, "domegas": dom}
    res = {"out": st["out"], "S": st["S"], "z": st["z"]}
    head = (x["q"], x["k"], x["v"], x["omega"])
    if kind == "infer":
        slim.forward_into(*head, C, ft, st["out"], st["S"], st["z"], st["wf"])
        return res
    if kind == "stream":
        slim.forward_into(*head, C, ft, st["out"], st["S"], st["z"], st["wf"], S_init=x["S0"],
                          z_init=x["z0"])
        return res
    grads = (st["dq"], st["dk"], st["dv"], st["domega"])
    if kind == "bidir":
        slim.forward_bidir_into(*head, C, ft, st["out"], st["S"], st["z"], st["wf"])
        slim.backward_bidir_into(*head, st["out"], x["dout"], st["S"], st["z"], C, ft, *grads,
                                 st["wb"])
    else:
        slim.forward_into(*head, C, ft, st["out"], st["S"], st["z"], st["wf"], S_lo=st["S_lo"],
                          z_lo=st["z_lo"])
        slim.backward_into(*head, st["out"], x["dout"], st["S"], st["z"], C, ft, *grads, st["wb"],
                           S_lo=st["S_lo"], z_lo=st["z_lo"])
    res.update(dq=st["dq"], dk=st["dk"], dv=st["dv"])
    if st["domega"] is not None:
        res["domega"] = st["domega"]
    return res


def work(case):
    """Algorithmic work of one pass.  Per row and layer: the forward's 8dM FLOPs
    (two projections, the state's delta, the readout) and the backward's 22dM;
    without projections (the quadratic map) 4dM and 10dM.  Bytes: inputs read
    and outputs written once."""
    B, H, L, d, M, s = (case[n] for n in ("B", "H", "L", "d", "M", "layers"))
    rows, es = B * H * L, 2 if case["dtype"] == "bf16" else 4
    kind, square = case["kind"], case["feature"] == "square"
    fwd, bwd = (4, 10) if square else (8, 22)
    om = 0 if square else M * d * 4
    state = B * H * M * (d + 1) * 4
    if kind in ("infer", "stream"):
        n = 2 if kind == "stream" else 1
        return {"bytes": rows * d * es * 4 + om + n * state, "flops": fwd * d * M * rows}
    tensors = 4 if kind == "stack" else 8  # x, dy, y, dx; or q, k, v, dout, out, dq, dk, dv
    return {"bytes": rows * d * es * tensors + s * (2 * om + state),
            "flops": (fwd + bwd) * d * M * rows * s}


# ------------------------------------------------------------------ 64-bit values
def _phi(x, omega, feature):
    x = x.double()
    if feature == "square":
        return x * x
    om = omega.double()
    p = x @ om.T
    if feature == "exp":
        return torch.exp(p - 0.5 * (x * x).sum(-1, keepdim=True)) / math.sqrt(om.shape[0])
    return torch.relu(p) / math.sqrt(om.shape[0])


def _attention(q, k, v, omega, feature, causal, S0=None, z0=None, T=64):
    """out, S, z of eq. 2 in double precision for [B, H, L, d] inputs, rows in
    blocks of T (zero-padded) with the exclusive prefix of the blocks' sums."""
    B, H, L, d = q.shape
    fq, fk, v = _phi(q, omega, feature), _phi(k, omega, feature), v.double()
    one = torch.cat([v, torch.ones_like(v[..., :1])], -1)
    if not causal:
        st = fk.transpose(-1, -2) @ one
        nd = fq @ st
    else:
        pad = (-L) % T

        def blocks(t):
            return torch.nn.functional.pad(t, (0, 0, 0, pad)).reshape(B, H, -1, T, t.shape[-1])

        bq, bk, b1 = blocks(fq), blocks(fk), blocks(one)
        delta = bk.transpose(-1, -2) @ b1
        incl = torch.cumsum(delta, 2)
        pre = incl - delta
        st = incl[:, :, -1]
        if S0 is not None:
            first = torch.cat([S0.double(), z0.double().unsqueeze(-1)], -1)
            pre = pre + first.unsqueeze(2)
            st = st + first
        nd = bq @ pre + torch.tril(bq @ bk.transpose(-1, -2)) @ b1
        nd = nd.reshape(B, H, L + pad, d + 1)[:, :, :L]
    den = nd[..., d:]
    zero = den == 0
    out = torch.where(zero, torch.zeros_like(nd[..., :d]), nd[..., :d] / den.masked_fill(zero, 1.0))
    return out, st[..., :d], st[..., d]


def exact(case, seed):
    x = _inputs(case, seed)
    ft, kind = case["feature"], case["kind"]

    def leaf(t):
        return t.double().requires_grad_(True)

    if kind == "stack":
        X = leaf(x["x"])
        oms = [leaf(o) for o in x["omegas"]] if x["omegas"] is not None else [None] * case["layers"]
        h, S, z = X, [], []
        for o in oms:
            u = case["d"] ** -0.25 * h / torch.sqrt((h * h).mean(-1, keepdim=True) + 1e-6)
            y, Sr, zr = _attention(u, u, u, o, ft, True)
            S.append(Sr.detach())
            z.append(zr.detach())
            h = h + y
        leaves = [X] + [o for o in oms if o is not None]
        gr = torch.autograd.grad(h, leaves, x["dy"].double())
        return {"y": h.detach(), "S": torch.stack(S), "z": torch.stack(z), "dx": gr[0],
                "domegas": torch.stack(gr[1:]) if len(gr) > 1 else None}
    if kind in ("infer", "stream"):
        out, S, z = _attention(x["q"], x["k"], x["v"], x["omega"], ft, True, x.get("S0"),
                               x.get("z0"))
        return {"out": out, "S": S, "z": z}
    leaves = [leaf(x[n]) for n in ("q", "k", "v")]
    if x["omega"] is not None:
        leaves.append(leaf(x["omega"]))
    om = leaves[3] if len(leaves) > 3 else None
    out, S, z = _attention(*leaves[:3], om, ft, kind == "train")
    gr = torch.autograd.grad(out, leaves, x["dout"].double())
    res = {"out": out.detach(), "S": S.detach(), "z": z.detach(), "dq": gr[0], "dk": gr[1],
           "dv": gr[2]}
    if om is not None:
        res["domega"] = gr[3]
    return res
