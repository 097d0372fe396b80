"""The work a user of libmdbf has it do, as cases that can be timed and whose results can be compared.

Four kinds of call, each through the public binding (paper_2512_24545_b200.mdbf):

    step    the seven projections of a decoder block: q, k, v on the hidden state, o, gate and up on the second hidden
            state, down - siblings where they share their input, as a decode or prefill step of a model runs them
    layer   one quantized linear layer on device buffers, or on pinned host buffers
    sum     a layer with residual compensation: several terms on one input
    msvid   the quantizer's projection of a dense factor (own signs, or a mask held fixed)
    admm    the quantizer's refinement of one factor

Layers are drawn like the repository's synthetic workloads: fair signs, Gaussian envelopes, Gaussian activations with one
per cent of the channels twenty times larger.  The quantizer's matrices are what it meets on a factor that a sum of a few
envelopes describes: positive envelopes of decreasing weight under random signs, with noise on top.
"""
from __future__ import annotations

import math
import weakref

import torch

from paper_2512_24545_b200 import mdbf as M

_TORCH = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


# ------------------------------------------------------------------------------------------------------------- cases
def listed():
    return [
        # the 256-square fp32 layer of the tests: the smallest call there is, fp32 all through
        _layer("fp32_small", d_out=256, d_in=256, k=128, l=4, T=8, env="f32", act="f32"),
        # one attention projection of a 7B-class decoder at one bit per weight, one token: a call whose latency counts
        _layer("decode_proj_4096", d_out=4096, d_in=4096, k=1664, l=16, T=1),
        # the same projection at 1.5 bits called on host buffers: copies in and out belong to the call
        _layer("host_proj_4096", d_out=4096, d_in=4096, k=2560, l=16, T=1, host=True),
        # a token through four blocks of a 7B-class decoder, replayed as one CUDA graph, as serving loops do
        _step("decode_blocks_7b", hidden=4096, kv=4096, ffn=11008, k_attn=1664, k_kv=1664, k_ffn=2560, l=16, T=1, blocks=4, graph=True),
        # a token through one 70B-class block: its 107 MB of packed weights stream from memory
        _step("decode_block_70b", hidden=8192, kv=1024, ffn=28672, k_attn=3712, k_kv=512, k_ffn=6016, l=16, T=1),
        # residual compensation with two single-envelope terms, together one bit per weight
        _sum("sum_two_terms", d_out=4096, d_in=4096, k=896, l=1, terms=2, T=1),
        # sixteen requests decoded together, the MLP of a 7B-class decoder at 1.5 bits
        _layer("batch_mlp_T16", d_out=11008, d_in=4096, k=3968, l=16, T=16),
        # sizes that fit no tile: a pruned layer, bf16 envelopes of rank 6, an odd batch
        _layer("batch_ragged", d_out=1723, d_in=2312, k=877, l=6, T=37, env="bf16"),
        # a prompt of ordinary length through one projection
        _layer("prefill_4096_T777", d_out=4096, d_in=4096, k=1664, l=16, T=777),
        # a 2048-token prompt through a 70B-class block
        _step("prefill_block_70b", hidden=8192, kv=1024, ffn=28672, k_attn=3712, k_kv=512, k_ffn=6016, l=16, T=2048),
        # quantizer, initialisation: a factor of the 70B-class gate projection
        _msvid("msvid_28672x6016", rows=28672, cols=6016, l=16, n_iter=4),
        # quantizer, refinement: three inner iterations on a factor of an 8192-square projection
        _admm("admm_8192_r3712", n=8192, m=8192, r=3712, l=16, n_inner=3, n_iter=8),
    ]


def draw(rng):
    """One more case of the same ranges: sizes spread over their logarithm, half of them multiples of 128, the others odd."""
    what = rng.choice(["layer1", "layer1", "step1", "sum", "host", "batch", "batch", "prefill", "prefill", "fp32", "msvid", "admm"])
    l = rng.choice([1, 2, 4, 6, 8, 12, 16, 16, 16])
    env = rng.choice(["f16", "f16", "bf16"])
    if what == "fp32":
        d_out, d_in = _size(rng, 128, 2048, 1), _size(rng, 128, 2048, 1)
        return _layer(None, d_out=d_out, d_in=d_in, k=_rank(rng, d_out, d_in, l), l=l, T=_log(rng, 1, 64), env="f32", act="f32")
    if what == "step1":
        hidden, ffn = _size(rng, 1024, 8192, 8), _size(rng, 2048, 14336, 8)
        kv = rng.choice([hidden, _size(rng, 256, hidden, 8)])
        return _step(None, hidden=hidden, kv=kv, ffn=ffn, k_attn=_rank(rng, hidden, hidden, l), k_kv=_rank(rng, kv, hidden, l),
                     k_ffn=_rank(rng, ffn, hidden, l), l=l, T=1, env=env, blocks=rng.choice([1, 2]), graph=rng.random() < 0.5)
    if what == "sum":
        d_out, d_in, terms = _size(rng, 512, 8192, 1), _size(rng, 512, 8192, 8), rng.choice([2, 2, 3])
        l = min(l, 4)
        return _sum(None, d_out=d_out, d_in=d_in, k=max(64, _rank(rng, d_out, d_in, l) // terms), l=l, terms=terms, T=1, env=env)
    if what == "msvid":
        rows, cols = _size(rng, 512, 16384, 1), _size(rng, 512, 6016, 4)
        return _msvid(None, rows=rows, cols=cols, l=l, n_iter=rng.choice([4, 8]), fixed_mask=rng.random() < 0.3)
    if what == "admm":
        n, m = _size(rng, 512, 8192, 1), _size(rng, 512, 8192, 1)
        return _admm(None, n=n, m=m, r=max(64, int(min(n, m) * rng.uniform(0.25, 0.45)) // 4 * 4), l=l, n_inner=rng.choice([1, 2, 3]),
                     n_iter=rng.choice([4, 8]), transposed=rng.random() < 0.5)
    d_out, d_in = _size(rng, 256, 14336, 1), _size(rng, 256, 14336, 8)
    T = {"layer1": 1, "host": rng.choice([1, 1, _log(rng, 2, 64)]), "batch": _log(rng, 2, 64), "prefill": _log(rng, 65, 2048)}[what]
    return _layer(None, d_out=d_out, d_in=d_in, k=_rank(rng, d_out, d_in, l), l=l, T=T, env=env, host=what == "host")


def _case(name, kind, **sizes):
    c = {"kind": kind, **sizes}
    return c if name is None else {"name": name, **c}


def _layer(name, d_out, d_in, k, l, T, env="f16", act="bf16", host=False):
    return _case(name, "layer", d_out=d_out, d_in=d_in, k=k, l=l, T=T, env=env, act=act, host=host)


def _step(name, hidden, kv, ffn, k_attn, k_kv, k_ffn, l, T, env="f16", blocks=1, graph=False):
    return _case(name, "step", hidden=hidden, kv=kv, ffn=ffn, k_attn=k_attn, k_kv=k_kv, k_ffn=k_ffn, l=l, T=T, env=env, act="bf16",
                 blocks=blocks, graph=graph)


def _sum(name, d_out, d_in, k, l, terms, T, env="f16"):
    return _case(name, "sum", d_out=d_out, d_in=d_in, k=k, l=l, terms=terms, T=T, env=env, act="bf16")


def _msvid(name, rows, cols, l, n_iter, fixed_mask=False):
    return _case(name, "msvid", rows=rows, cols=cols, l=l, n_iter=n_iter, fixed_mask=fixed_mask)


def _admm(name, n, m, r, l, n_inner, n_iter, transposed=False):
    return _case(name, "admm", n=n, m=m, r=r, l=l, n_inner=n_inner, n_iter=n_iter, transposed=transposed)


def _log(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _size(rng, lo, hi, step):
    """A size in [lo, hi]: a multiple of 128 half of the time, else any multiple of `step`."""
    step = 128 if rng.random() < 0.5 else step
    return min(hi, max(lo, _log(rng, lo, hi) // step * step))


def _rank(rng, d_out, d_in, l):
    """The inner rank that 1.0 to 1.5 bits per weight leave with 16-bit envelopes."""
    bits = rng.uniform(1.0, 1.5) * d_out * d_in - 16 * l * (d_out + d_in)
    k = max(64, int(bits / (d_out + d_in + 32 * l)))
    return k // 128 * 128 if k >= 128 and rng.random() < 0.5 else k


# ----------------------------------------------------------------------------------------------------------- prepare
class _Handle:
    """A packed layer that is given back with the state that holds it."""

    def __init__(self, gen, d_out, d_in, k, l, env, max_T):
        std = k ** -0.5 if env == "f32" else 0.02
        signs = [torch.randint(0, 2, (r, c), generator=gen, device="cuda", dtype=torch.int8) * 2 - 1 for r, c in ((d_out, k), (k, d_in))]
        envs = [torch.randn((r, l), generator=gen, device="cuda") * std for r in (d_out, k, k, d_in)]
        self.d_out, self.d_in = d_out, d_in
        self.address = M.mdbf_pack(d_out, d_in, k, l, M.DTYPES[env], max_T, *[t.data_ptr() for t in signs + envs], inputs_on_device=True,
                                   stream=_stream())
        weakref.finalize(self, M.mdbf_destroy, self.address)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _activations(gen, T, d_in, act):
    x = torch.randn((T, d_in), generator=gen, device="cuda")
    if act != "f32":
        big = torch.randperm(d_in, generator=gen, device="cuda")[: round(0.01 * d_in)]
        x[:, big] *= 20.0
    return x.to(_TORCH[act])


def _envelope(gen, rows, cols, l):
    """A positive matrix of rank l: log-normal outer products, each four fifths of the one before."""
    w = 0.8 ** torch.arange(l, device="cuda", dtype=torch.float32)
    a = torch.exp(0.25 * torch.randn((rows, l), generator=gen, device="cuda"))
    b = torch.exp(0.25 * torch.randn((cols, l), generator=gen, device="cuda"))
    return (a * (w / w.sum())) @ b.T


def _signs(gen, rows, cols):
    return torch.randint(0, 2, (rows, cols), generator=gen, device="cuda", dtype=torch.float32) * 2 - 1


def _device(*shape, dtype=torch.float32):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def prepare(case, seed):
    gen = _generator(seed)
    return {"layer": _prepare_layer, "step": _prepare_step, "sum": _prepare_sum, "msvid": _prepare_msvid, "admm": _prepare_admm}[case["kind"]](
        case, gen)


def _prepare_layer(c, gen):
    h = _Handle(gen, c["d_out"], c["d_in"], c["k"], c["l"], c["env"], c["T"])
    x = _activations(gen, c["T"], c["d_in"], c["act"])
    y = _device(c["T"], c["d_out"], dtype=_TORCH[c["act"]])
    if c["host"]:
        M.mdbf_prepare_host_staging(h.address)
        x, y = x.cpu().pin_memory(), y.cpu().pin_memory()
    return {"case": c, "layer": h, "x": x, "y": y}


def _prepare_sum(c, gen):
    hs = [_Handle(gen, c["d_out"], c["d_in"], c["k"], c["l"], c["env"], c["T"]) for _ in range(c["terms"])]
    return {"case": c, "layers": hs, "x": _activations(gen, c["T"], c["d_in"], c["act"]), "acc": _device(c["T"], c["d_out"]),
            "y": _device(c["T"], c["d_out"], dtype=_TORCH[c["act"]])}


def _prepare_step(c, gen):
    hidden, kv, ffn = c["hidden"], c["kv"], c["ffn"]
    shapes = ((hidden, hidden, c["k_attn"]), (kv, hidden, c["k_kv"]), (kv, hidden, c["k_kv"]), (hidden, hidden, c["k_attn"]),
              (ffn, hidden, c["k_ffn"]), (ffn, hidden, c["k_ffn"]), (hidden, ffn, c["k_ffn"]))
    blocks = []
    for _ in range(c["blocks"]):
        hs = [_Handle(gen, do, di, k, c["l"], c["env"], c["T"]) for do, di, k in shapes]
        xs = [_activations(gen, c["T"], d, c["act"]) for d in (hidden, hidden, hidden, ffn)]
        ys = [_device(c["T"], do, dtype=_TORCH[c["act"]]) for do, _, _ in shapes]
        blocks.append((hs, xs, ys))
    state = {"case": c, "blocks": blocks, "graph": None}
    if c["graph"]:
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            _run_blocks(state)
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                _run_blocks(state)
        torch.cuda.current_stream().wait_stream(stream)
        state["graph"] = graph
    return state


def _prepare_msvid(c, gen):
    rows, cols, l = c["rows"], c["cols"], c["l"]
    E = _envelope(gen, rows, cols, l)
    words = _device(rows, (cols + 31) // 32, dtype=torch.int32)
    if c["fixed_mask"]:                       # entries scattered about the envelope, under a mask that is given
        Z = E * (1.0 + 0.3 * torch.randn((rows, cols), generator=gen, device="cuda"))
        S = _signs(gen, rows, cols)
        Z *= S
        M.mdbf_pack_signs(S.to(torch.int8).data_ptr(), rows, cols, words.data_ptr(), True, _stream())
        torch.cuda.synchronize()
    else:                                     # Gaussian entries, as a factor of a trained matrix has
        Z = E * torch.randn((rows, cols), generator=gen, device="cuda")
    n = M.mdbf_msvid_workspace_bytes(rows, cols, l)
    return {"case": c, "Z": Z, "Q0": torch.randn((cols, l), generator=gen, device="cuda"), "S": words, "U": _device(rows, l),
            "V": _device(cols, l), "sigma": _device(l), "workspace": torch.empty(n, dtype=torch.uint8, device="cuda")}


def _prepare_admm(c, gen):
    """A factor near the end of its refinement: op(W) is its product with the fixed factor and a few per cent of noise, so
    that no entry of the iterate is near zero and the signs are settled."""
    n, m, r, l = c["n"], c["m"], c["r"], c["l"]
    U = _signs(gen, n, r) * _envelope(gen, n, r, l)
    V = _signs(gen, m, r) * _envelope(gen, m, r, l)
    W = U @ V.T
    W += 0.02 * float(W.std()) * torch.randn(W.shape, generator=gen, device="cuda")
    if c["transposed"]:
        W = W.T.contiguous()
    U *= 1.0 + 0.02 * torch.randn((n, r), generator=gen, device="cuda")
    nbytes = M.mdbf_admm_workspace_bytes(n, m, r, l)
    return {"case": c, "W": W, "V": V, "U": U, "Lambda": torch.zeros_like(U), "rho": 3.0 * float((V * V).sum()) / r,
            "Q0": torch.randn((r, l), generator=gen, device="cuda"), "S": _device(n, (r + 31) // 32, dtype=torch.int32), "Ul": _device(n, l),
            "Vl": _device(r, l), "sigma": _device(l), "U_tilde": _device(n, r),
            "workspace": torch.empty(nbytes, dtype=torch.uint8, device="cuda")}


# --------------------------------------------------------------------------------------------------------------- run
def run(state):
    return {"layer": _run_layer, "step": _run_step, "sum": _run_sum, "msvid": _run_msvid, "admm": _run_admm}[state["case"]["kind"]](state)


def _run_layer(s):
    c = s["case"]
    call = M.mdbf_linear_forward_host if c["host"] else M.mdbf_linear_forward
    call(s["layer"].address, s["x"].data_ptr(), s["y"].data_ptr(), c["T"], M.DTYPES[c["act"]], _stream())
    return s["y"]


def _run_sum(s):
    c = s["case"]
    M.mdbf_linear_forward_sum([h.address for h in s["layers"]], s["x"].data_ptr(), s["y"].data_ptr(), s["acc"].data_ptr(), c["T"],
                              M.DTYPES[c["act"]], _stream())
    return s["y"]


def _run_blocks(s):
    T, act, st = s["case"]["T"], M.DTYPES[s["case"]["act"]], _stream()
    for h, x, y in s["blocks"]:
        M.mdbf_linear_forward_siblings([h[0].address, h[1].address, h[2].address], x[0].data_ptr(), [t.data_ptr() for t in y[0:3]], T, act, st)
        M.mdbf_linear_forward(h[3].address, x[1].data_ptr(), y[3].data_ptr(), T, act, st)
        M.mdbf_linear_forward_siblings([h[4].address, h[5].address], x[2].data_ptr(), [t.data_ptr() for t in y[4:6]], T, act, st)
        M.mdbf_linear_forward(h[6].address, x[3].data_ptr(), y[6].data_ptr(), T, act, st)


def _run_step(s):
    if s["graph"] is not None:
        s["graph"].replay()
    else:
        _run_blocks(s)
    return [y for _, _, ys in s["blocks"] for y in ys]


def _run_msvid(s):
    c = s["case"]
    mid = (s["Z"].data_ptr(), s["S"].data_ptr(), c["rows"], c["cols"], c["l"], c["n_iter"], s["Q0"].data_ptr())
    end = (s["U"].data_ptr(), s["V"].data_ptr(), s["sigma"].data_ptr(), s["workspace"].data_ptr(), s["workspace"].numel(), _stream())
    if c["fixed_mask"]:
        M.mdbf_project_fixed_mask(*mid, *end)
    else:
        M.mdbf_msvid(mid[0], *mid[2:], mid[1], *end)
    return {"S": s["S"], "U": s["U"], "V": s["V"], "sigma": s["sigma"]}


def _run_admm(s):
    c = s["case"]
    rows, cols = (c["m"], c["n"]) if c["transposed"] else (c["n"], c["m"])
    M.mdbf_admm_factor_update(s["W"].data_ptr(), rows, cols, c["transposed"], s["V"].data_ptr(), c["r"], s["U"].data_ptr(),
                              s["Lambda"].data_ptr(), s["rho"], c["l"], c["n_inner"], c["n_iter"], s["Q0"].data_ptr(), s["S"].data_ptr(),
                              s["Ul"].data_ptr(), s["Vl"].data_ptr(), s["sigma"].data_ptr(), s["U_tilde"].data_ptr(),
                              s["workspace"].data_ptr(), s["workspace"].numel(), _stream())
    return {name: s[name] for name in ("U", "Lambda", "U_tilde", "S", "Ul", "Vl", "sigma")}


# ---------------------------------------------------------------------------------------------------- work, tolerance
def _forward_work(d_out, d_in, k, l, T, env, act):
    """Bytes of a layer (packed signs and envelopes) and its operations: the cheaper of the l sign products per token and of
    rebuilding each factor once."""
    weights = k * (d_out + d_in) / 8 + (4 if env == "f32" else 2) * l * (d_out + d_in + 2 * k)
    return weights, min(2.0 * l * T, 2.0 * T + 2.0 * l) * k * (d_out + d_in)


def work(case):
    c, kind = case, case["kind"]
    size = 4 if c.get("act") == "f32" else 2
    if kind in ("layer", "sum"):
        weights, flops = _forward_work(c["d_out"], c["d_in"], c["k"], c["l"], c["T"], c["env"], c["act"])
        terms = c.get("terms", 1)
        return {"bytes": terms * weights + size * c["T"] * (c["d_in"] + c["d_out"]), "flops": terms * flops}
    if kind == "step":
        hidden, kv, ffn = c["hidden"], c["kv"], c["ffn"]
        parts = [_forward_work(do, di, k, c["l"], c["T"], c["env"], c["act"]) for do, di, k in (
            (hidden, hidden, c["k_attn"]), (kv, hidden, c["k_kv"]), (kv, hidden, c["k_kv"]), (hidden, hidden, c["k_attn"]),
            (ffn, hidden, c["k_ffn"]), (ffn, hidden, c["k_ffn"]), (hidden, ffn, c["k_ffn"]))]
        activations = size * c["T"] * (3 * hidden + ffn + 3 * hidden + 2 * kv + 2 * ffn)
        return {"bytes": c["blocks"] * (sum(w for w, _ in parts) + activations), "flops": c["blocks"] * sum(f for _, f in parts)}
    if kind == "msvid":
        rows, cols, l, n = c["rows"], c["cols"], c["l"], c["n_iter"]
        return {"bytes": 4.0 * rows * cols + rows * cols / 8 + 4.0 * l * (rows + 2 * cols), "flops": (2 * n + 1) * 2.0 * l * rows * cols}
    n, m, r, l, inner, it = (c[key] for key in ("n", "m", "r", "l", "n_inner", "n_iter"))
    flops = 2.0 * n * m * r + m * r * r + r ** 3 / 3.0 + inner * (2.0 * n * r * r + (2 * it + 1) * 2.0 * l * n * r)
    return {"bytes": 4.0 * (n * m + m * r + 5 * n * r) + n * r / 8, "flops": flops}


def tolerance(case):
    if case["kind"] == "msvid":
        # with rows and columns in another order: rel up to 1.3e-5, max 2.2e-4; columns of two singular values ten times closer mix that much more
        return {"rel": 1e-4, "max": 3e-3, "differ": 0.0}
    if case["kind"] == "admm":
        # with the contraction in another order, over four passes: rel up to 1.1e-4 and max 7e-4, both in the dual, a difference of near equals
        return {"rel": 4e-4, "max": 3e-3, "differ": 1e-5}
    if case["act"] == "f32":
        return {"rel": 2e-6, "max": 1e-5}       # against fp64: rel 2e-7, max 1.3e-6
    return {"rel": 1e-2, "max": 0.1}            # bf16 kernels against the fp32 one: rel 2e-3 to 4.8e-3, max up to 4e-2
