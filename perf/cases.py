"""Performance cases: what a user of this framework has it do, through the
public binding (`paper_1503_00638_gb300.bsgpu`) and the batch engine.

The kinds of work (`kind` of a case) and the sizes they take in real use:

* ``cube``     precision reduction + Bitshuffle + LZ4 of a visibility cube
               (`compress_vis` / `compress_vis_ex`): one acquisition chunk of a
               small array up to the whole CHIME-shaped cube of the benchmark.
* ``uncube``   reading such a stream back (`decompress` with its block index).
* ``round``    precision reduction alone (`reduce_precision`).
* ``walk``     Bitshuffle + LZ4 of data that is already integers or float64
               (`compress`), every element size, blocks of 1 to 64 KiB, both
               match-search levels, lengths that fill no whole block.
* ``unwalk``   reading such a stream back, with or without a block index (a
               stream from another writer of the format carries none).
* ``shuffle``  Bitshuffle and its inverse without LZ4.
* ``batch``    the batched engine: uneven chunks compressed and read back.

Buffers that a program would keep (workspace, output) are made by `prepare`;
the stream buffers start zeroed, so that what a call does not write is alike
on every run.
"""
from __future__ import annotations

import math

import torch

from paper_1503_00638_gb300 import bsgpu, engine, synth


def listed():
    return [
        # one chunk of a 16-input array (the smoke test's cube): 1.1 MB, where
        # launches and the latency of one block count
        _cube("cube-small", 16, 16, 64, log2n=16),
        # the same chunk read back
        dict(_cube("uncube-small", 16, 16, 64, log2n=16), kind="uncube"),
        # the benchmark's CHIME-shaped cube, 1.08 GB
        _cube("cube-chime", 1024, 128, 16, log2n=17),
        # the same cube read back
        dict(_cube("uncube-chime", 1024, 128, 16, log2n=17), kind="uncube"),
        # a correlator's int32 output as it is written (time slowest), stored
        # as 8-byte samples in the paper's 4096-byte blocks, a time axis that
        # is no multiple of 16
        _cube("cube-int32-instrument", 48, 128, 40, log2n=17, dtype="i32", scale=4096.0,
              time_slowest=True, elem_size=8, block_bytes=4096),
        # a small array with the noise of the full covariance (8 inputs)
        _cube("cube-fullcov8", 1024, 8, 64, log2n=16, full_cov=True),
        # rounding alone with the compensated f, 128 inputs, to be handed on uncompressed
        dict(_cube("round-compensated", 128, 128, 16, log2n=17, compensate=True), kind="round"),
        # 16-bit samples, the better match search, the paper's block size, a
        # length that fills neither a block nor a group of eight
        _walk("walk-u16-level1", 32 * 2 ** 20 + 1237, 2, 4096, level=1),
        # float64 time streams in 32 KiB blocks
        _walk("walk-f64-32k", 32 * 2 ** 20, 8, 32768, floating=True),
        # int32 in 16 KiB blocks from a writer that kept no block index
        dict(_walk("unwalk-i32-16k-noindex", 48 * 2 ** 20 + 771, 4, 16384), kind="unwalk",
             index=False),
        # Bitshuffle alone and back, bytes (raw 8-bit voltages), a ragged end
        dict(_walk("shuffle-u8", 256 * 2 ** 20 + 4099, 1, 8192), kind="shuffle"),
        # the batched engine over uneven chunks: cubes and walks of 64 KiB to 64 MiB
        dict(name="batch-64", kind="batch", chunks=64, block_bytes=8192, pick=4),
    ]


def _cube(name, n_freq, n_inputs, n_time, *, log2n, f=0.01, dtype="f32", scale=1.0,
          time_slowest=False, compensate=False, full_cov=False, elem_size=4, block_bytes=8192):
    return {"name": name, "kind": "cube", "n_freq": n_freq, "n_inputs": n_inputs,
            "n_time": n_time, "log2n": log2n, "f": f, "dtype": dtype, "scale": scale,
            "time_slowest": time_slowest, "compensate": compensate, "full_cov": full_cov,
            "elem_size": elem_size, "block_bytes": block_bytes}


def _walk(name, n_elem, elem_size, block_bytes, *, level=0, floating=False):
    return {"name": name, "kind": "walk", "n_elem": n_elem, "elem_size": elem_size,
            "block_bytes": block_bytes, "level": level, "floating": floating, "index": True}


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, sizes log-uniform over what the listed ones span."""
    kind = rng.choice(["cube", "cube", "uncube", "round", "walk", "walk", "unwalk", "shuffle",
                       "batch"])
    if kind == "batch":
        return dict(kind="batch", chunks=_loguniform(rng, 4, 64), block_bytes=rng.choice(
            [2048, 4096, 8192]), pick=rng.randrange(1000))
    if kind in ("walk", "unwalk", "shuffle"):
        es = rng.choice([1, 2, 4, 8])
        case = _walk("", _loguniform(rng, 2 ** 20, 2 ** 28) // es + rng.randrange(64), es,
                     rng.choice([1024, 2048, 4096, 8192, 16384, 32768, 65536]),
                     level=rng.choice([0, 0, 0, 1]), floating=es == 8 and rng.random() < 0.5)
        case["kind"] = kind
        if kind == "unwalk":
            case["index"] = rng.random() < 0.5
    else:
        full_cov = kind != "uncube" and rng.random() < 0.15
        n_inputs = rng.randint(4, 16) if full_cov else _loguniform(rng, 4, 128)
        n_time = rng.choice([16, 32, 64, rng.randint(5, 100)])
        samples = _loguniform(rng, 2 ** 17, 2 ** 21 if full_cov else 2 ** 26)
        n_freq = max(1, samples // (synth.n_products(n_inputs) * n_time))
        i32 = rng.random() < 0.3
        case = _cube("", n_freq, n_inputs, n_time, log2n=rng.choice([16, 17]),
                     f=rng.choice([1e-3, 1e-2, 0.1]), dtype="i32" if i32 else "f32",
                     scale=4096.0 if i32 else 1.0, time_slowest=rng.random() < 0.25,
                     compensate=not full_cov and rng.random() < 0.25, full_cov=full_cov,
                     elem_size=rng.choice([4, 4, 8]), block_bytes=rng.choice([4096, 8192]))
        case["kind"] = kind
    del case["name"]
    return case


# -- inputs -----------------------------------------------------------------

def _cube_input(case, seed):
    """The visibility cube as the user holds it (see `_cube`)."""
    cfg = synth.VisConfig(case["n_freq"], case["n_inputs"], case["n_time"], 2 ** case["log2n"],
                          case["f"], seed=seed, drift=True)
    if case["full_cov"]:
        v = _physical_cube(cfg, seed)
    else:
        v = synth.visibilities_torch(cfg)
    if case["dtype"] == "i32":
        a = torch.view_as_real(v).double() * case["scale"]
        v = a.round_().clamp_(-2 ** 31, 2 ** 31 - 1).to(torch.int32)
        del a
    if case["time_slowest"]:
        v = v.permute(2, 0, 1, *range(3, v.dim())).contiguous()
    return v


def _physical_cube(cfg, seed):
    """A cube whose matrix at every (freq, time) is a sample covariance: a
    drifting point source plus receiver noise, and the Gaussian scatter of N
    samples around it (what `synth.visibilities_physical` draws one matrix at
    a time, with the scatter to first order)."""
    F, n, T = cfg.n_freq, cfg.n_inputs, cfg.n_time
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    A = 50.0 + 100.0 * torch.rand((F, n), generator=g, device="cuda", dtype=torch.float64)
    th0 = 2 * math.pi * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    t = torch.arange(T, device="cuda", dtype=torch.float64)
    th = 2 * math.pi * t[:, None] * torch.arange(n, device="cuda") / (n * cfg.t_sky) + th0
    u = torch.polar(torch.ones_like(th), th)                            # [T][n]
    s = A.sqrt()[:, None, :] * u[None]                                  # [F][T][n]
    R = cfg.rho * s[..., :, None] * s[..., None, :].conj()
    R = R + (1 - cfg.rho) * torch.diag_embed(A)[:, None].to(R.dtype)
    z = torch.randn((F, T, n, n, 2), generator=g, device="cuda", dtype=torch.float64)
    H = torch.view_as_complex(z)
    H = (H + H.mH) / 2
    a = torch.sqrt(A[:, None, :, None] * A[:, None, None, :] / cfg.n_samp)
    V = R + a * H
    ii, jj = torch.triu_indices(n, n, device="cuda")
    return V[..., ii, jj].permute(0, 2, 1).contiguous().to(torch.complex64)


def _walk_input(case, seed):
    return synth.random_walk_device(case["n_elem"], case["elem_size"], seed=seed,
                                    floating=case["floating"])


def _batch_specs(case):
    return synth.batch_specs(case["chunks"], case["pick"])


def _batch_input(case, seed):
    """Rounded cubes (16 inputs x 64 time, cut to the chunk's size) and random walks."""
    xs = []
    per_freq = synth.n_products(16) * 64 * 8
    for k, (nb, es, kind) in enumerate(_batch_specs(case)):
        if kind == "vis":
            cfg = synth.VisConfig(-(-nb // per_freq), 16, 64, 2 ** 16, 0.01, seed=seed * 1009 + k)
            cube = bsgpu.reduce_precision_c64(synth.visibilities_torch(cfg), cfg.n_samp, cfg.f)
            xs.append(cube.view(torch.uint8).reshape(-1)[:nb].clone())
        else:
            xs.append(synth.random_walk_torch(nb // es, es, seed=seed * 1009 + k))
    return xs


def _compress_cube(case, vis, **keep):
    N, B = 2.0 ** case["log2n"], case["block_bytes"] // case["elem_size"]
    plain = (case["dtype"] == "f32" and case["elem_size"] == 4 and
             not (case["time_slowest"] or case["compensate"] or case["full_cov"]))
    if plain:
        return bsgpu.compress_vis(vis, N, case["f"], B, **keep)
    return bsgpu.compress_vis_ex(vis, N, case["f"], compensate=case["compensate"],
                                 elem_size=case["elem_size"], block_elems=B,
                                 time_slowest=case["time_slowest"], full_cov=case["full_cov"],
                                 **keep)


def _cube_flags(case):
    return ((bsgpu.VIS_COMPENSATE if case["compensate"] else 0) |
            (bsgpu.VIS_TIME_SLOWEST if case["time_slowest"] else 0) |
            (bsgpu.VIS_FULL_COV if case["full_cov"] else 0))


def _samples(case):
    return case["n_freq"] * synth.n_products(case["n_inputs"]) * case["n_time"]


def _zeros(n):
    return torch.zeros(max(n, 256), dtype=torch.uint8, device="cuda")


def _reader(c):
    """What a reader of stream `c` has: its bytes, its index, room for the elements."""
    return {"stream": c.stream_bytes().clone(), "offsets": c.offsets, "n_elem": c.n_elem,
            "elem_size": c.elem_size, "block_elems": c.block_elems,
            "out": _zeros(c.n_elem * c.elem_size)[:c.n_elem * c.elem_size],
            "ws": bsgpu.new_workspace(bsgpu.workspace_size(
                bsgpu.OP_DECOMPRESS, c.n_elem, c.elem_size, c.block_elems))}


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("cube", "uncube", "round"):
        vis = _cube_input(case, seed)
        shape = (case["n_freq"], case["n_inputs"], case["n_time"])
        es = case["elem_size"]
        B = case["block_bytes"] // es
        if kind == "uncube":
            st.update(_reader(_compress_cube(case, vis)))
        elif kind == "round":
            st["vis"] = vis
            st["ws"] = bsgpu.new_workspace(bsgpu.vis_workspace_size_ex(
                bsgpu.OP_REDUCE_PRECISION, *shape, 4, 0, _cube_flags(case)))
            out = (case["n_freq"], synth.n_products(case["n_inputs"]), case["n_time"])
            st["out"] = torch.zeros(out if vis.dim() == 3 else out + (2,), dtype=vis.dtype,
                                    device="cuda")
        else:
            st["vis"] = vis
            st["out"] = _zeros(bsgpu.compress_bound(_samples(case) * 8 // es, es, B))
            st["ws"] = bsgpu.new_workspace(bsgpu.vis_workspace_size_ex(
                bsgpu.OP_COMPRESS_VIS, *shape, es, B, _cube_flags(case)))
    elif kind == "batch":
        xs = _batch_input(case, seed)
        es = [e for _, e, _ in _batch_specs(case)]
        eng = engine.BatchCodec(xs, es, [case["block_bytes"] // e for e in es])
        eng.stream_arena.zero_()
        eng.dec_arena.zero_()
        st["engine"] = eng
    else:
        x = _walk_input(case, seed)
        es = case["elem_size"]
        B = case["block_bytes"] // es
        if kind == "unwalk":
            c = bsgpu.compress(x, B, es, level=case["level"])
            st.update(_reader(c))
            if not case["index"]:
                st["offsets"] = None
        elif kind == "walk":
            st["x"] = x
            st["out"] = _zeros(bsgpu.compress_bound(case["n_elem"], es, B))
            st["ws"] = bsgpu.new_workspace(bsgpu.workspace_size(bsgpu.OP_COMPRESS, case["n_elem"],
                                                                es, B))
        else:
            st["x"] = x.view({1: torch.uint8, 2: torch.int16, 4: torch.int32, 8: torch.int64}[es])
            st["bits"] = torch.zeros_like(st["x"])
            st["back"] = torch.zeros_like(st["x"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "cube":
        c = _compress_cube(case, st["vis"], out=st["out"], ws=st["ws"])
        return {"stream": c.buf, "nbytes": c.nbytes_dev, "index": c.offsets}
    if kind == "round":
        return bsgpu.reduce_precision(st["vis"], 2.0 ** case["log2n"], case["f"],
                                      compensate=case["compensate"], out=st["out"], ws=st["ws"],
                                      time_slowest=case["time_slowest"],
                                      full_cov=case["full_cov"])
    if kind in ("uncube", "unwalk"):
        return bsgpu.decompress(st["stream"], st["stream"].numel(), st["n_elem"], st["elem_size"],
                                st["block_elems"], offsets=st["offsets"], out=st["out"],
                                ws=st["ws"])
    if kind == "walk":
        es = case["elem_size"]
        c = bsgpu.compress(st["x"], case["block_bytes"] // es, es, out=st["out"], ws=st["ws"],
                           level=case["level"])
        return {"stream": c.buf, "nbytes": c.nbytes_dev, "index": c.offsets}
    if kind == "shuffle":
        B = case["block_bytes"] // case["elem_size"]
        bits = bsgpu.bitshuffle(st["x"], B, out=st["bits"])
        return [bits, bsgpu.bitunshuffle(bits, B, out=st["back"])]
    eng = st["engine"]
    eng.compress()
    eng.decompress()
    return {"streams": eng.stream_arena, "nbytes": eng.out_bytes, "index": eng.offsets,
            "back": eng.dec_arena, "status": [eng.status_c, eng.status_d]}


# -- what a pass cannot do without -------------------------------------------

def _ratio(case):
    """Stream bytes per input byte, about: what the format leaves of these data."""
    if case["kind"] in ("cube", "uncube"):
        r = {1e-3: 0.42, 1e-2: 0.364, 0.1: 0.306}[case["f"]]
        return r * (0.78 if case["dtype"] == "i32" else 1.0)
    return {1: 1.0, 2: 0.63, 4: 0.32, 8: 0.165}[case["elem_size"]]


def work(case):
    kind = case["kind"]
    if kind == "batch":
        specs = _batch_specs(case)
        data = sum(b for b, _, _ in specs)
        streams = sum(b * (0.364 if k == "vis" else {2: 0.63, 4: 0.32, 8: 0.165}[e])
                      for b, e, k in specs)
        return {"bytes": int(2 * data + 2 * streams), "flops": 0}
    if kind in ("walk", "unwalk", "shuffle"):
        data = case["n_elem"] * case["elem_size"]
        if kind == "shuffle":
            return {"bytes": 4 * data, "flops": 0}
        return {"bytes": int(data * (1 + _ratio(case))), "flops": 0}
    data = 8 * _samples(case)
    if kind == "uncube":
        return {"bytes": int(data * (1 + _ratio(case))), "flops": 0}
    n = case["n_inputs"]
    flops = 0
    if case["full_cov"]:  # per sample: Cholesky, its inverse and X^H X, 8 real operations each step
        flops = case["n_freq"] * case["n_time"] * (8 * (n ** 3 // 6 + n ** 3 // 6 + n ** 3 // 6))
    return {"bytes": int(data * (2 if kind == "round" else 1 + _ratio(case))), "flops": flops}


# -- the rounding in plain torch ---------------------------------------------

def exact(case, seed):
    """The rounded cube for ``round`` cases (streams and bytes have no exact
    counterpart: they are compared as bytes).  The granularity follows from q
    in float32, as the interface defines it; the rounding itself is in 64
    bits."""
    if case["kind"] != "round" or case["full_cov"] or case["dtype"] != "f32":
        return None
    vis = _cube_input(case, seed)
    if case["time_slowest"]:
        vis = vis.permute(1, 2, 0).contiguous()
    F, P, T = vis.shape
    N, f, n = 2.0 ** case["log2n"], case["f"], case["n_inputs"]
    out = torch.empty((F, P, T), dtype=torch.complex128, device=vis.device)
    ii, jj = torch.triu_indices(n, n, device=vis.device)
    auto = (ii == jj)[:, None]
    for fr in range(F):
        re, im = vis[fr].real.contiguous(), vis[fr].imag.contiguous()
        A = re[ii == jj]                                       # [n][T]
        Ai, Aj = A[ii], A[jj]
        if case["compensate"]:
            om = 1.0 - (re * re + im * im) / (Ai * Aj)
            om = torch.where(om >= 0, om, torch.zeros_like(om))
            m = torch.where(auto, torch.ones_like(om), om).amin(0).clamp(max=1.0)
            c = (6.0 * (f * m.double()) / N).float()[None]
        else:
            c = torch.full((1, T), 6.0 * f / N, dtype=torch.float64, device=vis.device).float()
        q = torch.where(auto, 2.0 * c, c) * Ai * Aj
        usable = (q >= 2.0 ** -126) & torch.isfinite(q)
        mant, e = torch.frexp(torch.where(usable, q, torch.ones_like(q)))
        k = torch.div(e - 1 - (mant == 0.5).to(e.dtype), 2, rounding_mode="floor")
        g = ((k.to(torch.int64) + 1023) << 52).view(torch.float64)     # 2^k from its bits
        g = torch.where(usable, g, torch.zeros_like(g))

        def to_grid(x):
            x = x.double()
            return torch.where(g > 0, torch.round(x / torch.where(g > 0, g, 1.0)) * g, x)
        out[fr] = torch.complex(to_grid(re), torch.where(auto, im.double(), to_grid(im)))
    return out
