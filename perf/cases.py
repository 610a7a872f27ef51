"""The workloads whose time this library is judged by: what a program that
compresses simulation fields, reads them back or checks them asks of it.

A case is a dict of plain values.  `kind` says which calls a pass makes:
  plan        one execution of a captured plan on resident buffers (a time
              series written into the same buffers): the stream
  compress    one dls.compress call of a field held on the device: the stream
  into        the same on buffers that the caller keeps: the stream
  roundtrip   compress, decompress, verify: stream, field, report
  decompress  one stream back into a field
  verify      a reconstruction against its original: the report
  global      the global-basis mode, compression and decompression
A stream comes back as its size and the buffer that holds it (zeros after its
end): the caller's own output buffer, or the archive buffer that a program
using the one-call interface appends it to.  The fields are the package's
seeded stand-ins for simulation output.
"""
import math

import torch

from paper_2601_20113_gb300 import dls, synth, train_rank

PREC = {"fp64": dls.PREC_FP64, "fp32": dls.PREC_FP32, "tf32x3": dls.PREC_TF32X3, "tf32": dls.PREC_TF32,
        "bf16x3": dls.PREC_BF16X3, "bf16": dls.PREC_BF16}
RANK = {"search": dls.RANK_SEARCH, "learned": dls.RANK_LEARNED, "tail": dls.RANK_TAIL}
BOUND = {"abs": dls.EB_ABS, "rel": dls.EB_REL_RANGE, "nrmse": dls.EB_NRMSE}
_model = []


def _case(kind, field, dims, block, eb, bound="abs", prec="fp32", rank="learned", codec=0, dtype="f32", **kw):
    """dims = (nx, ny, nz, nt); eb: relative to the range for "abs" (turned into
    an absolute bound) and "rel", percent for "nrmse"."""
    c = dict(kind=kind, field=field, dtype=dtype, bound=bound, eb=eb, prec=prec, rank=rank, codec=codec)
    c.update(zip(("nx", "ny", "nz", "nt"), dims))
    c.update(zip(("bx", "by", "bz", "bt"), block))
    c.update(kw)
    return c


B16 = (16, 16, 16, 16)


def listed():
    return [
        # An in-situ compressor at scale: 4 GiB of resident float32 field, learned rank, one captured plan.
        dict(_case("plan", "modes3d", (256, 256, 256, 64), B16, 1e-3), name="insitu_4GiB"),
        # An archive at a tight bound, with the lossless stage; the modes need the Rayleigh-Ritz pass.
        dict(_case("plan", "modes3d", (256, 256, 64, 64), B16, 1e-4, rank="tail", codec=1), name="archive_tight_1GiB"),
        # Five variables on a grid that neither the blocks nor 16-byte lines divide, a bound per variable.
        dict(_case("plan", "multivar", (250, 190, 130, 50), B16, 1e-3, bound="rel", eb_last=1e-4), name="uneven_5var"),
        # The one-call interface with split-precision tensor-core products and the bisection it defaults to.
        dict(_case("compress", "modes3d", (128, 128, 128, 32), B16, 1e-3, bound="rel", prec="tf32x3", rank="search"),
             name="search_256MiB"),
        # The paper's own error target (an L2 percentage), no pointwise bound, ragged in every axis.
        dict(_case("compress", "modes3d", (150, 118, 61, 40), (16, 16, 8, 16), 1.0, bound="nrmse", rank="tail"),
             name="nrmse_ragged"),
        # A small two-dimensional float64 run, compressed, read back and checked: the smallest calls.
        dict(_case("roundtrip", "vortex2d", (64, 64, 1, 32), (8, 8, 1, 32), 1e-3, prec="fp64", rank="search", dtype="f64"),
             name="vortex_f64_small"),
        # The plain double-precision method on a float32 field of ordinary size.
        dict(_case("compress", "modes3d", (128, 128, 64, 32), B16, 1e-3, prec="fp64", rank="search"), name="plain_f32_128MiB"),
        # One step of a small simulation into buffers that it keeps: launches and latency.
        dict(_case("into", "modes3d", (64, 64, 64, 32), B16, 1e-3), name="oneshot_32MiB"),
        # Reading the 4 GiB field back.
        dict(_case("decompress", "modes3d", (256, 256, 256, 64), B16, 1e-3), name="read_4GiB"),
        # Reading five variables back from streams with the lossless stage, ragged blocks, a tighter bound.
        dict(_case("decompress", "multivar", (125, 95, 65, 50), B16, 3e-4, bound="rel", rank="tail", codec=1),
             name="read_ragged_rice"),
        # Checking 1 GiB of reconstruction against its original.
        dict(_case("verify", "modes3d", (256, 256, 64, 64), B16, 1e-3, rank="tail"), name="check_1GiB"),
        # Algorithm 1 as printed: one basis per variable, every patch of every snapshot, and back.
        dict(_case("global", "modes3d", (128, 128, 128, 16), (4, 4, 4, 1), 1.0, bound="nrmse", prec="fp64", rank="search"),
             name="global_128MiB"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plan", "plan", "compress", "compress", "into", "roundtrip", "decompress", "verify", "global"])
    if kind == "global":
        m = rng.choice([3, 4, 5])
        dims = tuple(m * _log(rng, 8, 128 // m) for _ in range(3)) + (rng.randint(4, 16),)
        return _case(kind, "modes3d", dims, (m, m, m, 1), rng.choice([0.3, 1.0, 3.0]), bound="nrmse", prec="fp64",
                     rank="search")
    if kind == "roundtrip":
        b = rng.choice([(8, 8, 1, 32), (16, 16, 1, 16), (12, 10, 1, 20)])
        dims = (_log(rng, 48, 256), _log(rng, 48, 256), 1, rng.randint(32, 64))
        return _case(kind, "vortex2d", dims, b, rng.choice([1e-2, 1e-3, 1e-4]), prec="fp64", rank="search", dtype="f64")
    prec = rng.choice(["fp32", "fp32", "fp32", "tf32x3", "bf16x3", "fp64"])
    if kind in ("decompress", "verify"):
        prec = "fp32"
    big = 1 << (24 if prec == "fp64" else 27 if kind != "plan" else 28)          # points
    b = rng.choice([B16, B16, B16, (16, 16, 8, 16), (8, 8, 8, 16), (32, 8, 4, 8), (12, 8, 8, 16), (13, 9, 5, 7)])
    nt = rng.choice([16, 32, 48, 50, 64])
    pts = _log(rng, 1 << 19, big)
    nx = _log(rng, 32, 256)
    ny = _log(rng, 32, 256)
    nz = max(b[2], min(256, pts // (nx * ny * nt)))
    if rng.random() < 0.5:
        nx, ny, nz = (max(16, v // 16 * 16) for v in (nx, ny, nz))
    field = rng.choice(["modes3d", "modes3d", "modes3d", "multivar"])
    if field == "multivar":
        nz = max(b[2], nz // 5)
    rank = "search" if prec == "fp64" else rng.choice(["learned", "tail", "tail", "search"])
    bound = rng.choice(["abs", "abs", "rel", "nrmse"])
    eb = rng.choice([0.1, 1.0]) if bound == "nrmse" else rng.choice([1e-2, 1e-3, 3e-4, 1e-4])
    return _case(kind, field, (nx, ny, nz, nt), b, eb, bound=bound, prec=prec, rank=rank,
                 codec=rng.choice([0, 0, 1]) if kind != "compress" else 0)


def _field(c, seed):
    dims = [c[k] for k in ("nx", "ny", "nz", "nt")]
    if c["field"] == "vortex2d":
        return synth.vortex2d(dims[0], dims[1], dims[3], seed=seed, device="cuda")
    if c["field"] == "multivar":
        return synth.multivar(*dims, seeds=tuple(seed * 8 + i for i in range(5)), device="cuda")
    return synth.modes3d(*dims, seed=seed, device="cuda")


def _params(c, f):
    if c["rank"] == "learned" and not _model:
        dls.set_rank_model(train_rank.load_model())
        _model.append(True)
    nv = f.shape[0]
    eb = [c["eb"]] * nv
    if "eb_last" in c:                       # the last two variables (pressure, temperature) at their own bound
        eb[-2:] = [c["eb_last"]] * 2
    if c["bound"] == "abs":
        eb = [e * float(f[v].max() - f[v].min()) for v, e in enumerate(eb)]
    block = tuple(c[k] for k in ("bx", "by", "bz", "bt"))
    return dls.make_params(tuple(f.shape), f.dtype, block, eb, BOUND[c["bound"]], 16, precision=PREC[c["prec"]],
                           rank_mode=RANK[c["rank"]], corr_codec=c["codec"])


def _buffers(p):
    return (torch.zeros(dls.compress_bound(p), dtype=torch.uint8, device="cuda"),
            torch.empty(dls.workspace_size(p), dtype=torch.uint8, device="cuda"))


def _stream(p, f):
    out, ws = _buffers(p)
    st, nb = dls.compress_into(p, f, out, ws)
    if st != dls.OK:
        raise dls.DlsError(st, "dls_compress")
    return out[:nb].clone()


def prepare(case, seed):
    c, f = dict(case), _field(case, seed)
    s = {"c": c, "field": f}
    if c["kind"] == "global":
        m = c["bx"]
        s["field"] = f[0].contiguous()
        s["out"] = torch.zeros(f.numel() * 4, dtype=torch.uint8, device="cuda")
        s["origins"] = synth.patch_origins((c["nx"], c["ny"], c["nz"]), (m, m, m), 4 * m ** 3, seed=seed)
        return s
    p = s["p"] = _params(c, f)
    if c["kind"] == "plan":
        s["out"], s["ws"] = _buffers(p)
        s["plan"] = dls.CompressPlan(p, f, s["out"], s["ws"])
    elif c["kind"] == "into":
        s["out"], s["ws"] = _buffers(p)
    elif c["kind"] in ("compress", "roundtrip"):
        s["out"] = torch.zeros(dls.compress_bound(p), dtype=torch.uint8, device="cuda")
    elif c["kind"] in ("decompress", "verify"):
        s["comp"] = _stream(p, f)
        s["recon"] = torch.empty_like(f)
        if c["kind"] == "verify":
            dls.decompress(s["comp"], s["recon"])
        else:
            del s["field"]
    return s


def _call(s):
    c, p = s["c"], s["p"]
    return dls.compress(s["field"], tuple(p.block), [p.eb[v] for v in range(p.nvars)], p.eb_type, p.rank_cap,
                        p.precision, p.rank_mode)


def _archived(s, comp):
    s["out"][: comp.numel()].copy_(comp)
    return {"bytes": comp.numel(), "stream": s["out"]}


def run(s):
    kind = s["c"]["kind"]
    if kind == "plan":
        return {"bytes": s["plan"].execute(), "stream": s["out"]}
    if kind == "compress":
        return _archived(s, _call(s))
    if kind == "into":
        st, nb = dls.compress_into(s["p"], s["field"], s["out"], s["ws"])
        if st != dls.OK:
            raise dls.DlsError(st, "dls_compress")
        return {"bytes": nb, "stream": s["out"]}
    if kind == "decompress":
        return {"field": dls.decompress(s["comp"], s["recon"])}
    if kind == "verify":
        return {"report": dls.verify(s["field"], s["recon"], s["comp"])}
    if kind == "global":
        comp = dls.gb_compress(s["field"], s["c"]["bx"], s["c"]["eb"], s["origins"])
        return {**_archived(s, comp), "field": dls.gb_decompress(comp)}
    comp = _call(s)
    rec = dls.decompress(comp)
    return {**_archived(s, comp), "field": rec, "report": dls.verify(s["field"], rec, comp)}


def exact(case, seed):
    """Streams and stream statistics have no value in 64 bits (bytes and counts
    compare as they are).  A reconstruction's is the field itself, from which
    it is off by the compression; the error measures of a verification are
    worked out here from the same two fields."""
    kind = case["kind"]
    if kind in ("plan", "compress", "into"):
        return None
    if kind in ("decompress", "roundtrip", "global"):
        f = _field(case, seed).double()
        return {"field": f[0] if kind == "global" else f}
    s = prepare(case, seed)
    x, y = s["field"].double(), s["recon"].double()
    d = x - y
    se, sx = [d[v].square().sum().item() for v in range(x.shape[0])], [x[v].square().sum().item() for v in range(x.shape[0])]
    none = {k: None for k in ("n_over_bound", "ratio", "n_points", "n_blocks", "n_raw_blocks", "n_corr", "n_esc", "mean_rank",
                              "bytes_header", "bytes_basis", "bytes_coeff", "bytes_corr", "bytes_esc", "bytes_raw",
                              "var_max_abs_err", "var_nrmse", "var_over", "var_eb", "status")}
    return {"report": {**none, "max_abs_err": d.abs().max().item(), "nrmse": 100.0 * math.sqrt(sum(se) / sum(sx)),
                       "sum_sq_err": sum(se), "sum_sq": sum(sx)}}


def work(case):
    """The field read (or written) once and its stream written (or read) once;
    the stream's size from the ratios these fields compress at.  Operations:
    the Gram of each block and, at the rank the bound leaves, projection and
    reconstruction."""
    es = 8 if case["dtype"] == "f64" else 4
    pts = case["nx"] * case["ny"] * case["nz"] * case["nt"] * (5 if case["field"] == "multivar" else 1)
    rel = case["eb"] if case["bound"] != "nrmse" else case["eb"] / 100.0
    ratio = 8.0 if case["kind"] == "global" else min(20.0, max(3.5, 12.5 + 3.8 * math.log(rel / 1e-3)))
    field, stream = pts * es, pts * es / ratio
    if case["kind"] == "global":
        m3 = case["bx"] ** 3
        return {"bytes": field + stream + stream + 2 * field, "flops": 2.0 * pts * m3}
    n = min(case["bt"], case["bx"] * case["by"] * case["bz"])
    r = min(n, max(2.0, -1.7 * math.log10(rel)))
    fwd, back = pts * (n + 1 + 4 * r), pts * 2 * r
    return {"plan": {"bytes": field + stream, "flops": fwd}, "compress": {"bytes": field + stream, "flops": fwd},
            "into": {"bytes": field + stream, "flops": fwd}, "decompress": {"bytes": field + stream, "flops": back},
            "verify": {"bytes": 2 * field, "flops": 6.0 * pts},
            "roundtrip": {"bytes": 4 * field + 2 * stream, "flops": fwd + back + 6.0 * pts}}[case["kind"]]
