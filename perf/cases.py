"""Timed cases of the reduction path: what a program that uses the library has
it do, through the public entry points, from fields whose cost is launches and
latency to the 513^3 field of the benchmark.

Operations (``op``):
  compress    field -> container, waiting for its size ("sync") or queued
              without host waits ("async")
  decompress  container -> field, header read on the host or on the device
  roundtrip   both directions in one pass
  batch       many small and uneven fields in one batched call
  train       recomposition forward and its adjoint backward under autograd,
              as in a loss on the reconstructed field
  lossless    byte or 16-bit keys -> container -> keys
  zfp         fixed-rate container and back
  host        host-resident field -> streamed container -> host field

``exact`` is the method restated in plain binary64 torch: canonical Huffman
decoding of every chunk in lockstep, the multilevel transform with dense 1-D
operators, and fixed-rate ZFP decoding one bit of every block at a time.
"""
import math
import struct

import numpy as np
import torch

from paper_2503_06322_gb300 import autograd, fields, hpdr

# Container bits per value of power-law fields at each relative bound, for work().
BITS = {1e-2: 9.5, 1e-3: 12.5, 1e-4: 19.5}
DTYPES = {"f32": torch.float32, "f64": torch.float64}


def listed():
    return [
        # a slice or a diagnostic written every step: the calls' latency
        dict(name="roundtrip_129x129_f32", op="roundtrip", dims="129x129", dtype="f32", tol=1e-3, mode=0, call="sync", grid="uniform"),
        # one rank's block of a decomposed domain, ragged in every dimension
        dict(name="roundtrip_130x67x45_f32", op="roundtrip", dims="130x67x45", dtype="f32", tol=1e-4, mode=0, call="async", grid="uniform"),
        # the benchmark's field (NYX-like): bulk compression and decompression queued on a stream
        dict(name="compress_513_f32", op="compress", dims="513x513x513", dtype="f32", tol=1e-3, mode=0, call="async", grid="uniform"),
        dict(name="decompress_513_f32", op="decompress", dims="513x513x513", dtype="f32", tol=1e-3, mode=0, call="async", grid="uniform"),
        # odd sizes at a tight bound: most codes leave the dictionary and are escaped
        dict(name="compress_300x431x517_f32", op="compress", dims="300x431x517", dtype="f32", tol=1e-4, mode=0, call="sync", grid="uniform"),
        dict(name="decompress_300x431x517_f32", op="decompress", dims="300x431x517", dtype="f32", tol=1e-4, mode=0, call="sync", grid="uniform"),
        # binary64 simulation output, non-dyadic sizes
        dict(name="roundtrip_500x500x100_f64", op="roundtrip", dims="500x500x100", dtype="f64", tol=1e-3, mode=0, call="async", grid="uniform"),
        # many uneven variables of one time step in one call
        dict(name="batch_48_fields_f32", op="batch", count=48, mix=3, lo=17, hi=513),
        # a training step through the transform
        dict(name="train_257_f32", op="train", dims="257x257x257", dtype="f32"),
        # keys of another quantizer through the entropy stage alone
        dict(name="lossless_64Mi_u8", op="lossless", n=1 << 26, key=1, scale=6.0),
        # fixed-rate storage of the same kind of field
        dict(name="zfp_300x431x517_f32_rate8", op="zfp", dims="300x431x517", dtype="f32", rate=8),
        # host-resident field in 64 MiB slabs: copies and kernels overlapped
        dict(name="host_513_f32_64MiB", op="host", dims="513x513x513", dtype="f32", tol=1e-3, slab=64 << 20),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _some_dims(rng, lo, hi, nd=None):
    """2-D or 3-D sizes with log-uniform node counts in [lo, hi] and uneven
    sides; whatever comes out, odd or even."""
    nd = nd or rng.choice((2, 3, 3))
    n = _log(rng, lo, hi)
    skew = [rng.uniform(-0.5, 0.5) for _ in range(nd)]
    mid = sum(skew) / nd
    dims = [max(5, int(n ** (1.0 / nd) * math.exp(s - mid))) for s in skew]
    if nd == 2:
        dims = [min(d, 8192) for d in dims]
    return "x".join(str(d) for d in dims)


def draw(rng):
    op = rng.choices(("compress", "decompress", "roundtrip", "batch", "train", "lossless", "zfp", "host"),
                     (6, 6, 4, 2, 2, 2, 1, 1))[0]
    tol = rng.choice((1e-2, 1e-3, 1e-4))
    dtype = rng.choice(("f32", "f32", "f32", "f64"))
    if op in ("compress", "decompress", "roundtrip"):
        hi = {"f32": 1.3e8, "f64": 2.4e7}[dtype]
        call = rng.choice(("sync", "async"))
        return dict(op=op, dims=_some_dims(rng, 2e3, hi / (2 if op == "roundtrip" else 1)), dtype=dtype, tol=tol,
                    mode=rng.choice((0, 0, 0, 1, 2)), call=call,
                    grid="stretched" if call == "sync" and rng.random() < 0.3 else "uniform")
    if op == "batch":
        return dict(op=op, count=rng.randint(4, 48), mix=rng.randint(4, 1000), lo=17, hi=int(_log(rng, 65, 385)))
    if op == "train":
        return dict(op=op, dims=_some_dims(rng, 2e3, 1.6e7 if dtype == "f32" else 4e6), dtype=dtype)
    if op == "lossless":
        key = rng.choice((1, 2))
        return dict(op=op, n=int(_log(rng, 1e4, 6e7)), key=key, scale=round(_log(rng, 2.0, 10.0 if key == 1 else 60.0), 2))
    if op == "zfp":
        return dict(op=op, dims=_some_dims(rng, 2e3, 6e7 if dtype == "f32" else 3e7, 3), dtype=dtype, rate=rng.choice((8, 16)))
    return dict(op=op, dims=_some_dims(rng, 4e6, 1.2e8, 3), dtype="f32", tol=tol, slab=rng.choice((32, 64, 128, 256)) << 20)


# ---------------------------------------------------------------------------
def _shape(case):
    return tuple(int(x) for x in case["dims"].split("x"))


def _field(shape, seed, dtype="f32"):
    """Power-law random field of zero mean and unit variance."""
    return fields.powerlaw_field_torch(shape, seed=seed, dtype=DTYPES[dtype])


def _batch_shapes(case):
    return fields.batch_shapes(case["count"], seed=case["mix"], lo=case["lo"], hi=case["hi"])


def prepare(case, seed):
    op = case["op"]
    s = {"op": op}
    if op in ("compress", "decompress", "roundtrip"):
        shape = _shape(case)
        u = _field(shape, seed, case["dtype"])
        coords = fields.node_coords(shape, seed, "stretched") if case["grid"] == "stretched" else None
        s.update(call=case["call"], tol=case["tol"], mode=case["mode"], coords=coords)
        if op == "decompress":
            s["buf"] = hpdr.hpdr_compress(u, case["tol"], mode=case["mode"], coords=coords).clone()
        else:
            s["u"] = u
        if op != "compress":
            s["rec"] = torch.empty_like(u)
        if case["call"] == "async":
            s["result"] = torch.zeros(2, dtype=torch.int64, device="cuda")
            s["status"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        if op != "decompress":
            s["out"] = torch.zeros(hpdr.hpdr_compress_bound(shape, u.dtype), dtype=torch.uint8, device="cuda")
    elif op == "batch":
        mix = _batch_shapes(case)
        s["fields"] = [_field(dims, 1000 * seed + i) for i, (dims, _) in enumerate(mix)]
        s["tols"] = [t for _, t in mix]
        cap = hpdr.batched_capacity([(u.shape, u.dtype) for u in s["fields"]])
        s["out"] = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    elif op == "train":
        shape = _shape(case)
        s["shape"] = shape
        s["coef"] = hpdr.hpdr_decompose(_field(shape, seed, case["dtype"])).requires_grad_(True)
        s["target"] = _field(shape, seed + 1, case["dtype"])
    elif op == "lossless":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        x = torch.empty(case["n"], device="cuda").exponential_(generator=g)
        x.sub_(torch.empty_like(x).exponential_(generator=g)).mul_(case["scale"]).round_()
        s["keys"] = ((x + 128).clamp_(0, 255).to(torch.uint8) if case["key"] == 1
                     else x.clamp_(-32768, 32767).to(torch.int16))
        s["out"] = torch.zeros(hpdr.lossless_bound(case["n"], case["key"]), dtype=torch.uint8, device="cuda")
        s["rec"] = torch.empty_like(s["keys"])
    elif op == "zfp":
        s["u"] = _field(_shape(case), seed, case["dtype"])
        s["rate"] = case["rate"]
        s["out"] = torch.zeros(hpdr.zfp_bound(s["u"].shape, case["rate"], s["u"].dtype), dtype=torch.uint8, device="cuda")
        s["rec"] = torch.empty_like(s["u"])
    else:
        shape = _shape(case)
        u = _field(shape, seed)
        s["u"] = torch.empty(shape, dtype=u.dtype, pin_memory=True)
        s["u"].copy_(u)
        s.update(tol=case["tol"], slab=case["slab"])
        s["out"] = torch.zeros(hpdr.streamed_bound(shape, u.dtype, case["slab"]), dtype=torch.uint8, pin_memory=True)
        s["rec"] = torch.empty(shape, dtype=u.dtype, pin_memory=True)
    return s


def _compress(s):
    """(container, bytes): the queued call leaves {bytes, status} on the device."""
    if s["call"] == "async":
        hpdr.hpdr_compress_async(s["u"], s["tol"], s["out"], s["result"], mode=s["mode"])
        return s["out"], s["result"]
    buf = hpdr.hpdr_compress(s["u"], s["tol"], mode=s["mode"], coords=s["coords"], out=s["out"])
    return buf, buf.numel()


def _decompress(s, buf):
    if s["call"] == "async":
        hpdr.hpdr_decompress_async(buf, s["rec"], s["status"])
        return s["rec"]
    return hpdr.hpdr_decompress(buf, out=s["rec"])


def run(state):
    """One pass.  Containers are returned as the whole buffer that the program
    keeps for them, cleared when it was made, beside their size."""
    s, op = state, state["op"]
    if op == "compress":
        _, n = _compress(s)
        return {"container": s["out"], "bytes": n}
    if op == "decompress":
        return {"field": _decompress(s, s["buf"])}
    if op == "roundtrip":
        buf, n = _compress(s)
        return {"container": s["out"], "bytes": n, "field": _decompress(s, buf)}
    if op == "batch":
        out, offs, sizes = hpdr.hpdr_compress_batched(s["fields"], s["tols"], out=s["out"])
        return {"containers": out, "offsets": np.array(offs), "bytes": np.array(sizes)}
    if op == "train":
        s["coef"].grad = None
        u = autograd.recompose(s["coef"], s["shape"])
        loss = (u - s["target"]).square().mean()
        loss.backward()
        return {"field": u.detach(), "loss": loss.detach(), "grad": s["coef"].grad}
    if op == "lossless":
        buf = hpdr.hpdr_lossless_compress(s["keys"], out=s["out"])
        return {"container": s["out"], "bytes": buf.numel(), "keys": hpdr.hpdr_lossless_decompress(buf, out=s["rec"])}
    if op == "zfp":
        buf = hpdr.hpdr_zfp_compress(s["u"], s["rate"], out=s["out"])
        return {"container": s["out"], "field": hpdr.hpdr_zfp_decompress(buf, out=s["rec"])}
    buf = hpdr.hpdr_compress_host_streamed(s["u"], s["tol"], slab_bytes=s["slab"], out=s["out"])
    return {"container": s["out"], "bytes": buf.numel(), "field": hpdr.hpdr_decompress_host_streamed(buf, out=s["rec"])}


def work(case):
    """Bytes in and out once each; about 40 operations a node and direction
    for the transform (interpolation, five-tap restriction and line solves)."""
    op = case["op"]
    if op == "batch":
        b = f = 0
        for dims, tol in _batch_shapes(case):
            n = math.prod(dims)
            b += n * (4 + BITS[tol] / 8)
            f += 40 * n
        return {"bytes": b, "flops": f}
    if op == "lossless":
        bits = math.log2(2 * math.e * case["scale"]) + 0.05     # entropy of a Laplacian in steps of one
        return {"bytes": 2 * case["n"] * (case["key"] + bits / 8), "flops": 0}
    n = math.prod(_shape(case))
    size = 8 if case["dtype"] == "f64" else 4
    if op == "train":       # coefficients and target in, field and gradient out
        return {"bytes": 4 * n * size, "flops": 80 * n}
    if op == "zfp":
        return {"bytes": 2 * n * (size + case["rate"] / 8), "flops": 0}
    ways = 1 if op in ("compress", "decompress") else 2
    return {"bytes": ways * n * (size + BITS[case["tol"]] / 8), "flops": ways * 40 * n}


# ---------------------------------------------------------------------------
# The method in binary64 torch.
def _hierarchy(xs):
    """[finest, ..., coarsest] coordinates of every dimension: one coarsening
    keeps every other node and the last one, until a dimension has two."""
    out = [xs]
    while all(len(x) > 2 for x in out[-1]):
        out.append([torch.cat([x[0:len(x) - 1:2], x[-1:]]) for x in out[-1]])
    return out


def _operators(xf, xc):
    """Dense 1-D prolongation P and correction (P^T M_f P)^-1 P^T M_f."""
    m, mc = len(xf), len(xc)
    pos = torch.arange(mc, device=xf.device) * 2
    pos[-1] = m - 1
    P = torch.zeros(m, mc, dtype=torch.float64, device=xf.device)
    P[pos, torch.arange(mc, device=xf.device)] = 1.0
    kept = torch.zeros(m, dtype=torch.bool, device=xf.device)
    kept[pos] = True
    new = (~kept).nonzero().reshape(-1)
    j = new // 2
    h = xc[j + 1] - xc[j]
    P[new, j] = (xc[j + 1] - xf[new]) / h
    P[new, j + 1] = (xf[new] - xc[j]) / h
    d = xf[1:] - xf[:-1]
    M = torch.diag(torch.cat([d, d[:0].new_zeros(1)]) / 3 + torch.cat([d[:0].new_zeros(1), d]) / 3)
    M += torch.diag(d / 6, 1) + torch.diag(d / 6, -1)
    return P, torch.linalg.solve(P.T @ M @ P, P.T @ M), kept


def _along(A, v, k):
    return torch.movedim(torch.tensordot(A, v, dims=([1], [k])), 0, k)


def _recompose64(coef, xs):
    """Field of a level-major coefficient stream on the grid of xs."""
    grids = _hierarchy(xs)
    at = math.prod(len(x) for x in grids[-1])
    v = coef[:at].reshape([len(x) for x in grids[-1]])
    for xf, xc in zip(grids[-2::-1], grids[:0:-1]):
        ops = [_operators(a, b) for a, b in zip(xf, xc)]
        kept = ops[0][2]
        for o in ops[1:]:
            kept = kept.unsqueeze(-1) & o[2]
        new = (~kept).reshape(-1).nonzero().reshape(-1)
        w = torch.zeros(kept.numel(), dtype=torch.float64, device=coef.device).index_put((new,), coef[at:at + len(new)])
        w = w.reshape(kept.shape)
        at += len(new)
        z = w
        for k, o in enumerate(ops):
            z = _along(o[1], z, k)
        v = v - z
        for k, o in enumerate(ops):
            v = _along(o[0], v, k)
        v = v + w
    return v


def _window(words, p):
    """62 bits from bit position p (most significant bit of a word first)."""
    i = (p >> 5).clamp_(max=len(words) - 3)
    off = p & 31
    a, b, c = words[i], words[i + 1], words[i + 2]
    hi = ((a << off) | (b >> (32 - off))) & 0xFFFFFFFF
    lo = ((b << off) | (c >> (32 - off))) & 0xFFFFFFFF
    return (hi << 30) | (lo >> 2)


def _dequantized(buf):
    """(coefficients, coordinates) that a container stands for."""
    head = bytes(buf[:128].cpu().numpy())
    _, ndim = struct.unpack_from("<II", head, 8)
    dims = struct.unpack_from("<3Q", head, 16)[:ndim]
    L, _, kind, D, K, s_lo = struct.unpack_from("<6I", head, 40)
    N, escapes, bits = struct.unpack_from("<3Q", head, 96)
    s_hi, W = struct.unpack_from("<HB", head, 120)
    at = 128
    q = buf[at:at + 8 * (L + 1)].clone().view(torch.float64)
    at += 8 * (L + 1)
    if kind & 0x100:
        flat = buf[at:at + 8 * sum(dims)].clone().view(torch.float64)
        xs = list(flat.split(list(dims)))
        at += 8 * sum(dims)
    else:
        xs = [torch.arange(d, dtype=torch.float64, device=buf.device) for d in dims]
    up = lambda v: (v + 15) & ~15   # noqa: E731
    at = up(at)
    lens = buf[at:at + s_hi - s_lo + 1].to(torch.int64)
    at = up(at + s_hi - s_lo + 1)
    chunks = -(-N // K)
    p = buf[at:at + 8 * chunks].clone().view(torch.int64).clone()
    at = up(at + 8 * chunks)
    words = buf[at:at + 4 * (-(-bits // 32))].clone().view(torch.int32).to(torch.int64) & 0xFFFFFFFF
    words = torch.cat([words, words.new_zeros(3)])
    # canonical codes in (length, symbol) order, aligned to the top of 62 bits
    order = sorted((int(n), i + s_lo) for i, n in enumerate(lens.tolist()) if n)
    code, prev, starts = 0, order[0][0], []
    for n, _ in order:
        code <<= n - prev
        prev = n
        starts.append(code << (62 - n))
        code += 1
    starts = torch.tensor(starts, device=buf.device)
    length = torch.tensor([n for n, _ in order], device=buf.device)
    symbol = torch.tensor([x for _, x in order], device=buf.device)
    codes = torch.empty(K, chunks, dtype=torch.int64, device=buf.device)
    for t in range(K):
        at_code = torch.searchsorted(starts, _window(words, p), right=True) - 1
        sym = symbol[at_code]
        p += length[at_code]
        k = sym - D // 2
        if escapes:
            z = _window(words, p) >> (62 - W)
            esc = sym == 0
            k = torch.where(esc, (z >> 1) ^ -(z & 1), k)
            p += esc * W
        codes[t] = k
    codes = codes.t().reshape(-1)[:N].to(torch.float64)
    at = 0
    for l, xl in enumerate(_hierarchy(xs)[::-1]):
        end = math.prod(len(x) for x in xl)
        codes[at:end] *= q[l]
        at = end
    return codes, xs


def _zfp64(buf, dims, dtype, rate):
    """Fixed-rate ZFP decoding, one bit of every block at a time."""
    d, dev = len(dims), buf.device
    P, EB = (32, 9) if dtype == "f32" else (64, 12)
    B, bits = 4 ** d, rate * 4 ** d
    nbk = [-(-n // 4) for n in dims]
    nb = math.prod(nbk)
    words = buf[64:64 + nb * bits // 8].clone().view(torch.int32).reshape(nb, bits // 32).t().to(torch.int64)
    u = torch.zeros(nb, B, dtype=torch.int64, device=dev)
    flat, row = u.reshape(-1), torch.arange(nb, device=dev) * B
    n = torch.zeros(nb, dtype=torch.int64, device=dev)      # coefficients already significant
    i, k = n.clone(), torch.full_like(n, P - 1)             # next coefficient, plane
    scan = torch.zeros(nb, dtype=torch.bool, device=dev)    # after a positive group test
    emax = n.clone()
    live = (words[0] & 1) == 1
    for t in range(1, bits):
        bit = (words[t >> 5] >> (t & 31)) & 1
        if t <= EB:
            emax += bit << (t - 1)
            continue
        on = live & (k >= 0)
        verb = on & (i < n)
        test = on & ~verb & ~scan
        run_ = on & ~verb & scan
        put = verb | run_
        flat.index_add_(0, (row + i).clamp_(max=flat.numel() - 1), torch.where(put, bit << k.clamp(min=0), 0))
        i = i + put.to(torch.int64)
        n = torch.maximum(n, i)
        scan = torch.where(test, bit == 1, scan & ~(run_ & (bit == 1)))
        over = on & ~scan & (i >= n) & ((test & (bit == 0)) | (n >= B))
        scan = scan & (n < B)
        over = over | (on & (i >= B))
        k = k - over.to(torch.int64)
        i = torch.where(over, 0, i)
    M = 0xAAAAAAAA if P == 32 else -0x5555555555555556
    q = (u ^ M) - M
    if P == 32:
        q = ((q & 0xFFFFFFFF) ^ 0x80000000) - 0x80000000
    cls = (0, 1, 2, 2)
    perm = sorted(range(B), key=lambda j: (sum(cls[(j >> (2 * m)) & 3] for m in range(d)), j))
    blk = torch.empty_like(q)
    blk[:, torch.tensor(perm, device=dev)] = q
    blk = blk.reshape([nb] + [4] * d)

    def pair(s, e):
        x = s + ((e + (e & 1)) >> 1)
        return x, x - e

    for ax in range(1, d + 1):
        S, D, d0, d1 = blk.unbind(ax)
        s0, s1 = pair(S, D)
        blk = torch.stack(pair(s0, d0) + pair(s1, d1), ax)
    e = (emax - (1 << (EB - 1)) - (P - 5)).to(torch.float64).reshape([nb] + [1] * d)
    v = torch.where(live.reshape(e.shape), blk.to(torch.float64) * torch.exp2(e), 0.0)
    v = v.reshape(nbk + [4] * d).permute([x for m in range(d) for x in (m, d + m)]).reshape([4 * b for b in nbk])
    return v[tuple(slice(0, m) for m in dims)].contiguous()


def exact(case, seed):
    op = case["op"]
    if op in ("compress", "batch", "lossless"):
        return None                                        # bytes and keys
    if op == "train":
        s = prepare(case, seed)
        c = s["coef"].detach().double().requires_grad_(True)
        xs = [torch.arange(n, dtype=torch.float64, device="cuda") for n in s["shape"]]
        u = _recompose64(c, xs)
        loss = (u - s["target"].double()).square().mean()
        loss.backward()
        return {"field": u.detach(), "loss": loss.detach(), "grad": c.grad}
    s = prepare(case, seed)
    if op == "decompress":
        return {"field": _recompose64(*_dequantized(s["buf"]))}
    r = run(s)                                             # its container is the input of the way back
    torch.cuda.synchronize()
    if op == "zfp":
        return {"container": None, "field": _zfp64(r["container"], _shape(case), case["dtype"], case["rate"])}
    if op == "roundtrip":
        return {"container": None, "bytes": None, "field": _recompose64(*_dequantized(r["container"]))}
    buf = r["container"]
    slabs, = struct.unpack_from("<I", bytes(buf[:64].numpy()), 8)
    parts = []
    for j in range(slabs):
        at, size = struct.unpack_from("<2Q", bytes(buf[64 + 32 * j:96 + 32 * j].numpy()), 16)
        parts.append(_recompose64(*_dequantized(buf[at:at + size].cuda())))
    return {"container": None, "bytes": None, "field": torch.cat(parts)}
