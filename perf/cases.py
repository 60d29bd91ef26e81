"""What the framework is measured on: applies, solves and DFTs of the operators that it serves.

Operators (plain data, the same for every seed; an uploaded operator is kept and used by all
states of a process, as a program that serves right-hand sides keeps it):
  ex1 / ex2b / ex3   small operators of the paper's examples, by the framework's own builder;
  chain1d            the block shapes of Example 1 at large N without its minutes of host building:
                     ragged blocks of 26 to 90 rows, log2 N butterfly stages, HIF nodes of 64, 26,
                     26 ... unknowns per level and a root of 28.  Unitary blocks, HIF factors near
                     the identity: K-dot is as well conditioned as Example 1's and G-dot as good a
                     preconditioner, so that the solves take the iterations that they take there;
  chain2d            the same with the blocks of Example 3 (200 to 256 rows, HIF cells of 256,
                     edges of about 60, a large root);
  grt256             the shapes of Example 3 at n = 256, the benchmark's operator: 548 million
                     entries in 8 stages of blocks up to 415 x 358, ragged, HIF cells, edges, root.
Right-hand sides are standard complex Gaussians drawn from the seed, as everywhere in this
repository.  A case names the entry point (`call`), the operator, the vectors' type, the precision
and the number of right-hand sides.
"""

import functools
import math
import struct

import numpy as np
import torch

from paper_2105_02995_gb300 import binding
from paper_2105_02995_gb300.builder import build_operator

PRECISION = {"fp64": binding.FIO_P64, "double_float": binding.FIO_PDF, "fp32": binding.FIO_P32,
             "tf32": binding.FIO_PTF32, "bf16": binding.FIO_PBF16, "split_tf32": binding.FIO_PTF32X3}
METHOD = {"pcg": binding.FIO_PCG, "gmres": binding.FIO_GMRES, "ir": binding.FIO_IR}
WIDE = ("fp64", "double_float")  # precisions of complex128 vectors
BUILT = {("ex1", 256): (1e-7, 1e-6), ("ex1", 1024): (1e-7, 1e-6), ("ex1", 4096): (1e-7, 1e-6),
         ("ex2b", 1024): (1e-7, 1e-6), ("ex3", 32): (1e-5, 1e-3)}


def _apply(name, call, op, n, b, prec, tuned=False):
    return {"name": name, "call": call, "op": op, "n": n, "b": b, "prec": prec, "tuned": tuned}


def _solve(name, op, n, b, method, inner, outer):
    return {"name": name, "call": "solve", "op": op, "n": n, "b": b, "method": method, "inner": inner, "outer": outer}


def listed():
    return [
        # the smallest direct solve of the serving mix: one right-hand side, all launches and latency
        _apply("inverse 1D 1024 fp32 b1", "inv", "ex1", 1024, 1, "fp32"),
        # an ordinary served batch on a small operator, host buffers in and out, odd count
        _apply("inverse host 1D 4096 fp32 b13", "inv_host", "ex1", 4096, 13, "fp32"),
        # the solver's default method on one right-hand side in FP64 (a single user's request)
        _solve("gmres 1D 4096 fp64 b1", "ex1", 4096, 1, "gmres", "fp64", "fp64"),
        # the large-N sweep of Example 1: direct solve, complex128, the wide batch
        _apply("inverse 1D 65536 fp64 b64", "inv", "chain1d", 65536, 64, "fp64"),
        # the same sweep in complex64, few right-hand sides, kernels tuned as the sweep does
        _apply("inverse 1D 65536 fp32 b8", "inv", "chain1d", 65536, 8, "fp32", True),
        # the benchmark's headline: generalized Radon transform n = 256, complex64, b = 32, tuned
        _apply("inverse 2D 256 fp32 b32", "inv", "grt256", 256, 32, "fp32", True),
        # the plain FP64 path of the same operator: forward apply of one right-hand side
        _apply("forward 2D 256 fp64 b1", "K", "grt256", 256, 1, "fp64"),
        # its adjoint apply in FP64 for a batch, as the Krylov solvers issue it
        _apply("adjoint 2D 256 fp64 b16", "Kadj", "grt256", 256, 16, "fp64"),
        # the tensor-core arithmetic of refinement's corrections on the same operator
        _apply("inverse 2D 256 split tf32 b32", "inv", "grt256", 256, 32, "split_tf32", True),
        # served solves to 1e-10: refinement with double-float residuals, split-TF32 corrections
        _solve("refinement 2D 128 b32", "chain2d", 128, 32, "ir", "split_tf32", "double_float"),
        # the paper's solver on a ragged batch: PCG in FP64
        _solve("pcg 1D 16384 fp64 b5", "chain1d", 16384, 5, "pcg", "fp64", "fp64"),
        # the last step of the full solve u = K F f: the inverse DFT of a batch
        _apply("inverse DFT 2D 256 fp32 b32", "Finv", "grid2d", 256, 32, "fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "small2d", "chain1d", "chain1d", "chain2d", "chain2d", "solve", "solve", "dft"])
    if kind == "dft":
        op, n = rng.choice([("grid1d", 1 << rng.randint(8, 17)), ("grid2d", 1 << rng.randint(4, 9))])
        return _unnamed(_apply("", rng.choice(["F", "Finv"]), op, n, _log(rng, 1, 48), rng.choice(["fp32", "fp64"])))
    if kind == "solve":
        op, n, b = rng.choice([("chain1d", _log(rng, 2048, 40000), _log(rng, 1, 32)),
                               ("chain2d", rng.randint(48, 128), _log(rng, 1, 32)), ("ex1", 4096, _log(rng, 1, 64))])
        method = rng.choice(["pcg", "gmres", "ir"])
        inner = rng.choice(["fp64", "fp32", "split_tf32"] if method == "ir" else ["fp64", "fp32"])
        return _unnamed(_solve("", op, n, b, method, inner, rng.choice(WIDE) if method == "ir" else "fp64"))
    op, n, most = {"small": ("ex1", rng.choice([256, 1024, 4096]), 128), "small2d": ("ex3", 32, 128),
                   "chain1d": ("chain1d", _log(rng, 1024, 65536), 64),
                   "chain2d": ("chain2d", rng.randint(40, 144), 64)}[kind]
    return _unnamed(_apply("", rng.choice(["K", "Kadj", "G", "inv", "inv_host"]), op, n, _log(rng, 1, most),
                           rng.choice(["fp32", "fp32", "fp64", "fp64", "double_float"])))


def _unnamed(case):
    del case["name"]
    return case


# ---- operators ---------------------------------------------------------------------------------
# A stage: (in-place?, role, in_len, out_len, M complex128 [nblk, R, C], rows read int32 [nblk, C],
# rows written int32 [nblk, R]), -1 and 0 in the padding.

def _sizes(total, nblk, lo, hi, rng):
    """nblk block sizes in lo..hi that add up to total."""
    s = np.clip(np.round(rng.normal(total / nblk, 0.12 * total / nblk, nblk)).astype(np.int64), lo, hi)
    while s.sum() != total:
        d = int(np.sign(total - s.sum()))
        free = np.flatnonzero(s < hi if d > 0 else s > lo)
        at = rng.permutation(free)[:abs(int(total - s.sum()))]
        s[at] += d
    return s


def _even(v):
    return int(v) + (int(v) & 1)


def _lists(order, sizes, width):
    idx = np.full((len(sizes), width), -1, np.int32)
    mask = np.arange(width)[None, :] < sizes[:, None]
    idx[mask] = order[:int(sizes.sum())]
    return idx


def _unitary(size, rng):
    q, _ = np.linalg.qr(rng.standard_normal((size, size)) + 1j * rng.standard_normal((size, size)))
    return q


def _unitary_stage(N, lo, hi, rng):
    """Ragged square unitary blocks between two random orders of the N unknowns."""
    nblk = max(1, round(2 * N / (lo + hi)), -(-N // hi))
    s = _sizes(N, nblk, min(lo, N // nblk), hi, rng)
    w = _even(s.max())
    M = np.zeros((nblk, w, w), np.complex128)
    base = {}
    for k in range(nblk):
        m = int(s[k])
        if m not in base:
            base[m] = _unitary(m, rng)
        phase = np.exp(2j * np.pi * rng.random(2 * m))
        np.multiply(base[m], phase[:m, None], out=M[k, :m, :m])
        M[k, :m, :m] *= phase[m:]
    return (0, 0, N, N, M, _lists(rng.permutation(N).astype(np.int32), s, w),
            _lists(rng.permutation(N).astype(np.int32), s, w))


def _random_stage(in_len, out_len, nblk, rng, pool, ragged):
    """Ragged rectangular blocks of random entries that keep the vectors' size."""
    c, r = in_len / nblk, out_len / nblk
    cs = _sizes(in_len, nblk, int(0.6 * c), int(1.3 * c) + 1, rng) if ragged else np.full(nblk, int(c))
    rs = _sizes(out_len, nblk, int(0.6 * r), int(1.3 * r) + 1, rng) if ragged else np.full(nblk, int(r))
    R, C = _even(rs.max()), _even(cs.max())
    M = np.zeros((nblk, R, C), np.complex128)
    for k in range(nblk):
        m, n = int(rs[k]), int(cs[k])
        at = int(rng.integers(0, len(pool) - m * n))
        np.multiply(pool[at:at + m * n].reshape(m, n), 1 / math.sqrt(max(m, n)), out=M[k, :m, :n])
    return (0, 0, in_len, out_len, M, _lists(rng.permutation(in_len).astype(np.int32), cs, C),
            _lists(rng.permutation(out_len).astype(np.int32), rs, R))


def _hif_stage(N, nblk, lo, hi, role, rng, pool, near):
    """Disjoint blocks near the identity on part of the unknowns."""
    nblk = max(1, min(nblk, N // hi))
    s = rng.integers(lo, hi + 1, nblk)
    w = _even(s.max())
    M = np.zeros((nblk, w, w), np.complex128)
    for k in range(nblk):
        m = int(s[k])
        at = int(rng.integers(0, len(pool) - m * m))
        M[k, :m, :m] = pool[at:at + m * m].reshape(m, m) * (near / math.sqrt(m))
        M[k, range(m), range(m)] += 1
    idx = _lists(rng.permutation(N).astype(np.int32), s, w)
    return (1, role, N, N, M, idx, idx)


def _pool(rng, n):
    return (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * math.sqrt(0.5)


@functools.lru_cache(maxsize=2)
def _stages(op, n):
    """(d, butterfly stages, HIF stages, root) of an operator that this file makes."""
    rng = np.random.Generator(np.random.PCG64(20210506 + n))
    if op == "chain1d":
        N = n
        pool = _pool(rng, 1 << 16)
        bf = [_unitary_stage(N, 16, 16, rng) if N % 16 == 0 else _unitary_stage(N, 12, 18, rng)]
        bf += [_unitary_stage(N, 26, 90, rng) for _ in range(max(2, round(math.log2(N)) - 4))]
        hif, k = [_hif_stage(N, N // 64, 64, 64, 1, rng, pool, 1e-3)], N // 128
        while k >= 2:
            hif.append(_hif_stage(N, k, 23, 28, 1, rng, pool, 1e-3))
            k //= 2
        return 1, bf, hif, [_hif_stage(N, 1, 28, 28, 3, rng, pool, 1e-3)]
    if op == "chain2d":
        N = n * n
        pool = _pool(rng, 1 << 22)
        bf = [_unitary_stage(N, 12, 16, rng)] + [_unitary_stage(N, 200, 256, rng) for _ in range(4)]
        hif = [_hif_stage(N, N // 256, 256, 256, 1, rng, pool, 1e-2), _hif_stage(N, N // 128, 48, 70, 2, rng, pool, 1e-2)]
        side = min(1346, N // 3)
        return 2, bf, hif, [_hif_stage(N, 1, side, side, 3, rng, pool, 1e-2)]
    N = n * n  # grt256
    pool = _pool(rng, 1 << 23)
    lens = [N, N, 256400, 424700, 367000, 420400, 256000, N, N]
    blocks = [N // 16] + [N // 64] * 6 + [N // 16]
    bf = [_random_stage(lens[k], lens[k + 1], blocks[k], rng, pool, 0 < k < 7) for k in range(8)]
    hif = [_hif_stage(N, 256, 256, 256, 1, rng, pool, 0.1), _hif_stage(N, 512, 55, 82, 2, rng, pool, 0.1),
           _hif_stage(N, 64, 360, 420, 1, rng, pool, 0.1), _hif_stage(N, 128, 95, 130, 2, rng, pool, 0.1),
           _hif_stage(N, 16, 420, 466, 1, rng, pool, 0.1), _hif_stage(N, 32, 95, 120, 2, rng, pool, 0.1)]
    return 2, bf, hif, [_hif_stage(N, 1, 1346, 1346, 3, rng, pool, 0.1)]


@functools.lru_cache(maxsize=2)
def _packed(op, n):
    """The operator's packed factor buffer (the format of include/fio.h)."""
    if (op, n) in BUILT:
        return build_operator(op, n, *BUILT[op, n])[0]
    if op in ("grid1d", "grid2d"):  # a DFT needs the grid alone: one stage of scaled identities
        d, N = (1, n) if op == "grid1d" else (2, n * n)
        eye = np.broadcast_to(np.eye(16, dtype=np.complex128), (N // 16, 16, 16))
        idx = np.arange(N, dtype=np.int32).reshape(-1, 16)
        bf, hif, root = [(0, 0, N, N, eye, idx, idx)], [], []
    else:
        d, bf, hif, root = _stages(op, n)
        N = n ** d
    stages = bf + hif + root
    at = -(-(256 + 64 * len(stages)) // 256) * 256
    data, table, places = at, [], []
    for inplace, role, in_len, out_len, M, rows_in, rows_out in stages:
        offs = []
        for a in (M, rows_in, rows_out):
            offs.append(at)
            at += -(-a.nbytes // 256) * 256
        places.append(offs)
        table.append(struct.pack("<IIIIqqQQQII", inplace, *M.shape, in_len, out_len, *offs, 0, role))
    buf = np.zeros(at, np.uint8)
    for offs, st in zip(places, stages):
        for o, a in zip(offs, st[4:]):
            buf[o:o + a.nbytes] = np.ascontiguousarray(a).reshape(-1).view(np.uint8)
    words, total = buf[data:].view(np.uint64), 0
    for k in range(0, len(words), 1 << 24):
        w = words[k:k + (1 << 24)]
        odd = 2 * np.arange(k, k + len(w), dtype=np.uint64) + np.uint64(1)
        total = (total + int(np.sum(w * odd, dtype=np.uint64))) % (1 << 64)
    head = struct.pack("<8sIIqqIIIIddQQQQ", b"FIOPACK1", 1, d, n, N, len(bf), len(hif), len(root), 0, 0.0, 0.0,
                       256, data, at, total)
    buf[:len(head)] = np.frombuffer(head, np.uint8)
    buf[256:256 + 64 * len(table)] = np.frombuffer(b"".join(table), np.uint8)
    return buf.tobytes()


@functools.lru_cache(maxsize=4)
def _operator(op, n):
    handle = binding.Operator(_packed(op, n))
    _packed.cache_clear()
    _stages.cache_clear()
    handle.tuned_for = set()
    return handle


# ---- the cases ---------------------------------------------------------------------------------

def _vectors(case, seed):
    wide = case["call"] == "solve" or case["prec"] in WIDE
    N = case["n"] ** (2 if case["op"] in ("chain2d", "grt256", "grid2d", "ex3") else 1)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dtype = torch.complex128 if wide else torch.complex64
    return torch.randn((case["b"], N), dtype=torch.complex128, device="cuda", generator=g).to(dtype).t()


def prepare(case, seed):
    op = _operator(case["op"], case["n"])
    u = _vectors(case, seed)
    if case["call"] == "solve":
        return {"case": case, "op": op, "u": u}
    prec = PRECISION[case["prec"]]
    if case["tuned"] and (case["b"], prec) not in op.tuned_for:  # once per operator and batch width
        op.autotune(case["b"], prec)
        op.tuned_for.add((case["b"], prec))
    if case["call"] == "inv_host":
        u = np.asfortranarray(u.cpu().numpy())
        return {"case": case, "op": op, "u": u, "f": np.empty_like(u, order="F"), "prec": prec}
    return {"case": case, "op": op, "u": u, "f": torch.empty_like(u.t()).t(), "prec": prec}


def run(state):
    case, op, u = state["case"], state["op"], state["u"]
    call = case["call"]
    if call == "solve":
        f, _ = op.solve(u, method=METHOD[case["method"]], inner=PRECISION[case["inner"]], tol=1e-10, maxit=60,
                        outer=PRECISION[case["outer"]])
        return f
    if call == "inv_host":
        return op.apply_inv_host(u, state["f"], state["prec"])
    if call in ("F", "Finv"):
        return getattr(op, "apply_" + call)(u, state["f"])
    return getattr(op, "apply_" + call)(u, state["f"], state["prec"])


def _shapes(op, n):
    """(butterfly entries, HIF entries, root entries), about, without making the operator."""
    lg = max(2.0, math.log2(n))
    N = n * n if op in ("ex3", "chain2d", "grt256") else n
    if op == "grt256":
        return 548e6, 34e6, 1346.0 ** 2
    if op == "chain2d":
        return N * (14 + 4 * 230.0), N * (256 + 27.0), float(min(1346, N // 3)) ** 2
    if op == "ex3":
        return 1.6e6, 2.6e5, 447.0 ** 2
    if op == "chain1d":
        return N * (16 + 62.0 * max(2, round(lg) - 4)), N * 69.0, 784.0
    return N * (32 + 55.0 * max(2.0, lg - 4)), N * 69.0, 784.0


def work(case):
    b, n = case["b"], case["n"]
    N = n * n if case["op"] in ("ex3", "chain2d", "grt256", "grid2d") else n
    bf, hif, root = _shapes(case["op"], n) if not case["op"].startswith("grid") else (0, 0, 0)
    if case["call"] == "solve":  # the least that reaches 1e-10: two corrections and their residuals
        entry = {"fp64": 16, "fp32": 8, "split_tf32": 8}[case["inner"]]
        return {"bytes": 2 * (16 * bf + entry * (bf + 2 * hif + root)) + 32.0 * N * b,
                "flops": 16.0 * b * (2 * bf + 2 * hif + root)}
    size = 16 if case["prec"] in WIDE else 8
    if case["call"] in ("F", "Finv"):
        return {"bytes": 2.0 * size * N * b, "flops": 5.0 * N * b * math.log2(N)}
    once = {"K": bf, "Kadj": bf, "G": hif + root, "inv": bf + hif + root, "inv_host": bf + hif + root}[case["call"]]
    twice = hif if case["call"] in ("G", "inv", "inv_host") else 0
    return {"bytes": size * once + 2.0 * size * N * b, "flops": 8.0 * b * (once + twice)}


# ---- the same in 64 bits, by torch alone -------------------------------------------------------

def _parse(buf):
    n_bf, n_hif, n_root = struct.unpack_from("<III", buf, 32)
    out = []
    for k in range(n_bf + n_hif + n_root):
        inplace, nblk, R, C, in_len, out_len, om, oi, oo, _, _ = struct.unpack_from("<IIIIqqQQQII", buf, 256 + 64 * k)
        M = torch.frombuffer(buf, dtype=torch.complex128, count=nblk * R * C, offset=om) if nblk else None
        i = torch.frombuffer(buf, dtype=torch.int32, count=nblk * C, offset=oi) if nblk else None
        o = torch.frombuffer(buf, dtype=torch.int32, count=nblk * R, offset=oo) if nblk else None
        if nblk:
            out.append((inplace, M.view(nblk, R, C), i.long().view(nblk, C), o.long().view(nblk, R), in_len, out_len))
        else:
            out.append(None)
    return out[:n_bf], out[n_bf:n_bf + n_hif], out[n_bf + n_hif:]


def _through(stage, x, adjoint):
    if stage is None:
        return x
    inplace, M, rows_in, rows_out, in_len, out_len = stage
    y = x.clone() if inplace else torch.zeros((in_len if adjoint else out_len, x.shape[1]), dtype=x.dtype, device=x.device)
    src, dst = (rows_out, rows_in) if adjoint else (rows_in, rows_out)
    src, dst = src.to(x.device), dst.to(x.device)
    for k in range(0, M.shape[0], 256):
        m, s, d = M[k:k + 256].to(x.device), src[k:k + 256], dst[k:k + 256]
        g = x[s.clamp_min(0)] * (s >= 0).unsqueeze(-1)
        z = torch.matmul(m.mH if adjoint else m, g)
        y[d[d >= 0]] = z[d >= 0]
    return y


def _forward(ops, x):
    for st in ops[0]:
        x = _through(st, x, False)
    return x


def _adjoint(ops, x):
    for st in reversed(ops[0]):
        x = _through(st, x, True)
    return x


def _middle(ops, x):
    for st in ops[1] + ops[2]:
        x = _through(st, x, False)
    for st in reversed(ops[1]):
        x = _through(st, x, True)
    return x


def exact(case, seed):
    u = _vectors(case, seed).to(torch.complex128)
    call = case["call"]
    if call in ("F", "Finv"):
        n = case["n"]
        d = 2 if case["op"] == "grid2d" else 1
        x = u.t().reshape([case["b"]] + [n] * d)
        dims = tuple(range(1, d + 1))
        k = torch.arange(n, device=u.device)
        sign = 1.0 - 2.0 * (k % 2).double()
        sign = sign[:, None] * sign[None, :] if d == 2 else sign
        y = torch.fft.fftn(x * sign, dim=dims) / n ** d if call == "F" else torch.fft.ifftn(x, dim=dims) * n ** d * sign
        return y.reshape(case["b"], -1).t()
    buf = _packed(case["op"], case["n"])
    ops = _parse(bytearray(buf) if case["op"] != "grt256" else buf)
    if call == "solve":
        if case["op"].startswith("chain"):  # unitary
            return _adjoint(ops, u)
        K = _forward(ops, torch.eye(u.shape[0], dtype=torch.complex128, device=u.device))
        return torch.linalg.solve(K, u)
    if call == "K":
        return _forward(ops, u)
    if call == "Kadj":
        return _adjoint(ops, u)
    y = _middle(ops, u if call == "G" else _adjoint(ops, u))
    return y.cpu().numpy() if call == "inv_host" else y
