"""Calls of the C entry points on a library that is linked against the recording runtime (runtime.cpp, launches.cu).

Run as a program, in a process of its own without the real library: `calls.py <library> <kind> <count> <seed>` makes
`count` seeded calls of a kind, each with a workspace of exactly the queried size, and prints what they reached outside their
buffers.  Addresses are made up; nothing is dereferenced."""
import ctypes
import math
import random
import sys

F32, BF16 = 0, 1
ACCUMULATE, GRADS_F32 = 1, 2

# Backward calls whose tiles of dU and dV do not fit the machine together, few of one and many of the other: m, k, n, r
WIDE = [(8192, 1500, 6000, 375), (8192, 1504, 6016, 376), (4096, 1024, 4096, 1024), (8192, 768, 3072, 768), (4096, 1280, 5120, 320),
        (4096, 6000, 1500, 375), (4944, 2048, 3768, 512), (2500, 1032, 4104, 520), (8192, 1024, 4096, 512), (8192, 4096, 1024, 512),
        (11209, 3072, 768, 768), (4756, 1728, 6912, 432)]

# Convolution backwards and the bytes that they can do with: N, H, W, C, R, O, kernel, stride, pad
LEAST = [((128, 32, 32, 256, 64, 256, 3, 1, 1), 44040192), ((64, 28, 28, 160, 40, 160, 3, 1, 1), 16001024), ((64, 28, 28, 160, 40, 160, 3, 2, 1), 9979904),
         ((64, 28, 28, 320, 80, 320, 3, 1, 1), 29954048), ((64, 28, 28, 320, 80, 320, 1, 1, 0), 28864512), ((60, 28, 28, 128, 8, 128, 3, 1, 1), 7002112),
         ((30, 16, 16, 96, 48, 64, 3, 1, 1), 10062848), ((8, 9, 11, 72, 24, 40, 3, 2, 1), 508416), ((16, 14, 14, 64, 33, 64, 3, 1, 1), 7207168)]


class Library:
    def __init__(self, path):
        self.L = ctypes.CDLL(path)
        self.L.host_faults.restype = self.L.host_launches.restype = ctypes.c_char_p
        for name in ("pf_lowrank_linear_workspace", "pf_lowrank_linear_grouped_workspace", "pf_lowrank_conv_workspace", "pf_bias_act_bwd_workspace"):
            getattr(self.L, name).restype = ctypes.c_size_t
        self.next = 1 << 40

    def query(self, name, *args):
        i64 = ctypes.c_int64
        return getattr(self.L, name)(*(a if isinstance(a, ctypes.c_int) else i64(a) for a in args))

    def call(self, name, args, scratch):
        """args: int -> int64, ctypes values as they are, (bytes, offset) -> the address of a new buffer `offset` bytes behind a
        256-byte boundary, None -> null.  `scratch`: bytes of the workspace that ends the list, None for an entry without."""
        regions, out = [], []
        for a in list(args) + ([(scratch, 0)] if scratch is not None else []):
            if isinstance(a, tuple):
                regions.append((self.next + a[1], a[0]))
                out.append(ctypes.c_void_p(self.next + a[1]))
                self.next += (a[0] + (1 << 24)) >> 20 << 20
            else:
                out.append(ctypes.c_int64(a) if isinstance(a, int) else ctypes.c_void_p(None) if a is None else a)
        if scratch is not None:
            out.append(ctypes.c_size_t(scratch))
        u64 = ctypes.c_uint64 * len(regions)
        self.L.host_regions(len(regions), u64(*(b for b, _ in regions)), u64(*(n for _, n in regions)))
        status = getattr(self.L, name)(*out, ctypes.c_void_p(None))
        return status, self.L.host_faults().decode(), self.L.host_launches().decode()


def c(v):
    return ctypes.c_int(v)


def linear(lib, m, k, n, r, dtype, *, bwd, stash=True, dX=True, flags=0, act=False, pads=(0,) * 8, offset=0, static=False, must=False):
    """One linear call; pads: elements added to the pitches of x, U, V, y or dY, T, dX, dU, dV; must: the array without
    allocation holds it."""
    size = 2 if dtype == BF16 else 4
    gsize = 4 if flags & GRADS_F32 else size

    def mat(rows, cols, pad, size=size):
        ld = cols + pad
        return [(((rows - 1) * ld + cols) * size, offset * size), ld]

    x, U, V, y, T = mat(m, k, pads[0]), mat(k, r, pads[1]), mat(n, r, pads[2]), mat(m, n, pads[3]), mat(m, r, pads[4])
    sizes = [m, k, n, r, c(dtype)]
    none = [None, 0]
    if not bwd:
        args = x + U + V + ([(n * size, 0) if act else None, c(1)] if act else []) + y + (T if stash else none) + sizes
        if static:
            return lib.call("pf_lowrank_linear_fwd_static", args, None)
        return lib.call("pf_lowrank_linear_fwd_act" if act else "pf_lowrank_linear_fwd", args,
                        lib.query("pf_lowrank_linear_workspace", m, k, n, r, c(dtype), c(0)))
    args = x + U + V + y + (T if stash else none) + (mat(m, k, pads[5]) if dX else none) + mat(k, r, pads[6], gsize) + mat(n, r, pads[7], gsize) + sizes
    return lib.call("pf_lowrank_linear_bwd_ex", args + [ctypes.c_uint(flags)], lib.query("pf_lowrank_linear_workspace", m, k, n, r, c(dtype), c(1)))


def grouped(lib, g, m, k, n, r, dtype, *, bwd, stash=True, dX=True, shared=False, gap=0):
    size = 2 if dtype == BF16 else 4

    def mats(rows, cols, count=g):
        step = rows * cols + gap
        return [(((count - 1) * step + rows * cols) * size, 0), cols, step if count > 1 or g == 1 else 0]

    none = [None, 0, 0]
    x = mats(m, k, 1 if shared else g)
    sizes = [m, k, n, r, c(dtype)]
    T = mats(m, r) if stash else none
    room = lib.query("pf_lowrank_linear_grouped_workspace", c(g), m, k, n, r, c(dtype), c(int(bwd)))
    if not bwd:
        return lib.call("pf_lowrank_linear_grouped_fwd", [c(g)] + x + mats(k, r) + mats(n, r) + mats(m, n) + T + sizes, room)
    return lib.call("pf_lowrank_linear_grouped_bwd", [c(g)] + x + mats(k, r) + mats(n, r) + mats(m, n) + T +
                    (mats(m, k, 1 if shared else g) if dX else none) + mats(k, r) + mats(n, r) + sizes, room)


def conv(lib, N, H, W, C, R, O, kernel, stride, pad, dtype, *, bwd, stash=True, dX=True, flags=0, room=None):
    size = 2 if dtype == BF16 else 4
    gsize = 4 if flags & GRADS_F32 else size
    Ho, Wo = (H + 2 * pad - kernel) // stride + 1, (W + 2 * pad - kernel) // stride + 1
    x, U, V, y, T = ((v * size, 0) for v in (N * H * W * C, kernel * kernel * C * R, O * R, N * Ho * Wo * O, N * Ho * Wo * R))
    sizes = [c(v) for v in (N, H, W, C, R, O, kernel, kernel, stride, pad, dtype)]
    room = room or lib.query("pf_lowrank_conv_workspace", *sizes, c(int(bwd)))
    T = T if stash else None
    if not bwd:
        return lib.call("pf_lowrank_conv_fwd", [x, U, V, y, T] + sizes, room)
    return lib.call("pf_lowrank_conv_bwd_ex", [x, U, V, y, T, (N * H * W * C * size, 0) if dX else None, (kernel * kernel * C * R * gsize, 0),
                                               (O * R * gsize, 0)] + sizes + [ctypes.c_uint(flags)], room)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    step = rng.choice((64, 64, 8, 8, 4, 1))
    return max(1, _log(rng, lo, hi) // step * step)


def draw(rng, kind):
    """Keyword arguments of one call of a kind: linear, linear_f32, grouped, conv or conv_f32, _bwd for the gradients."""
    bwd = kind.endswith("_bwd")
    dtype = F32 if "f32" in kind else BF16
    kw = dict(bwd=bwd, stash=rng.random() < 0.7)
    if bwd:
        kw["dX"] = rng.random() < 0.8
        kw["flags"] = rng.choice((0, 0, ACCUMULATE, GRADS_F32, ACCUMULATE | GRADS_F32))
    if kind.startswith("conv"):
        C = rng.choice((3, 16, 64, 96, 128, 160, 192, 256, 320, 512))
        R, H, stride = max(1, C // rng.choice((2, 4, 4, 8))), _log(rng, 3, 64), rng.choice((1, 1, 1, 2, 3))
        kernel = rng.choice((3, 3, 3, 1, 5))
        W = max(3, H - rng.choice((0, 0, 0, 1, 2)))
        pad = kernel // 2 if W < kernel else rng.choice((kernel // 2, kernel // 2, 0, 1))
        return conv, (_log(rng, 1, 256), H, W, C, R, rng.choice((C, 2 * C, _width(rng, 8, 1024))), kernel, stride, pad, dtype), kw
    k, n = _width(rng, 16, 8192), _width(rng, 16, 8192)
    r = min(k, n, _width(rng, 8, 1024) if rng.random() < 0.5 else max(8, k // 4))
    if kind.startswith("grouped"):
        kw.pop("flags", None)
        return grouped, (rng.choice((1, 2, 3, 4, 8, 16)), _log(rng, 1, 8192), k, n, r, F32 if rng.random() < 0.2 else BF16), \
            dict(kw, shared=rng.random() < 0.5, gap=rng.choice((0, 0, 8, 3)))
    if rng.random() < 0.3:
        kw["pads"] = tuple(rng.choice((0, 0, 8, 1, 4)) for _ in range(8))
    kw["offset"] = rng.choice((0, 0, 0, 8, 1))
    if not bwd:
        kw["act"] = rng.random() < 0.3
        kw["static"] = not kw["act"] and rng.random() < 0.3
    return linear, (_log(rng, 1, 40000), k, n, r, dtype), kw


def fixed(kind):
    if kind in ("linear", "linear_bwd"):          # ragged widths at pitches of whole 16-byte pieces
        for m in (20, 300, 2100, 19500):
            yield linear, (m, 60, 140, 28, BF16), dict(bwd=kind == "linear_bwd", pads=(4,) * 8)
    if kind == "linear":                          # ... which the array without allocation takes too, however many rows
        for shape, pads in (((40000, 512, 2044, 128), (0, 0, 0, 4, 0)), ((200000, 64, 60, 32), (0, 0, 0, 4, 0)), ((600000, 64, 64, 28), (0, 4, 4, 0, 4)),
                            ((1900, 512, 2044, 192), (0, 0, 0, 4, 0)), ((43000, 64, 60, 100), (0, 0, 0, 4, 4)), ((43000, 64, 64, 100), (0, 0, 0, 0, 4)), ((2047, 1500, 1504, 8), (0,) * 8), ((30001, 100, 100, 60), (4,) * 8)):
            yield linear, shape + (BF16,), dict(bwd=False, static=True, must=True, pads=pads, stash=pads[4] != 0)
    if kind == "linear_bwd":
        for shape in WIDE:
            for flags in (0, ACCUMULATE, GRADS_F32):
                yield linear, shape + (BF16,), dict(bwd=True, flags=flags)
            yield linear, shape + (BF16,), dict(bwd=True, stash=False, dX=False)


    if kind == "conv":                            # tall images of few columns, which the boxes of the tensor-core kernels do not reach
        for W, stride in ((4, 4), (3, 3), (1, 3)):
            yield conv, (40, 1400, W, 64, 72, 64, 3, stride, 1, BF16), dict(bwd=False)
    if kind == "conv_bwd":                        # workspaces from before some of these calls had a use for more
        for shape, room in LEAST:
            for flags in (0, ACCUMULATE, GRADS_F32):
                yield conv, shape + (BF16,), dict(bwd=True, flags=flags, room=room)
                yield conv, shape + (BF16,), dict(bwd=True, stash=False, dX=False, flags=flags, room=room)


def main(path, kind, count, seed):
    lib, rng = Library(path), random.Random(f"{kind} {seed}")
    bad = 0
    for fn, args, kw in list(fixed(kind)) + [draw(rng, kind) for _ in range(count)]:
        status, faults, launches = fn(lib, *args, **kw)
        if status == 3 and kw.get("static") and not kw.get("must"):
            continue                              # a problem that the fixed array does not hold is refused
        if kind.startswith("conv") and "simt_gemm_kernel" in launches and "repack" in launches:
            faults += "copies for kernels that decline the call\n"
        if status != 0 or faults or not launches:
            bad += 1
            print(kind, args, kw, "status", status, faults.strip() or "no launch" if not launches else faults.strip())
    print("calls reaching outside their buffers:", bad)


if __name__ == "__main__":
    main(sys.argv[1], sys.argv[2], int(sys.argv[3]), int(sys.argv[4]))
