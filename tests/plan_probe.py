"""The launch that the library plans for a call (plan_probe.cu, compiled
against the library's own headers and linked to it)."""
import ctypes
import functools
import os
import subprocess

from paper_2508_05773_gb300 import build as native_build

HERE = os.path.dirname(os.path.abspath(__file__))
FAMILIES = ("plain", "discs", "point", "moving")


class _Plan(ctypes.Structure):
    _fields_ = [(k, ctypes.c_int32) for k in ("tps", "bpt", "threads", "family", "rows", "ns", "local", "tiles")]
    _fields_ += [("smem", ctypes.c_int64)]

    def as_dict(self):
        d = {k: int(getattr(self, k)) for k, _ in self._fields_}
        d["family"] = FAMILIES[d["family"]]
        return d


@functools.lru_cache(maxsize=None)
def lib():
    so = native_build.build()
    out = os.path.join(native_build.BUILD, f"plan_probe.{os.getpid()}.so")
    subprocess.run([native_build._nvcc(), *native_build.ARCH, *native_build.NVFLAGS, "-shared",
                    os.path.join(HERE, "plan_probe.cu"), so, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(so),
                    "-o", out], check=True, capture_output=True, text=True)
    L = ctypes.CDLL(out)
    os.unlink(out)
    L.probe_ctx.restype = ctypes.c_void_p
    L.probe_ctx.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int64]
    L.probe_free.argtypes = [ctypes.c_void_p]
    L.probe_single.argtypes = [ctypes.c_void_p] + [ctypes.c_int] * 4 + [ctypes.POINTER(_Plan)]
    L.probe_batch.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.POINTER(_Plan)]
    return L


def single(solver, n_obs, n_pts, S=None, H=None):
    """A live solver's plain solve of n_obs obstacles and n_pts path rows."""
    out = _Plan()
    assert lib().probe_single(solver.ctx, S or solver.S, H or solver.H, n_obs, n_pts, ctypes.byref(out)) == 0
    return out.as_dict()


def batch(solver, insts):
    """A live solver's batch of instance dicts."""
    import paper_2508_05773_gb300 as pkg
    arr = pkg.make_instances(insts)
    out = _Plan()
    assert lib().probe_batch(solver.ctx, ctypes.cast(arr, ctypes.c_void_p), len(insts), ctypes.byref(out)) == 0
    return out.as_dict()


def _shapes(count, *args):
    out = (ctypes.c_int32 * 128)()
    n = count(*args, out, 64)
    return [(out[2 * i], out[2 * i + 1]) for i in range(n)]


def plain_candidates(context, n_obs, n_pts):
    """(lanes, threads) of the shapes that the plain autotuner times."""
    return _shapes(lib().probe_plain_candidates, ctypes.c_void_p(context.ctx), n_obs, n_pts)


def batch_candidates(context):
    return _shapes(lib().probe_batch_candidates, ctypes.c_void_p(context.ctx))


def alignments():
    a, b = ctypes.c_int64(), ctypes.c_int64()
    lib().probe_alignments(ctypes.byref(a), ctypes.byref(b))
    return int(a.value), int(b.value)


class HostContext:
    """A context for planning alone, without a GPU: 152 SMs and the shared
    memory of a GB300 block."""

    def __init__(self, params, max_obstacles=16, max_path_pts=4096, num_sms=152, smem_limit=231424, **kw):
        lib()  # (built before the library is loaded)
        from paper_2508_05773_gb300 import _native
        self._p = _native.params_from_dict(params, max_obstacles, max_path_pts, kw.get("threads_per_sample", 0),
                                           kw.get("block_threads", 0), kw.get("max_batch", 0), 0, 0, 0, 0, 0, 0, 0)
        self.S, self.H = int(params["S"]), int(params["H"])
        self.ctx = lib().probe_ctx(ctypes.byref(self._p), num_sms, smem_limit)

    def close(self):
        lib().probe_free(self.ctx)
