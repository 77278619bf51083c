"""The library's host code on a CUDA runtime of stand-ins (fake_cuda.cpp): what
it launches, in which shapes, and how it takes failing calls, without a GPU."""
import concurrent.futures as cf
import ctypes
import glob
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(os.path.dirname(HERE))
BUILD = os.path.join(HERE, "_build")
DTYPES = {"u8": 0, "f16": 1, "f32": 2}
ELEM = {"u8": 1, "f16": 2, "f32": 4}
DIRECT, GROUPED, TABLE, H2D = range(4)


class Record(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("kind", "dtype", "dm_per_thread", "dm_warps",
                                            "time_warps", "chan_per_stage", "words", "beams")] + \
        [("tiles", ctypes.c_longlong), ("nsamp_out", ctypes.c_longlong),
         ("null_pointers", ctypes.c_int), ("captured", ctypes.c_int)]

    @property
    def shape(self):
        return (self.dm_per_thread, self.dm_warps, self.time_warps, self.chan_per_stage,
                self.words)


def build() -> str:
    csrc = os.path.join(ROOT, "paper_1111_6399_gb300", "csrc")
    include = os.path.join(ROOT, "include")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    os.makedirs(BUILD, exist_ok=True)
    out = os.path.join(BUILD, "libdd_host.so")
    sources = sorted(glob.glob(os.path.join(csrc, "*.cpp"))) + \
        [os.path.join(HERE, "fake_cuda.cpp")]
    deps = sources + glob.glob(os.path.join(csrc, "*.h")) + glob.glob(os.path.join(include, "*.h"))
    if os.path.exists(out) and all(os.path.getmtime(d) <= os.path.getmtime(out) for d in deps):
        return out
    objs = [os.path.join(BUILD, os.path.basename(s) + ".o") for s in sources]

    def one(job):
        src, obj = job
        subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-ffp-contract=off", "-I", include,
                        "-I", csrc, "-I", os.path.join(cuda, "include"), "-c", src, "-o", obj],
                       check=True)

    with cf.ThreadPoolExecutor(8) as ex:
        list(ex.map(one, zip(sources, objs)))
    # -Bsymbolic: its own runtime, also in a process that has loaded CUDA's.
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", out, *objs, "-lpthread", "-ldl"],
                   check=True)
    return out


class Host:
    """The library on the stand-ins; buffers are addresses that nothing reads."""

    IN, OUT = 1 << 20, 1 << 21

    def __init__(self):
        self.lib = ctypes.CDLL(build())
        self.lib.dd_last_error.restype = ctypes.c_char_p
        self.lib.fake_allocations.restype = ctypes.c_longlong

    def reset(self):
        self.lib.fake_reset()

    def records(self, *kinds):
        buf = (Record * 4096)()
        n = self.lib.fake_records(buf, len(buf))
        return [r for r in buf[:n] if not kinds or r.kind in kinds]

    def plan(self, nchan, fch1, foff, tsamp, dms):
        dms = np.ascontiguousarray(dms, dtype=np.float32)
        p = ctypes.c_void_p()
        st = self.lib.dd_plan(nchan, ctypes.c_double(fch1), ctypes.c_double(foff),
                              ctypes.c_double(tsamp), ctypes.c_void_p(dms.ctypes.data), len(dms),
                              ctypes.byref(p))
        assert st == 0, self.lib.dd_last_error()
        self.lib.dd_plan_maxshift.restype = ctypes.c_int64
        self.lib.dd_plan_maxshift.argtypes = [ctypes.c_void_p]
        return p

    def sizes(self, plan, nsamp_out):
        nin = nsamp_out + self.lib.dd_plan_maxshift(plan)
        return [ctypes.c_int64(v) for v in ((nin + 15) // 16 * 16, nin,
                                            (nsamp_out + 3) // 4 * 4, nsamp_out)]

    def execute(self, plan, dtype, nsamp_out, host=False):
        pin, nin, pout, nout = self.sizes(plan, nsamp_out)
        call = self.lib.dd_execute_host if host else self.lib.dd_execute
        return call(plan, ctypes.c_void_p(self.IN), DTYPES[dtype], pin, nin,
                    ctypes.c_void_p(self.OUT), pout, nout, *([] if host else [None]))

    def batch(self, plans, dtype, lengths):
        b = ctypes.c_void_p()
        arr = (ctypes.c_void_p * len(plans))(*[p.value for p in plans])
        assert self.lib.dd_batch_create(arr, len(plans), DTYPES[dtype], ctypes.byref(b)) == 0
        for i, (p, n) in enumerate(zip(plans, lengths)):
            pin, nin, pout, nout = self.sizes(p, n)
            assert self.lib.dd_batch_set_io(b, i, ctypes.c_void_p(self.IN), pin, nin,
                                            ctypes.c_void_p(self.OUT), pout, nout) == 0
        return b

    def batch_execute(self, batch):
        return self.lib.dd_batch_execute(batch, None)
