"""Plan-time decisions of libdd.so on a machine without a GPU: a child process
preloads fake_cudart.c, makes plans and batches and reports what they start
with. (Run as a program this file is that child.)"""
import ctypes
import json
import os
import subprocess
import sys
import types

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
PACKAGE = "paper_1601_05052_gb300"
# band: lowest channel MHz, band top MHz, sampling time s, trial DM step
BANDS = {"lband": (1400.0, 1500.0, 64e-6, 0.5), "apertif": (1420.0, 1720.0, 50e-6, 0.25),
         "wide": (1250.0, 1550.0, 100e-6, 0.25), "lowfreq": (120.0, 180.0, 204.8e-6, 0.05),
         "lofar": (138.0, 144.25, 5e-6, 0.25)}


def probe(requests, tmp_path):
    """Answers of the child to each request {"setups": [[band, beams, channels,
    trials, samples, type], ...] or "tables": [[delays, samples, type], ...], "set": variant of the first plan,
    "refuse": variant that it refuses, "transposed": variant and launch order that
    a tuning cache holds for its adjoint's plan, "ask": [...]}."""
    from paper_1601_05052_gb300 import _build
    _build.build()
    so = os.path.join(str(tmp_path), "libfake_cudart.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-w", "-o", so,
                    os.path.join(HERE, "fake_cudart.c")], check=True)
    env = dict(os.environ, LD_PRELOAD=so, FAKE_CUDART=so)
    env["DD_TUNE_CACHE"] = os.path.join(str(tmp_path), "tune_cache")
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], input=json.dumps(requests),
                       capture_output=True, text=True, env=env, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout)


class FwdArgsHead(ctypes.Structure):
    """The leading members of a forward kernel's argument (dd_fwd_tile.cuh)."""
    _fields_ = ([("in_", ctypes.c_void_p), ("w", ctypes.c_void_p), ("out", ctypes.c_void_p),
                 ("C", ctypes.c_int32), ("D", ctypes.c_int32),
                 ("S", ctypes.c_int64), ("stride", ctypes.c_int64)]
                + [(n, ctypes.c_int32) for n in
                   "Dt Ts C_pad cch stages warps_dm stage_data stage_offs n_dtiles n_ttiles B "
                   "ttile0 dtile0 grid_tt grid_dt time_major".split()])


class Launch(ctypes.Structure):
    _fields_ = [("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_size_t), ("arg0", ctypes.c_ubyte * 256)]


def _child():
    # the package's binding without its __init__, which needs torch
    pkg = types.ModuleType(PACKAGE)
    pkg.__path__ = [os.path.join(ROOT, PACKAGE)]
    sys.modules[PACKAGE] = pkg
    sys.path.insert(0, ROOT)
    import importlib
    L = importlib.import_module(PACKAGE + "._lib")
    lib = L.load()
    fake = ctypes.CDLL(os.environ["FAKE_CUDART"])
    fake.fake_launch.restype = ctypes.POINTER(Launch)
    fake.fake_upload.restype = ctypes.c_void_p

    def plan(band, beams, chan, dm, out, dtype):
        lo, hi, t_samp, step = BANDS[band]
        f = (ctypes.c_double * chan)(*[lo + c * (hi - lo) / chan for c in range(chan)])
        d = (ctypes.c_double * dm)(*[i * step for i in range(dm)])
        p = ctypes.c_void_p()
        L.check(lib.dd_plan_create(ctypes.byref(p), chan, f, hi - (hi - lo) / chan, t_samp, dm, d,
                                   out, beams, L.DTYPES[dtype]))
        return p

    def variant(fn, *args):
        v = L.Variant()
        L.check(fn(*args, ctypes.byref(v)))
        return list(v.as_tuple())

    def order(p):
        o = ctypes.c_int32()
        L.check(lib.dd_plan_get_launch_order(p, ctypes.byref(o)))
        return o.value

    def launches(call):
        fake.fake_launch_reset()
        L.check(call())
        res = []
        for i in range(fake.fake_launch_count()):
            x = fake.fake_launch(i).contents
            e = {"grid": list(x.grid), "block": list(x.block), "smem": x.smem}
            if x.smem:
                a = FwdArgsHead.from_buffer_copy(bytes(x.arg0))
                e["args"] = {n: getattr(a, n) for n, _ in FwdArgsHead._fields_[3:]}
            res.append(e)
        return res

    def cache_transposed(p, setup, entry):
        """A tuning-cache line for the adjoint's plan: D channels, C trials,
        delays M - delay over the padded input rows."""
        _, beams, chan, dm, _, _ = setup
        sh = (ctypes.c_int32 * (chan * dm))()
        L.check(lib.dd_plan_shifts(p, sh))
        m = (max(sh) + 3) // 4 * 4
        h = 1469598103934665603
        for c in range(chan):
            for d in range(dm):
                for byte in (m - sh[d * chan + c]).to_bytes(4, "little"):
                    h = (h ^ byte) * 1099511628211 % (1 << 64)
        key = "fake/t0/C%d/D%d/S%d/B%d/%x" % (dm, chan, lib.dd_plan_input_stride(p), beams, h)
        with open(os.environ["DD_TUNE_CACHE"], "a") as f:
            f.write(" ".join([key] + [str(x) for x in entry]) + "\n")

    def work_list(b, n):
        """Channels of the plans in the order that a batch's launch takes them."""
        bufs = (ctypes.c_void_p * n)(*[ptr.value] * n)
        L.check(lib.dd_batch_execute(b, bufs, bufs, bufs, None))
        size = ctypes.c_size_t()
        raw = ctypes.string_at(fake.fake_upload(ctypes.byref(size)), size.value)
        step = size.value // n
        return [FwdArgsHead.from_buffer_copy(raw[i * step:]).C for i in range(n)]

    def fits_and_keeps(table, out, dtype):
        """Whether a sub-band variant of the preference list fits a delay
        table's plan, and whether the library says that its sums keep groups."""
        chan, dm = len(table[0]), len(table)
        sh = (ctypes.c_int32 * (chan * dm))(*[x for row in table for x in row])
        p = ctypes.c_void_p()
        L.check(lib.dd_plan_create_from_shifts(ctypes.byref(p), chan, dm, sh, out, 1,
                                               L.DTYPES[dtype]))
        keeps = getattr(lib, "_ZN2dd12keeps_groupsEP9dd_plan_s")
        keeps.restype = ctypes.c_bool
        fits = [lib.dd_plan_set_variant(p, ctypes.byref(L.Variant(*v))) == 0
                for v in ((6, 4, 8, 16, 1, 32, 2), (4, 4, 8, 16, 1, 16, 2), (2, 8, 4, 8, 1, 16, 2),
                          (2, 8, 4, 4, 2, 8, 2))]
        answer = [any(fits), keeps(p)]
        lib.dd_plan_destroy(p)
        return answer

    def tuned(p):
        """What dd_tune settles on where the plan's own tile and order are the
        fastest there is, and the tile in the other order the slowest."""
        v = L.Variant()
        L.check(lib.dd_plan_get_variant(p, ctypes.byref(v)))
        fake.fake_favour(v.dm_per_thread * v.warps_dm, 32 * v.samples_per_thread * v.warps_time,
                         v.chans_per_stage)
        rep = L.TuneReport()
        L.check(lib.dd_tune(p, 400, ctypes.byref(rep)))
        return [variant(lib.dd_plan_get_variant, p), order(p), list(rep.best.as_tuple()), rep.best_ms]

    answers = []
    buf = ctypes.create_string_buffer(4096)
    ptr = ctypes.c_void_p((ctypes.addressof(buf) + 255) & ~255)
    for req in json.loads(sys.stdin.read()):
        if "tables" in req:
            answers.append([fits_and_keeps(*t) for t in req["tables"]])
            continue
        plans = [plan(*s) for s in req["setups"]]
        ans = {"plans": [variant(lib.dd_plan_get_variant, p) for p in plans],
               "orders": [order(p) for p in plans]}
        ask = req.get("ask", [])
        if "set" in req:
            L.check(lib.dd_plan_set_variant(plans[0], ctypes.byref(L.Variant(*req["set"]))))
        if "refuse" in req:
            assert lib.dd_plan_set_variant(plans[0], ctypes.byref(L.Variant(*req["refuse"])))
            ans["message"] = lib.dd_last_error_message().decode()
        if "transposed" in req:
            cache_transposed(plans[0], req["setups"][0], req["transposed"])
        if "adjoint" in ask:
            ans["adjoint"] = variant(lib.dd_adjoint_get_variant, plans[0])
            ans["adjoint_launches"] = launches(
                lambda: lib.dd_adjoint(plans[0], ptr, ptr, ptr, ptr, None, None))
        if "batch" in ask:
            b = ctypes.c_void_p()
            L.check(lib.dd_batch_create(ctypes.byref(b), len(plans),
                                        (ctypes.c_void_p * len(plans))(*[p.value for p in plans])))
            ans["batch"] = variant(lib.dd_batch_get_variant, b)
            ans["batch_channels"] = work_list(b, len(plans))
            lib.dd_batch_destroy(b)
        if "tune" in ask:
            ans["tuned"] = tuned(plans[0])
        if "stream" in ask:
            s = ctypes.c_void_p()
            L.check(lib.dd_stream_create(ctypes.byref(s), plans[0]))
            ans["stream_launches"] = launches(lambda: lib.dd_stream_push(s, ptr, ptr, ptr, None))
            lib.dd_stream_destroy(s)
        for p in plans:
            lib.dd_plan_destroy(p)
        answers.append(ans)
    print(json.dumps(answers))


if __name__ == "__main__":
    _child()
