"""Host side of the context's and the trainer's scratch: what is cleared, allocated and
freed before which launch, on a CUDA runtime without a device (fake_cudart.cpp, preloaded
into a child process) that traces the calls.  No kernel runs."""
import os
import re
import subprocess
import sys
import textwrap

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
    import ctypes, os, sys
    sys.path.insert(0, %r)
    import numpy as np
    from paper_2206_02607_gb300 import crom as c
    from workloads import gen
    fake = ctypes.CDLL(os.environ["LD_PRELOAD"])
    fake.fake_limit.argtypes = [ctypes.c_size_t]
    note = lambda t: fake.fake_note(t.encode())
    S = 0x4440                       # a stream of the caller's, non-blocking
    keep = []
    def arr(a, t):
        keep.append(np.ascontiguousarray(a, dtype=t))
        return keep[-1].ctypes.data
    def ok(rc):
        assert rc == 0, (rc, c.last_error())
    def context(m=2, r=8, width=128, hidden=5):
        h, d = ctypes.c_void_p(), c.crom_decoder_desc(m, r, width, hidden)
        ok(c.raw_call("crom_create", ctypes.byref(h), ctypes.byref(d), 0))
        p = np.ascontiguousarray(gen.pack_params(gen.xavier_decoder(gen.DecoderSpec(m, r, width, hidden), seed=1)), np.float32)
        keep.append(p)
        ok(c.raw_call("crom_set_weights", h, p.ctypes.data, p.size, 0, S))
        return h
    def step(h, sizes, prec, gn=2, r=8, m=2, stream=S, status=0, bound=0):
        n, tot = len(sizes), int(sum(sizes))
        sd = c.crom_step_desc(c.CROM_PDE_HEAT, gn, 1e-5)
        rc = c.raw_call("crom_step", h, ctypes.byref(sd), prec, n, arr(np.zeros((n, r)), np.float64),
                        arr(np.ones(n), np.float32), None, arr(gen.ragged_offsets(np.array(sizes)), np.int32),
                        arr(np.zeros((tot, m)), np.float32), tot, bound or max(sizes), arr(np.zeros(n), np.int32), stream)
        assert rc == status, (rc, c.last_error())
""" % ROOT


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    sys.path.insert(0, ROOT)
    from paper_2206_02607_gb300 import build
    from paper_2206_02607_gb300.build import _nvcc
    build()
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", inc, os.path.join(HERE, "fake_cudart.cpp"), "-o", so,
                    "-ldl"], check=True)
    return so


@pytest.fixture
def trace(fake, tmp_path):
    def run(body):
        log = str(tmp_path / "trace")
        env = dict(os.environ, LD_PRELOAD=fake, FAKE_CUDART_TRACE=log)
        src = textwrap.dedent(PRELUDE) + textwrap.dedent(body)
        res = subprocess.run([sys.executable, "-c", src], env=env, capture_output=True, text=True, timeout=300)
        assert res.returncode == 0, res.stderr[-3000:]
        with open(log) as f:
            return f.read().splitlines()
    return run


def kernels(lines):
    return [re.sub(r"^launch (\S+) .*", r"\1", x) for x in lines if x.startswith("launch ")]


CLEARS = {
    "fp32_few_samples": "step(context(), [200], c.CROM_PREC_FP32)",
    "fp32_batch": "step(context(), [300] * 40, c.CROM_PREC_FP32)",
    "dealt": "step(context(), [4096] * 8, c.CROM_PREC_F16X2)",
    "whole": "step(context(), [64] * 1000, c.CROM_PREC_F16)",
    "reconstruction": """
        h = context()
        ok(c.raw_call("crom_reconstruct", h, c.CROM_PREC_F16X2, 1, arr(np.zeros(8), np.float64), 4096,
                      arr(np.zeros((4096, 2)), np.float32), arr(np.zeros(4096), np.float32), S))
    """,
    "trainer": """
        for prec in (c.CROM_PREC_FP32, c.CROM_PREC_BF16_MIXED):
            for how in ("new", "set", "load"):
                t, d = ctypes.c_void_p(), c.crom_decoder_desc(2, 8, 64, 3)
                ok(c.raw_call("crom_trainer_create", ctypes.byref(t), ctypes.byref(d), 256, 2, 64, 0))
                ok(c.raw_call("crom_trainer_set_precision", t, prec))
                n = ctypes.c_size_t()
                ok(c.raw_call("crom_trainer_param_count", t, ctypes.byref(n)))
                p = arr(np.zeros(n.value), np.float32)
                if how == "set":
                    ok(c.raw_call("crom_trainer_set_params", t, p, n.value, 0, S))
                if how == "load":
                    path = (os.environ["FAKE_CUDART_TRACE"] + ".ckpt").encode()
                    ok(c.raw_call("crom_trainer_save", t, path))
                    ok(c.raw_call("crom_trainer_load", t, path))
                ok(c.raw_call("crom_train_step", t, arr(np.zeros((2, 256)), np.float32), arr(np.zeros((2, 64)), np.int32),
                              arr(np.zeros((256, 2)), np.float32), 1e-3, None, S))
    """,
}


@pytest.mark.parametrize("case", sorted(CLEARS))
def test_clears_and_copies_are_complete_before_the_first_launch(trace, case):
    """The first call of a size on a non-blocking stream: every clear and copy that the
    library made elsewhere is complete before a kernel of the call's stream can use it."""
    lines = trace(CLEARS[case])
    assert kernels(lines)
    assert [x for x in lines if x.startswith("UNORDERED")] == []


@pytest.mark.parametrize("case", sorted(CLEARS))
def test_scratch_is_made_ready_without_a_stream(trace, case):
    """A stream made before a context's or trainer's first launches slows all later ones."""
    assert [x for x in trace(CLEARS[case]) if x.startswith("stream")] == []


@pytest.mark.parametrize("sizes", ["[4096] * 8", "[64] * 1000"])
@pytest.mark.parametrize("prec", ["F16X2", "F16"])
def test_the_timeout_flag_is_cleared_before_the_step_can_set_it(trace, sizes, prec):
    """Dealt form (few instances): a clear of the flag on the step's stream, after the last
    step's launches and before this one's first; whole form: the ordering kernel does it."""
    lines = trace(f"""
        h = context()
        for k in range(2):
            note("step")
            step(h, {sizes}, c.CROM_PREC_{prec})
    """)
    flag = next(x for x in lines if x.startswith("malloc")).split()[1].split("+")[0] + "+4"  # the context's first array
    for part in "\n".join(lines).split("\nstep\n")[1:]:
        part = part.splitlines()
        first = next(i for i, x in enumerate(part) if "step_tc_kernel" in x)
        cleared = [x for x in part[:first] if x.startswith(f"memset {flag} 4 stream 0x4440")]
        assert cleared or any("order_kernel" in x for x in part[:first]), part


STEADY = {
    "dealt_after_whole": ["step(h, [64] * 1000, c.CROM_PREC_F16X2)", "step(h, [1000] * 8, c.CROM_PREC_F16)",
                          "step(h, [1000] * 8, c.CROM_PREC_F16X2)", "step(h, [6000] * 10, c.CROM_PREC_F16X2)"],
    "dealt_after_fp32": ["step(h, [10000], c.CROM_PREC_FP32)", "step(h, [64] * 20, c.CROM_PREC_F16X2, gn=1)",
                         "step(h, [1000] * 8, c.CROM_PREC_F16X2)"],
    "few_samples_fp32": ["step(h, [64] * 1000, c.CROM_PREC_FP32)", "step(h, [200], c.CROM_PREC_FP32)",
                         "step(h, [100] * 3, c.CROM_PREC_FP32)"],
}


@pytest.mark.parametrize("case", sorted(STEADY))
def test_steps_within_earlier_sizes_free_nothing(trace, case):
    """Once a context has stepped a batch of the largest sizes, smaller steps free no
    array, whatever form they take: a graph recorded with any of them stays valid."""
    first, *rest = STEADY[case]
    body = ["h = context()", first, 'note("steady")'] + rest + ['note("end")', 'ok(c.raw_call("crom_destroy", h))']
    lines = trace("\n".join(body))
    a, b = lines.index("steady"), lines.index("end")
    assert [x for x in lines[a:b] if x.startswith("free")] == []
    made = {x.split()[1] for x in lines if x.startswith("malloc #")}
    assert made == {x.split()[1] for x in lines if x.startswith("free #")}      # all given back


def test_a_step_without_room_for_its_rows_takes_the_whole_form(trace):
    """Where the dealt form's rows cannot be allocated, the groups take whole instances
    (which need 8 bytes a sample); with room again, the step is dealt."""
    lines = trace("""
        h = context()
        fake.fake_limit(500000)          # the targets take 262144 bytes, the rows more
        step(h, [4096] * 8, c.CROM_PREC_F16X2)
        note("room")
        fake.fake_limit(1 << 40)
        step(h, [4096] * 8, c.CROM_PREC_F16X2)
    """)
    a = lines.index("room")
    assert any(x.startswith("malloc refused") for x in lines[:a])
    assert [("order" in k) for k in kernels(lines[:a])] == [True, False]
    assert [("order" in k) for k in kernels(lines[a:])] == [False, False]


@pytest.mark.parametrize("warm,call,whole", [("[64] * 1000, c.CROM_PREC_F16X2", "[1000] * 8, c.CROM_PREC_F16X2", True),
                                             ("[64] * 1000, c.CROM_PREC_FP32", "[200], c.CROM_PREC_FP32", False)])
def test_a_recorded_step_within_earlier_sizes_allocates_nothing(trace, warm, call, whole):
    """While the caller records its stream, a step within the sizes of an earlier one
    allocates nothing, although its form has not run before."""
    lines = trace(f"""
        h = context()
        step(h, {warm})
        note("recording")
        fake.fake_capturing(1)
        step(h, {call})
        fake.fake_capturing(0)
    """)
    part = lines[lines.index("recording"):]
    assert not any("malloc" in x for x in part), part
    assert len(kernels(part)) == 2 and ("order" in kernels(part)[0]) == whole


@pytest.mark.parametrize("B,S", [(2, 64), (1, 4000), (64, 4096)])
def test_mixed_precision_buffers_are_of_the_stated_size(trace, B, S):
    """The sizes that crom_trainer_set_precision states: two bytes per point, unit and
    activation array, and a weight gradient's partial sums for the K ranges in use.  A tenth
    more and a megabyte for the column sums and the small arrays."""
    w, L = 256, 5
    lines = trace(f"""
        t, d = ctypes.c_void_p(), c.crom_decoder_desc(2, 8, {w}, {L})
        ok(c.raw_call("crom_trainer_create", ctypes.byref(t), ctypes.byref(d), 4096, {B}, {S}, 0))
        note("mixed")
        ok(c.raw_call("crom_trainer_set_precision", t, c.CROM_PREC_BF16_MIXED))
    """)
    made = sum(int(x.split()[2]) for x in lines[lines.index("mixed"):] if x.startswith("malloc #"))
    stated = (L + 2) * B * S * w * 2 + (L - 1) * min(64, -(-B * S // 64)) * w * w * 4
    assert stated / 2 < made < 1.1 * stated + (1 << 20), (made, stated)


# kind, side, ny, fields, steps, whether the steps are one launch: shapes at which the one
# launch was measured slower than a launch per step (False), and their neighbours
FOM_ROUTES = [("HEAT2D_NEUMANN_FIELD", 127, 10, 4, False), ("HEAT2D_NEUMANN_FIELD", 127, 10, 50, True),
              ("HEAT2D_NEUMANN", 121, 1, 4, False), ("HEAT2D_NEUMANN", 121, 1, 12, True),
              ("HEAT2D_NEUMANN", 97, 10, 8, True), ("ADVDIFF2D_PERIODIC", 99, 10, 4, False),
              ("ADVDIFF2D_PERIODIC_CENTRAL", 97, 10, 8, True), ("HEAT2D_NEUMANN_FIELD", 125, 1000, 1, False),
              ("HEAT2D_NEUMANN_FIELD", 125, 1000, 3, True), ("HEAT2D_NEUMANN", 127, 3000, 1, False),
              ("HEAT2D_NEUMANN", 117, 3000, 1, True), ("ADVDIFF2D_PERIODIC", 180, 300, 1, False),
              ("ADVDIFF2D_PERIODIC", 180, 300, 3, True), ("ADVDIFF2D_PERIODIC", 164, 300, 1, True),
              ("HEAT2D_NEUMANN_FIELD", 180, 600, 1, False), ("HEAT2D_NEUMANN_FIELD", 212, 600, 1, True),
              ("HEAT1D_DIRICHLET_FIELD", 1500, 16000, 1, False), ("HEAT1D_DIRICHLET_FIELD", 700, 8000, 2, False),
              ("HEAT1D_DIRICHLET_FIELD", 1500, 16000, 3, True), ("HEAT1D_DIRICHLET", 1024, 8000, 1, False),
              ("HEAT1D_DIRICHLET", 1024, 16000, 1, True)]


def test_full_order_steps_take_the_faster_launches(trace):
    body = "p = 0x7f0000000000          # not read: no kernel runs\n"
    for kind, n, nb, steps, _ in FOM_ROUTES:
        two_d = not kind.startswith("HEAT1D")
        body += (f'note("shape")\nok(c.raw_call("crom_fom_step", c.CROM_FOM_{kind}, {nb}, {n}, {n if two_d else 1}, '
                 f"p, p, p, 1e-9, {steps}, p, p + (1 << 34), S))\n")
    parts = "\n".join(trace(body)).split("shape")[1:]
    for (kind, n, nb, steps, one), part in zip(FOM_ROUTES, parts, strict=True):
        ks = kernels(part.splitlines())
        got = len(ks) == 1 and any(k in ks[0] for k in ("fom_field", "fom_tile", "fom_wide", "fom_line"))
        assert got == one, (kind, n, nb, steps, ks)
        assert got or len(ks) == steps, (kind, n, nb, steps, ks)


# m, r, width, layers, activation, call, points (or codes x points), the kernel: shapes at
# which the tile kernel was measured slower than the general one, and above the lines
FP32_ROUTES = [(3, 1, 224, 4, 0, "decode 17", 3364, "fwd_fp32"), (3, 1, 224, 4, 0, "decode 17", 4200, "fwd_tile"),
               (2, 2, 128, 3, 0, "decode 16", 3264, "fwd_fp32"), (2, 2, 128, 3, 0, "decode 16", 3800, "fwd_tile"),
               (1, 12, 224, 5, 0, "tangent", 3492, "fwd_fp32"), (1, 12, 224, 5, 0, "tangent", 4500, "fwd_tile"),
               (2, 1, 32, 5, 1, "recon 42", 926, "fwd_fp32"), (2, 1, 32, 5, 1, "recon 42", 3000, "fwd_tile"),
               (2, 1, 32, 5, 0, "recon 42", 926, "fwd_tile"), (3, 4, 64, 1, 0, "decode 27", 3483, "fwd_fp32"),
               (3, 4, 64, 1, 0, "decode 27", 4500, "fwd_tile"), (2, 8, 128, 5, 0, "decode 31", 16384, "fwd_tile"),
               (2, 16, 256, 5, 0, "recon 8", 65536, "fwd_tile")]


def test_fp32_calls_take_the_faster_kernel(trace):
    body = "p = 0x7f0000000000          # not read: no kernel runs\n"
    for m, r, W, L, act, call, n, _ in FP32_ROUTES:
        name, arg = (call + " 0").split()[:2]
        body += f"""h, d = ctypes.c_void_p(), c.crom_decoder_desc({m}, {r}, {W}, {L}, {act}, 5.0)
ok(c.raw_call("crom_create", ctypes.byref(h), ctypes.byref(d), 0))
w = np.ascontiguousarray(gen.pack_params(gen.xavier_decoder(gen.DecoderSpec({m}, {r}, {W}, {L}), seed=1)), np.float32)
ok(c.raw_call("crom_set_weights", h, w.ctypes.data, w.size, 0, S))
note("shape")
if "{name}" == "decode":
    ok(c.raw_call("crom_decode", h, 1, p, p, p, {n}, {arg}, p, S))
elif "{name}" == "tangent":
    ok(c.raw_call("crom_tangent_velocity", h, 1, p, p, 1e-3, p, p, {n}, p, S))
else:
    ok(c.raw_call("crom_reconstruct", h, c.CROM_PREC_FP32, {arg}, p, {n}, p, p, S))
"""
    parts = "\n".join(trace(body)).split("shape")[1:]
    for shape, part in zip(FP32_ROUTES, parts, strict=True):
        assert shape[-1] in kernels(part.splitlines())[-1], shape


# layers, sizes, precision, iterations, whether the tiles are dealt: shapes at which the
# dealt form was measured slower than whole instances (False), and their neighbours
DEAL_ROUTES = [(2, "[96] * 244", "F16", 2, False), (5, "[96] * 244", "F16", 2, True), (2, "[96] * 200", "F16", 2, True),
               (2, "[32] * 627", "F16X2", 3, False), (5, "[73] * 430", "F16", 3, False), (5, "[140] * 430", "F16", 3, True),
               (3, "[20, 54] * 298", "F16X2", 2, False), (5, "[4096] * 8", "F16", 2, True), (2, "[200]", "F16X2", 2, True)]


def test_tiles_are_dealt_where_that_is_faster(trace):
    body = ""
    for hidden, sizes, prec, gn, _ in DEAL_ROUTES:
        body += f'h = context(hidden={hidden})\nnote("shape")\nstep(h, {sizes}, c.CROM_PREC_{prec}, gn={gn})\n'
    parts = "\n".join(trace(body)).split("shape")[1:]
    for (hidden, sizes, prec, gn, dealt), part in zip(DEAL_ROUTES, parts, strict=True):
        ks = kernels(part.splitlines())
        assert (not any("order" in k for k in ks)) == dealt, (hidden, sizes, prec, gn, ks)
        assert len(ks) == (gn if dealt else 2), ks


# layers, sizes, bound on them, precision, iterations, whether the tiles are dealt: few
# tiles per instance, and bounds above what the instances hold
LOOSE_DEAL_ROUTES = [(3, "[15] * 20", 60, "F16X2", 3, False), (5, "[15] * 19 + [200]", 200, "F16X2", 3, True),
                     (2, "[12, 8]", 64, "F16", 2, False), (4, "[40] * 8", 256, "F16", 2, True),
                     (3, "[22]", 252, "F16X2", 3, False), (3, "[22]", 252, "F16X2", 1, True), (3, "[40]", 252, "F16X2", 3, True)]


def test_tiles_are_dealt_by_the_samples_there_are(trace):
    body = ""
    for hidden, sizes, bound, prec, gn, _ in LOOSE_DEAL_ROUTES:
        body += f'h = context(hidden={hidden})\nnote("shape")\nstep(h, {sizes}, c.CROM_PREC_{prec}, gn={gn}, bound={bound})\n'
    parts = "\n".join(trace(body)).split("shape")[1:]
    for (hidden, sizes, bound, prec, gn, dealt), part in zip(LOOSE_DEAL_ROUTES, parts, strict=True):
        ks = kernels(part.splitlines())
        assert (not any("order" in k for k in ks)) == dealt, (hidden, sizes, bound, prec, gn, ks)


# m, r, width, layers, sizes, bound, iterations, the kernel
FP32_STEP_ROUTES = [(1, 1, 128, 1, "[213]", 213, 1, "fwd_fp32"), (1, 1, 128, 1, "[16]", 16, 1, "fwd_small"),
                    (2, 2, 32, 2, "[47] * 3", 47, 1, "fwd_fp32"), (2, 8, 32, 2, "[47] * 3", 47, 1, "fwd_small"),
                    (2, 8, 64, 1, "[2181] * 2", 2181, 3, "fwd_fp32"), (2, 2, 64, 1, "[40] * 1400", 40, 2, "fwd_tile"),
                    (3, 6, 32, 1, "[50] * 388", 71, 3, "fwd_fp32"), (3, 12, 32, 2, "[1768]", 6284, 3, "fwd_fp32"),
                    (1, 12, 128, 1, "[33] * 34", 62, 1, "fwd_fp32"), (2, 8, 96, 1, "[10286]", 10286, 1, "fwd_fp32"),
                    (1, 12, 32, 2, "[20000] * 2", 20678, 2, "fwd_fp32"), (1, 12, 32, 2, "[600] * 80", 600, 2, "fwd_tile"), (3, 6, 32, 4, "[150] * 95", 194, 2, "fwd_fp32"),
                    (3, 6, 64, 4, "[150] * 95", 194, 2, "fwd_tile"), (2, 8, 128, 5, "[300] * 64", 300, 2, "fwd_tile")]


def test_fp32_steps_take_the_faster_kernel(trace):
    body = ""
    for m, r, width, hidden, sizes, bound, gn, _ in FP32_STEP_ROUTES:
        body += f'h = context({m}, {r}, {width}, {hidden})\nnote("shape")\nstep(h, {sizes}, c.CROM_PREC_FP32, gn={gn}, r={r}, m={m}, bound={bound})\n'
    parts = "\n".join(trace(body)).split("shape")[1:]
    for shape, part in zip(FP32_STEP_ROUTES, parts, strict=True):
        assert all(shape[-1] in k for k in kernels(part.splitlines())), (shape, kernels(part.splitlines()))


def test_shared_memory_limits_are_never_lowered(trace):
    """A kernel's limit is the process's: a call that sets it to its own need takes it from
    other threads and from later calls within the default (a step of few samples followed
    by a tangent velocity that needs more than the step did, and less than the default)."""
    lines = trace("""
        p = 0x7f0000000000          # not read: no kernel runs
        h = context(1, 29, 32, 1)
        step(h, [40] * 4, c.CROM_PREC_FP32, r=29, m=1)
        ok(c.raw_call("crom_tangent_velocity", h, 1, p, p, 1e-3, p, p, 6, p, S))
        for r, n in ((8, 200), (2, 40), (16, 100)):
            step(context(2, r), [n], c.CROM_PREC_FP32, r=r)
            step(context(2, r), [n] * 60, c.CROM_PREC_FP32, r=r)
        for kind, n, nb in (("HEAT2D_NEUMANN", 127, 3), ("HEAT2D_NEUMANN", 57, 3), ("HEAT2D_NEUMANN", 100, 1),
                            ("HEAT2D_NEUMANN", 200, 1), ("HEAT2D_NEUMANN", 64, 1), ("ADVDIFF2D_PERIODIC", 97, 3),
                            ("ADVDIFF2D_PERIODIC", 57, 3), ("ADVDIFF2D_PERIODIC", 256, 64), ("ADVDIFF2D_PERIODIC", 100, 2)):
            ok(c.raw_call("crom_fom_step", getattr(c, "CROM_FOM_" + kind), nb, n, n, p, p, p, 1e-9, 20, p, p + (1 << 34), S))
        for n in (8192, 300, 7000):
            ok(c.raw_call("crom_fom_step", c.CROM_FOM_HEAT1D_DIRICHLET, 2, n, 1, p, p, p, 1e-9, 20, p, p + (1 << 34), S))
    """)
    assert [x for x in lines if x.startswith(("TOO MUCH", "LOWERED"))] == []
