"""Host code of the library over a stand-in for the CUDA runtime and cuFFT
(fake_cuda.c, preloaded in a child process): what is freed and allocated when
a call fails half-way, and which kernels a call launches.  No GPU is used."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, sys
sys.path.insert(0, %r)
from paper_1611_09322_gb300 import _lib
lib = _lib.load()
fake = ctypes.CDLL(None)
fake.fake_mallocs.restype = fake.fake_live.restype = fake.fake_launches.restype = ctypes.c_long
fake.fake_cost.argtypes = [ctypes.c_char_p, ctypes.c_double]
fake.fake_slow_start.argtypes = [ctypes.c_int, ctypes.c_double]
P = ctypes.c_void_p(64)  # kernels do not run: no position is read

def params(**kw):
    p = _lib.pse_params()
    p.tol, p.use_graph = 1e-3, -1
    for k, v in kw.items():
        setattr(p, k, v)
    return p

def create(L, **kw):
    c = ctypes.c_void_p()
    st = lib.pse_create_ex(ctypes.byref(c), L, 1.0, ctypes.byref(params(**kw)))
    assert st == 0, st
    return c

# grid points per unit length at xi a = 0.5, tol 1e-3 (k_cut / pi)
_info = _lib.pse_plan_info()
assert lib.pse_plan(60.0, 1.0, ctypes.byref(params(xi=0.5)), ctypes.byref(_info)) == 0
per_length = _info.k_cut / 3.141592653589793

def launches(name):
    return fake.fake_launches(name.encode())
""" % ROOT


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    from paper_1611_09322_gb300 import build
    build.build_cuda()
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", os.path.join(HERE, "fake_cuda.c"), "-o", so], check=True)

    def run(body):
        script = str(tmp_path_factory.mktemp("case") / "case.py")
        with open(script, "w") as f:
            f.write(PRELUDE + body)
        r = subprocess.run([sys.executable, script], env=dict(os.environ, LD_PRELOAD=so), cwd=ROOT,
                           capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
    return run


def test_failed_call_at_another_n_frees_no_buffer_in_use(child):
    """A call at a new N that fails after the old N's buffers were freed, at
    any of its allocations, leaves nothing behind: the next call at the old N
    allocates again.  On a 250^3 grid, where few particles take the library's
    own transforms and many cuFFT, the plan is made with the context: no later
    call depends on it."""
    child("""
c = ctypes.c_void_p()
fake.fake_fail_plans(1)
assert lib.pse_create_ex(ctypes.byref(c), 250.0, 1.0, ctypes.byref(params(xi=0.5, grid_M=250))) == 4
c = create(250.0, xi=0.5, grid_M=250)
few, many = 1000, 3_000_000
assert lib.pse_sample(c, few, P, 1, 1, P, None) == 0 and launches("k_fft_x") == 1
live = fake.fake_live()
for k in (1, 2, 5, 15, 25):
    fake.fake_fail_malloc(k)
    assert lib.pse_sample(c, many, P, 1, 1, P, None) == 2
    fake.fake_reset()
    assert lib.pse_sample(c, few, P, 1, 1, P, None) == 0
    assert fake.fake_mallocs() > 20 and fake.fake_live() == live
fake.fake_fail_plans(1)
fake.fake_reset()
assert lib.pse_sample(c, many, P, 1, 1, P, None) == 0 and launches("k_fft_x") == 0
lib.pse_destroy(c)
""")


@pytest.mark.parametrize("stored_ms,list_ms", [(0.5, 1.0), (1.0, 0.5)])
def test_timed_fp64_product_is_kept_at_another_n(child, stored_ms, list_ms):
    """autotune bit 2 in FP64 times the stored pair blocks against the list
    shapes once per context; the choice holds at every later N."""
    want = (1, 1, 1) if stored_ms < list_ms else (1, 0, 0)  # products, stored ones, pair evaluations
    child(f"""
c = create(40.0, xi=0.5, precision=1, autotune=4)
fake.fake_cost(b"k_lz_matvec", {list_ms})
fake.fake_cost(b"k_lz_matvec_stored", {stored_ms})
for N in (1000, 2000, 1000):
    assert lib.pse_sample_f64(c, N, P, 1, 1, P, None, None, None) == 0
    fake.fake_reset()
    assert lib.pse_sample_f64(c, N, P, 1, 2, P, None, None, None) == 0
    n = launches("k_lz_matvec"), launches("k_lz_matvec_stored"), launches("k_pairs")
    assert n == {want}, (N, n)
lib.pse_destroy(c)
""")


@pytest.mark.parametrize("N,M", [(1000, 48), (8192, 147), (8193, 48), (69999, 48), (70000, 64)])
def test_stage_timer_launches_what_a_sample_does(child, N, M):
    """pse_profile_stages: the kernels of pse_sample, each counted in a stage,
    with the one-launch cell list (up to 8192 particles) and without it, with
    cuFFT and with the library's own transforms."""
    child(f"""
N, M = {N}, {M}
names = ["k_cells_few", "k_bin", "k_scan", "k_scatter", "k_place", "k_fft", "k_wave_noise", "k_grid_aos", "k_interp",
         "k_nbr", "k_lz_init", "k_lz_matvec", "k_lz_update", "k_lz_final"]
c = create(60.0, xi=0.5, grid_M=M)
assert lib.pse_sample(c, N, P, 1, 1, P, None) == 0
fake.fake_reset()
assert lib.pse_sample(c, N, P, 1, 1, P, None) == 0
sample = [launches(n) for n in names]
assert sum(sample) == launches("k_"), sample
fake.fake_reset()
ms, nl = (ctypes.c_double * len(_lib.STAGES))(), (ctypes.c_int * len(_lib.STAGES))()
assert lib.pse_profile_stages(c, N, P, 1, 1, P, ms, nl, None) == 0
assert [launches(n) for n in names] == sample, dict(zip(names, sample))
assert sum(nl) == launches("k_"), dict(zip(_lib.STAGES, nl))
lib.pse_destroy(c)
""")


# grid, its sites per particle, own transforms in samples, in forces calls
@pytest.mark.parametrize("M,per,sample,forces", [
    (64, 20, 0, 0), (125, 20, 0, 0), (126, 20, 1, 1), (126, 4, 1, 1), (128, 20, 0, 0), (140, 4, 1, 1), (144, 20, 0, 0),
    (160, 4, 1, 1), (162, 4, 1, 1), (200, 4, 1, 1), (216, 8, 0, 1), (216, 13, 1, 1), (225, 4, 0, 1), (225, 8, 1, 1),
    (245, 4, 0, 1), (245, 8, 1, 1), (250, 8, 0, 1), (250, 11, 1, 1), (256, 20, 0, 0), (288, 11, 0, 1), (288, 13, 1, 1),
    (378, 20, 0, 1), (378, 31, 1, 1), (486, 31, 1, 1), (490, 40, 0, 0)])
def test_rule_for_the_transforms(child, M, per, sample, forces):
    """Which transforms samples and forces calls take, on both sides of every
    line of the rule."""
    child(f"""
M, N = {M}, int({M} ** 3 / {per})
c = create(1.2 * M, xi=0.4, grid_M=M, max_iter=4)
fake.fake_reset()
assert lib.pse_sample(c, N, P, 1, 1, P, None) == 0
assert (launches("k_fft_"), launches("k_wave_noise")) == ((3, 0) if {sample} else (0, 1))
fake.fake_reset()
assert lib.pse_sample_with_forces(c, N, P, P, 1, 1, 1.0, 1.0, P, None) == 0
assert (launches("k_fft_"), launches("k_wave_apply")) == ((5, 0) if {forces} else (0, 1))
lib.pse_destroy(c)
""")


COSTS = """
def costs(own, c2r):  # ms: each own pass; the C2R; noise and copy take 0.2 each
    for name, ms in ((b"k_fft_", own), (b"C2R", c2r), (b"k_wave_noise", 0.2), (b"k_grid_aos", 0.2)):
        fake.fake_cost(name, ms)
"""


@pytest.mark.parametrize("own,c2r,M", [(0.1, 1.0, 126), (1.0, 1.0, 120), (0.37, 0.9, 126), (0.38, 0.9, 120)])
def test_grid_tuning_times_the_transforms_that_run(child, own, c2r, M):
    """autotune bit 0: of the grids 120, 125, 128 (noise kernel, cuFFT, copy)
    and 126 and 135 (three passes of the library's own, counted 1.15 times) the
    first of the faster kind is taken; two species too."""
    child(COSTS + f"""
costs({own}, {c2r})
L = 120 / per_length  # the planned grid is 120
info = _lib.pse_plan_info()
c = create(L, xi=0.5, autotune=1)
assert lib.pse_get_plan(c, ctypes.byref(info)) == 0
assert info.M == {M}, info.M
lib.pse_destroy(c)
c = ctypes.c_void_p()
radii = (ctypes.c_double * 2)(1.0, 1.5)
costs({own}, {c2r} - 0.2)  # the noise is a launch per species
assert lib.pse_create_poly(ctypes.byref(c), L, 2, radii, ctypes.byref(params(xi=0.5, autotune=1))) == 0
assert lib.pse_get_plan(c, ctypes.byref(info)) == 0 and info.M == {M}, info.M
lib.pse_destroy(c)
""")


def test_xi_tuning_predicts_with_the_transforms_that_run(child):
    """pse_tune_xi: a candidate's predicted time is the start's, less its
    xi-dependent stages, plus the scaled real part and the wave part as it
    would run on the candidate's grid: 1.15 times three passes of 0.1 ms, or
    0.2 + 0.9 + 0.2 ms.  The reported t_wave is the start grid's."""
    child(COSTS + """
costs(0.1, 0.9)
fake.fake_cost(b"k_nbr", 0.3)
fake.fake_cost(b"k_lz_matvec", 0.5)
out = _lib.pse_xi_tuning()
assert lib.pse_tune_xi(119.9 / per_length, 1.0, ctypes.byref(params(xi=0.5)), 50000, P, 3.0, 2, ctypes.byref(out), None) == 0
assert out.M_tried[0] == 120 and abs(out.t_wave - 1.3) < 1e-5 and abs(out.t_real - 0.8) < 1e-5
seen = set()
for k in range(1, out.n_tried):
    M = out.M_tried[k]
    wave = out.ms_pred[k] - (out.ms_start - out.t_real - out.t_wave + out.t_real * (0.5 / out.xi_tried[k]) ** 3)
    own = M >= 126 and M not in (128, 144)
    seen.add(own)
    assert abs(wave - (0.345 if own else 1.3)) < 1e-5, (M, wave)
assert out.n_tried == 8 and True in seen
""")


def test_xi_tuning_keeps_the_fastest_of_three_rounds(child):
    """A trial whose first samples run slow (clocks, a first round) counts
    with its fastest round of `reps` samples."""
    child("""
fake.fake_cost(b"k_lz_matvec", 0.5)
fake.fake_cost(b"k_wave_noise", 0.2)  # (no launch of the library's own transforms)
fake.fake_slow_start(2 + 3 + 3, 2.0)  # the untimed samples and two rounds of three
out = _lib.pse_xi_tuning()
assert lib.pse_tune_xi(119.9 / per_length, 1.0, ctypes.byref(params(xi=0.5)), 50000, P, 3.0, 3, ctypes.byref(out), None) == 0
assert out.n_tried == 8 and out.M_tried[0] == 120
assert all(min(abs(t - 0.5), abs(t - 0.7)) < 1e-5 for t in out.ms_tried), list(out.ms_tried)
""")
