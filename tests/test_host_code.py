"""The library's host code without a GPU: its objects linked with a stand-in for
the CUDA runtime (fake_cudart.cpp) that records launches, counts memory and
refuses what the runtime refuses.  Nothing is computed."""
import ctypes
import glob
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1012_3615_gb300 import abi, build

    build.build()
    out = str(tmp_path_factory.mktemp("fake") / "libbrillouin_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build_nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, "-o", out,
                    os.path.join(HERE, "fake_cudart.cpp")] + sorted(glob.glob(os.path.join(build.BUILD, "*.o"))),
                   check=True, capture_output=True, text=True)
    lib = ctypes.CDLL(out)
    for name, (res, args) in abi.SIGNATURES.items():
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_used.restype = ctypes.c_size_t
    lib.fake_budget.argtypes = [ctypes.c_size_t]
    lib.fake_refuse.argtypes = [ctypes.c_long, ctypes.c_long]
    lib.cudaMemGetInfo.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    lib.cudaStreamBeginCapture.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.cudaStreamEndCapture.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    lib.cudaGraphInstantiate.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_ulonglong]
    for n in ("cudaGraphLaunch",):
        getattr(lib, n).argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    for n in ("cudaGraphDestroy", "cudaGraphExecDestroy"):
        getattr(lib, n).argtypes = [ctypes.c_void_p]
    return lib


def build_nvcc():
    import shutil

    from paper_1012_3615_gb300 import build

    return shutil.which(build.NVCC) or "/usr/local/cuda/bin/nvcc"


@pytest.fixture
def fake(lib):
    lib.fake_reset()
    made = []

    class Fake:
        def __init__(self):
            self.lib = lib

        def op(self, L=(8, 8, 8, 8), device=0, comp=0, prec=0):
            """a context on a device with hopping fields built from links somewhere"""
            from paper_1012_3615_gb300 import abi

            lib.fake_device(device)
            lat = abi.bri_lattice((ctypes.c_int * 4)(*L), (ctypes.c_int * 4)(1, 1, 1, -1))
            h = ctypes.c_void_p()
            assert lib.bri_create(ctypes.byref(lat), ctypes.byref(h)) == 0
            made.append((device, h))
            return h

        def apply(self, h, nrhs=1, prec=0, stream=None):
            return lib.bri_apply(h, 1 << 50, 1 << 56, nrhs, 0.1, 0, prec, stream)

        def build(self, h, prec=0, comp=0):
            return lib.bri_build_hops(h, 1 << 57, prec, comp, None)

        def solve(self, h, mode, nrhs=1, maxit=8):
            from paper_1012_3615_gb300 import abi

            info = (abi.bri_solve_info * nrhs)()
            return lib.bri_solve(h, 1 << 50, 1 << 56, nrhs, 0.1, 1e-10, maxit, mode, info, 1 << 40)

        def log(self):
            text = lib.fake_log().decode().split("\n")
            lib.fake_clear_log()
            return [t for t in text if t]

    yield Fake()
    lib.fake_reset()
    for device, h in made:
        lib.fake_device(device)
        lib.bri_destroy(h)
    assert lib.fake_used() == 0  # nothing outlives its context


@pytest.mark.parametrize("L", [(8, 8, 8, 8), (11, 12, 12, 12), (16, 16, 16, 32)])
def test_fp64_apply_on_two_devices(fake, L):
    """the opt-in to the FP64 apply's shared memory belongs to each device"""
    for device in (0, 1):
        h = fake.op(L, device)
        assert fake.build(h) == 0
        assert fake.apply(h) == 0, fake.lib.bri_last_error(h)
        assert any("k_dslash_fx" in t for t in fake.log())


def _weights(lib, h, lam, rho):
    assert lib.bri_set_weights(h, (ctypes.c_double * 5)(*lam), (ctypes.c_double * 5)(*rho)) == 0


def test_solver_graphs_follow_the_operator(fake):
    """captured iterations hold the weights by value and the fields by address:
    after either changed they are captured again, and after neither they are not"""
    h = fake.op()
    assert fake.build(h, prec=1, comp=0) == 0
    wilson = [4.0, -0.5, 0, 0, 0], [0, 0.5, 0, 0, 0]
    for mode in (0, 1):
        fake.lib.fake_fill(0x3f if mode else 0)  # norms, so that the mixed solve runs
        for what, want in (("first", True), ("same", False), ("weights", True), ("links", False)):
            if what == "weights":
                _weights(fake.lib, h, *wilson)
            elif what == "links":  # same buffers, new contents
                assert fake.build(h, prec=1, comp=0) == 0
            fake.log()
            fake.solve(h, mode)
            log = fake.log()
            assert any(t.startswith("captured") for t in log) == want, (mode, what)
            assert any(t.startswith("replayed") for t in log), (mode, what)
            assert not any(t.startswith("STALE") for t in log), (mode, what)
        _weights(fake.lib, h, [1.9, -0.1, -0.1, -0.1, -0.1], [0, 0.1, 0.1, 0.1, 0.1])
    # another storage of the fields takes other memory
    assert fake.lib.bri_store_hops(h, 1, 1, None) == 0
    fake.log()
    fake.solve(h, 1)
    log = fake.log()
    assert any(t.startswith("captured") for t in log) and not any(t.startswith("STALE") for t in log)


def _capture(fake, stream, body):
    s = ctypes.c_void_p(stream)
    assert fake.lib.cudaStreamBeginCapture(s, 1) == 0
    body()
    g = ctypes.c_void_p()
    assert fake.lib.cudaStreamEndCapture(s, ctypes.byref(g)) == 0
    return g


def _instantiate(fake, g):
    e = ctypes.c_void_p()
    assert fake.lib.cudaGraphInstantiate(ctypes.byref(e), g, 0) == 0
    return e


def test_captured_fp64_apply_owns_its_work_space(fake):
    """no allocation nodes (they forbid a second executable graph); one work space
    per graph, shared by the applies of one stream, taken again by the next
    capture once the graph and its executable forms are gone"""
    h = fake.op((8, 8, 8, 8))
    assert fake.build(h) == 0 and fake.apply(h) == 0
    base = fake.lib.fake_used()
    s = 1 << 41

    def twice():
        assert fake.apply(h, 2, stream=s) == 0 and fake.apply(h, 1, stream=s) == 0

    g = _capture(fake, s, twice)
    one = fake.lib.fake_used() - base
    assert 2 * 4096 * 196 <= one < 3 * 4096 * 196
    e1, e2 = _instantiate(fake, g), _instantiate(fake, g)
    fake.lib.cudaGraphDestroy(g)
    fake.lib.cudaGraphExecDestroy(e1)
    g2 = _capture(fake, s, twice)  # e2 is alive: its work space is not taken
    assert fake.lib.fake_used() - base == 2 * one
    fake.log()
    fake.lib.cudaGraphLaunch(e2, None)
    assert [t.split()[0] for t in fake.log()] == ["replayed"] * 4
    fake.lib.cudaGraphExecDestroy(e2)
    fake.lib.cudaGraphDestroy(g2)
    for _ in range(5):
        g = _capture(fake, s, twice)
        fake.lib.cudaGraphDestroy(g)
    assert fake.lib.fake_used() - base == 2 * one


def test_captured_fp64_apply_without_memory(fake):
    """no memory for the work space: the FP64 kernel is captured"""
    h = fake.op((8, 8, 8, 8))
    assert fake.build(h) == 0
    fake.log()
    fake.lib.fake_refuse(0, 1)
    g = _capture(fake, 1 << 41, lambda: fake.apply(h, stream=1 << 41))
    log = fake.log()
    assert any("k_dslash" in t for t in log) and not any("_fx" in t for t in log)
    fake.lib.cudaGraphDestroy(g)


F64, F32, FULL, TWO_ROW = 0, 1, 0, 1
SITE_COPY = 5760  # bytes of the fixed-point copy


def _kind(log):
    """which FP64 apply ran"""
    return {"fx" if "k_dslash_fx" in t else "fp64" for t in log if t.startswith("run") and "k_dslash" in t}


def test_fixed_point_copy_only_with_room(fake):
    """the copy is taken where three times as much stays free, and tried again by
    the next build"""
    h = fake.op((8, 8, 8, 8))
    need = 4096 * (576 + SITE_COPY)
    fake.lib.fake_budget(need + 4 * 4096 * SITE_COPY - 4096)
    assert fake.build(h) == 0 and fake.apply(h) == 0
    assert _kind(fake.log()) == {"fp64"}
    fake.lib.fake_budget(1 << 40)
    assert fake.build(h) == 0 and fake.apply(h) == 0
    assert _kind(fake.log()) == {"fx"}


@pytest.mark.parametrize("what", ["store", "solve", "force"])
def test_fixed_point_copy_gives_way(fake, what):
    """a required allocation that fails takes the memory of the copy; the solver's
    graphs that read it go with it"""
    lib = fake.lib
    h = fake.op((8, 8, 8, 8))
    assert fake.build(h) == 0 and fake.apply(h) == 0 and fake.solve(h, 0) == 0
    assert "fx" in str(fake.log())
    lib.fake_budget(lib.fake_used() + 4096 * 200)
    if what == "store":
        assert lib.bri_store_hops(h, F32, FULL, None) == 0
    elif what == "solve":
        lib.fake_budget(1 << 40)
        assert lib.bri_store_hops(h, F32, TWO_ROW, None) == 0
        lib.fake_budget(lib.fake_used() + 4096 * 200)
        assert fake.solve(h, 4, nrhs=2) == 0
    else:
        lib.fake_budget(lib.fake_used() + 4096 * (2 * SITE_COPY - 1000))
        assert lib.bri_force(h, 1 << 50, 1 << 56, 1 << 57, 0.0, 1, None) == 0
    fake.log()
    assert fake.apply(h) == 0 and fake.solve(h, 0) == 0
    log = fake.log()
    assert _kind(log) == {"fp64"} and not any("STALE" in t or "replayed" in t and "_fx" in t for t in log)
    lib.fake_budget(1 << 40)
    assert fake.build(h) == 0 and fake.apply(h) == 0 and fake.solve(h, 0) == 0
    log = fake.log()
    assert _kind(log) == {"fx"} and not any("STALE" in t for t in log)


def test_fixed_point_copy_stays_for_a_program_graph(fake):
    """a captured apply of the program reads the copy for as long as its graph is
    there: an allocation that fails then is reported, and the next launch is not
    taken for the failure"""
    lib = fake.lib
    h = fake.op((8, 8, 8, 8))
    assert fake.build(h) == 0
    g = _capture(fake, 1 << 41, lambda: fake.apply(h, stream=1 << 41))
    e = _instantiate(fake, g)
    lib.cudaGraphDestroy(g)
    lib.fake_budget(lib.fake_used() + 4096 * 200)
    assert lib.bri_store_hops(h, F32, FULL, None) == -2  # BRI_ENOMEM
    fake.log()
    lib.cudaGraphLaunch(e, None)
    assert not any("STALE" in t for t in fake.log())
    assert fake.apply(h) == 0
    lib.cudaGraphExecDestroy(e)
    assert lib.bri_store_hops(h, F32, FULL, None) == 0


def test_fixed_point_copy_stays_when_it_would_not_do(fake):
    lib = fake.lib
    h = fake.op((8, 8, 8, 8))
    assert fake.build(h) == 0
    lib.fake_budget(lib.fake_used() + 4096 * 2000)
    ev = (ctypes.c_double * 4)()
    st = lib.bri_eigs_ddag_d(h, ev, None, None, 4, ctypes.c_double(0.1), 2000, ctypes.c_double(1e-8), F64, None, None)
    assert st == -2  # 2,001 vectors of 192 bytes a site
    fake.log()
    assert fake.apply(h) == 0
    assert _kind(fake.log()) == {"fx"}


def test_pool_memory_gives_way_first(fake):
    lib = fake.lib
    h = fake.op((8, 8, 8, 8))
    assert fake.build(h) == 0
    before = lib.fake_used()
    assert fake.apply(h, 30) == 0
    assert lib.fake_used() - before > 4096 * 196 * 29
    lib.fake_budget(lib.fake_used())
    assert lib.bri_store_hops(h, F32, TWO_ROW, None) == 0
    fake.log()
    assert fake.apply(h) == 0
    assert _kind(fake.log()) == {"fx"}


def test_work_space_refused_after_the_first_chunk(fake):
    """32 right-hand sides a launch: the other 8 through the FP64 kernel, at their
    own addresses"""
    h = fake.op((8, 8, 8, 8))
    assert fake.build(h) == 0
    fake.log()
    fake.lib.fake_refuse(1, 1)
    field = 4096 * 12 * 16
    assert fake.apply(h, 40) == 0
    log = [t for t in fake.log() if "k_dslash" in t]
    assert len(log) == 2 and "_fx" in log[0] and "_fx" not in log[1]
    assert "in %x out %x" % ((1 << 56) + 32 * field, (1 << 50) + 32 * field) in log[1]


def test_calls_that_run_out_of_memory_can_be_repeated(fake):
    """every allocation of a call refused in turn (with what would give way): the
    call succeeds or says so, and its repetition leaves the context with the same
    memory as one that never failed"""
    lib = fake.lib

    def run(refuse):
        """memory of a context whose calls were all repeated, and whether one failed"""
        lib.fake_reset()
        at = lib.fake_used()
        h = fake.op((8, 8, 8, 8))
        failed = False
        calls = [lambda: fake.build(h, prec=F32, comp=FULL), lambda: fake.apply(h), lambda: fake.solve(h, 1),
                 lambda: lib.bri_store_hops(h, F32, TWO_ROW, None), lambda: lib.bri_store_hops(h, F32, FULL, None),
                 lambda: lib.bri_set_clover(h, ctypes.c_double(1.0), None), lambda: fake.solve(h, 4, nrhs=2),
                 lambda: fake.solve(h, 0), lambda: lib.bri_set_clover(h, ctypes.c_double(0.0), None)]
        for i, call in enumerate(calls):
            lib.fake_refuse(*(refuse[1:] if refuse and refuse[0] == i else (-1, 0)))
            st = call()
            assert st in (0, -2), (refuse, i, st)
            failed = failed or st != 0
            lib.fake_refuse(-1, 0)
            if st:
                assert call() == 0, (refuse, i)
        # what may have given way comes back (the copy; a new set of solver vectors
        # without graphs, then one graph), and idle work space goes
        assert fake.build(h, prec=F32, comp=FULL) == 0 and fake.solve(h, 4, nrhs=3) == 0 and fake.solve(h, 0) == 0
        lib.fake_refuse(0, 1)
        assert lib.bri_store_hops(h, F32, TWO_ROW, None) == 0
        return lib.fake_used() - at, failed

    want, failed = run(None)
    assert not failed
    hits = 0
    for i in (0, 2, 3, 4, 5, 6, 7):
        for k in range(30):
            used, failed = run((i, k, 9))
            hits += failed
            assert used == want, (i, k, used, want)
    assert hits > 20


def test_fp32_sums_without_loss(tmp_path):
    """the accumulator of the FP32 solver's dot products: sums of FP32 numbers of
    any sign and size as exact as FP64 gives them, to 2^-44 of the sum of their
    magnitudes (one element a thread went to FP64 by itself)"""
    from paper_1012_3615_gb300 import build

    src = tmp_path / "sum.cu"
    src.write_text(r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "sum.cuh"
int main() {
    srand(5);
    double worst = 0;
    for (int t = 0; t < 20000; t++) {
        bri::SumF32 s;
        double ref = 0, size = 0;
        const int n = 1 + t % 12;
        for (int i = 0; i < n; i++) {
            const float v = (float)(std::ldexp(rand() / (double)RAND_MAX - 0.5, rand() % 30 - 15));
            s.add(v);
            ref += v;
            size += std::fabs(v);
        }
        worst = std::fmax(worst, std::fabs(s.get() - ref) / size);
    }
    printf("%.3e", worst);
}
""")
    exe = str(tmp_path / "sum")
    subprocess.run([build_nvcc()] + build.FLAGS + ["-o", exe, str(src)], check=True, capture_output=True, text=True)
    assert float(subprocess.run([exe], check=True, capture_output=True, text=True).stdout) <= 2.0**-44


def test_tuning_the_fp64_apply(fake, tmp_path, monkeypatch):
    """one shape in fixed point: nothing is timed, kept or written; the FP64 kernel,
    where that one runs, is tuned"""
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("BRI_TUNE_CACHE", str(cache))
    lib = fake.lib
    h = fake.op((8, 8, 8, 8))
    assert lib.bri_tune(h, F64, 1, None) == -8  # BRI_ESTATE: no fields
    assert fake.build(h) == 0
    fake.log()
    assert lib.bri_tune(h, F64, 1, None) == 0
    assert fake.log() == [] and lib.bri_get_threads(h, F64, 1) == 128 and not cache.exists()
    _weights(lib, h, [1e-300] * 5, [1e-300] * 5)
    assert lib.bri_tune(h, F64, 1, None) == 0
    assert _kind(fake.log()) == {"fp64"} and cache.exists()
