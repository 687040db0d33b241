"""What libfe asks of the CUDA runtime, call by call, checked without a GPU.

A child process preloads fake_cuda.c in place of the CUDA runtime, cuBLAS and cuSOLVER and drives
the C ABI; the log of allocations, copies and launches is then compared with what the library
promises.  Faults that could reach the GPU (an address used after it was freed, a launch outside
the limits, a misaligned access) are shown here and nowhere else.
"""
import os
import re
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.join(os.path.dirname(HERE), "paper_2504_00998_gb300")

PRELUDE = """
import ctypes as C, importlib.util, time
spec = importlib.util.spec_from_file_location("fe_lib", {lib!r})
L = importlib.util.module_from_spec(spec)
spec.loader.exec_module(L)
lib = L.load()
fake = C.CDLL({fake!r})
fake.fake_log.restype = C.c_char_p
fake.fake_fail_malloc.argtypes = [C.c_size_t]

def mesh(ncell, p, L3=(4.0, 4.0, 4.0)):
    d = L.FeMeshDesc()
    for k in range(3):
        d.L[k], d.ncell[k] = L3[k], ncell[k]
    d.p = p
    h = C.c_void_p()
    L.call("fe_mesh_create", C.byref(d), C.byref(h))
    return h

def host(n):                    # n doubles, 16-byte aligned
    b = C.create_string_buffer(8 * n + 16)
    host.keep.append(b)
    return (C.addressof(b) + 15) // 16 * 16
host.keep = []

def log():
    return fake.fake_log().decode()
"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    """Runs a script against the fake runtime and returns what it printed."""
    from paper_2504_00998_gb300 import build
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "fake_cuda.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", so, os.path.join(HERE, "fake_cuda.c")],
                   check=True)
    prelude = PRELUDE.format(lib=os.path.join(PKG, "_lib.py"), fake=so)

    def run(script):
        r = subprocess.run([sys.executable, "-c", prelude + script], capture_output=True, text=True,
                           timeout=120, env=dict(os.environ, LD_PRELOAD=so))
        assert r.returncode == 0, r.stderr
        return r.stdout

    return run


@pytest.mark.parametrize("p", [4, 5])
@pytest.mark.parametrize("first", ["fe_poisson_apply_K_f32", "fe_poisson_apply_K"])
def test_stiffness_scratch_is_never_freed(child, p, first):
    """A graph captured around one stiffness product stays valid after the other: both keep the
    address of their scratch for the mesh's life, in either order."""
    out = child(f"""
h = mesh((3, 3, 3), {p})
x, y = host(4000), host(4000)
fake.fake_reset()
for name in ({first!r}, "fe_poisson_apply_K", "fe_poisson_apply_K_f32"):
    L.call(name, h, x, y)
print(log())
""")
    assert "k_cell_apply" in out and "k_cell64" in out
    assert not re.search("^free ", out, re.M), out


def test_stiffness_scratch_has_one_stream(child):
    """The double product's scratch serves one stream at a time: a product on another stream, and
    one inside the caller's capture, take the scratch-free kernel until a solve has waited for
    the first stream's products."""
    out = child("""
h = mesh((2, 2, 2), 4)
x, y = host(2000), host(2000)
A, B = C.c_void_p(0x1000), C.c_void_p(0x2000)
def product(stream, capture=False):
    L.call("fe_mesh_set_stream", h, stream)
    fake.fake_reset()
    if capture:
        fake.cudaStreamBeginCapture(stream, 0)
    L.call("fe_poisson_apply_K", h, x, y)
    if capture:
        fake.cudaStreamEndCapture(stream, C.byref(C.c_void_p()))
    print("cell" if "k_cell64" in log() else "sweep" if "kron_kernel" in log() else log())
def solve(stream):
    L.call("fe_mesh_set_stream", h, stream)
    bc, info = L.FePoissonBC(), L.FeSolveInfo()
    bc.kind, bc.rtol, bc.max_iter = L.FE_BIAS_CEF, 1e-10, 10
    L.call("fe_poisson_solve_load", h, x, C.byref(bc), None, y, C.byref(info))
product(A, capture=True)
product(A)
product(A, capture=True)
product(B)
solve(B)
product(B)
product(A)
solve(A)
product(B)
product(A)
""")
    assert out.split() == ["sweep", "cell", "sweep", "sweep", "sweep", "cell", "cell", "sweep"]


# 192 tiles of 64 columns, 257 and 341 of 48, the most columns taken (256 of 64)
@pytest.mark.parametrize("n,tiles", [(12288, 192), (12289, 257), (16321, 341), (16384, 256)])
def test_rayleigh_ritz_of_many_columns_launches(child, n, tiles):
    """Every launch of a double Rayleigh-Ritz stays within the grid limits up to the widest
    block that is accepted, and the Gram grid has every pair of column tiles."""
    out = child(f"""
h = mesh((16, 16, 9), 4)        # 143,360 nodes; no kernel runs, so the blocks are only addresses
L.call("fe_set_potential", h, 0x1000)
fake.fake_reset()
st = lib.fe_rayleigh_ritz(h, 0x10000, {n}, {n + n % 2}, 0x1000, L.FE_F64)
print(st, lib.fe_last_error().decode() if st else "ok")
print(log())
""")
    assert out.startswith("0 ok"), out.splitlines()[0]
    grids = re.findall(r"^launch \S*k_gram_partial\S* 1 (\d+) (\d+) ", out, re.M)
    assert grids and set(grids) == {(str(tiles), str(tiles))}


# memory of this device, off its alignment, of another device, unknown to CUDA (fake_cuda.c)
@pytest.mark.parametrize("veff,copied", [(1 << 25, False), ((1 << 25) + 4, True), (1 << 22, True),
                                         (1 << 16, True)])
def test_set_potential_copies_what_a_kernel_must_not_read(child, veff, copied):
    out = child(f"""
h = mesh((2, 2, 2), 3)
fake.fake_reset()
L.call("fe_set_potential", h, {veff})
print(log())
""")
    copies = re.findall(r"^copy 3 \S+ (\S+) ", out, re.M)
    assert copies == ([hex(veff)] if copied else []), out
    assert "k_set_potential" in out


# 65,535 and 65,536 tiles of eight 16-byte groups, and the 65,535 tiles of 128 vectors that the
# term once took
@pytest.mark.parametrize("prec,nvec", [("FE_F64", 16 * 65535), ("FE_F64", 16 * 65535 + 1),
                                       ("FE_F32", 32 * 65535 + 1), ("FE_F32", 128 * 65535)])
def test_nonlocal_term_of_many_vectors_launches(child, prec, nvec):
    out = child(f"""
h = mesh((1, 1, 2), 1)
L.call("fe_set_potential", h, 1 << 25)
one = (C.c_double * 6)(*[2.0] * 6)
L.call("fe_set_nonlocal", h, 2, one, one, (C.c_double * 8)(*[1.0] * 8), 3.0)
ld = ({nvec} + 3) // 4 * 4
fake.fake_reset()
st = lib.fe_apply_H(h, 1 << 32, 1 << 40, {nvec}, ld, L.{prec})
print(st, lib.fe_last_error().decode() if st else "ok")
print(log())
""")
    assert out.startswith("0 ok"), out.splitlines()[0]
    tiles = -(-nvec // (16 if prec == "FE_F64" else 32))
    y, z = map(int, re.search(r"k_nl_project\S* 2 (\d+) (\d+) 256 ", out).groups())
    assert tiles <= y * z < tiles + y


def test_solve_without_memory_for_the_eigenbases(child):
    """The default solve needs the tables of the separable preconditioner for speed only: when
    they cannot be allocated the other iterations solve, and the next solve tries again.  (The
    bytes 0x40 read as 32.5 everywhere, so the residual is above the tolerance and planes count
    as free; 4 x 4 x 4 cells of p = 4 are chains of 16, 16 and 17 nodes.)"""
    out = child("""
fake.fake_fill(0x40)
h = mesh((4, 4, 4), 4)
x, y = host(4352), host(4352)
tables = 4 * (2 * (16 * 16 + 16 * 16 + 17 * 17) + 16 + 16 + 17)
def solve():
    fake.fake_reset()
    bc, info = L.FePoissonBC(), L.FeSolveInfo()
    bc.kind, bc.rtol, bc.max_iter = L.FE_BIAS_CEF, 1e-3, 32
    st = lib.fe_poisson_solve_load(h, x, C.byref(bc), None, y, C.byref(info))
    print(st, f" {tables}\\n" in log(), "k_sep_gemm" in log(), "graph" in log())
fake.fake_fail_malloc(tables)
solve()
solve()
fake.fake_fail_malloc(0)
solve()
""")
    assert out.splitlines()[:2] == ["0 True False True"] * 2, out
    assert out.splitlines()[2].split()[1:3] == ["True", "True"], out


@pytest.mark.parametrize("nz", [1, 7, 96, 1000, 4001, 2000000])
def test_segment_rule_of_long_slabs(child, nz):
    """The z segments of a launch are those of least (layers + 1) x CTAs an SM over every segment
    count, found without trying each: a launch on two million layers takes well under the 20 ms
    that trying them took."""
    out = child(f"""
h = mesh((1, 1, {nz}), 2)
L.call("fe_set_potential", h, 1 << 25)
best = 1.0
for _ in range(5):
    fake.fake_reset()
    t0 = time.perf_counter()
    L.call("fe_apply_H", h, 1 << 32, 1 << 40, 16, 16, L.FE_F32)
    best = min(best, time.perf_counter() - t0)
print(best)
print(log())
""")
    def cost(s):
        z = -(-nz // s)
        segs = -(-nz // z)
        return (z + (segs > 1)) * max(1.5, -(-segs // 152)), s, segs

    segs = min(map(cost, range(1, min(nz, 20000) + 1)))[2]
    assert int(re.search(r"sweep_kernel\S* (\d+) 1 1 ", out).group(1)) == segs
    assert float(out.split()[0]) < 2e-3
