"""Arrays of a caller that a call's kernels must not use in place: too short for
the call, overlapping another array of it, at an odd address, in managed memory,
or on the host beside others on the device.

Short arrays are refused with an error before any kernel reads or writes them.
They are the last 512 bytes of an allocation of 2 MiB - 128 KiB, whose pages are
2 MiB, so that no call here could reach unmapped memory.  The other arrays give
the results of host arrays: the same bits for the stresses, which are formed
element by element, and 1e-12 relative where up to eight elements are added in
any order (K x, dJ/du).
"""
import ctypes

import numpy as np
import pytest

from paper_1707_04228_gb300 import inputs

pytestmark = pytest.mark.gpu

ALLOC, SHORT = (2 << 20) - (128 << 10), 512


class Raw:
    """A bare address, as a C program passes it."""

    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address

    def is_contiguous(self):
        return True


@pytest.fixture(scope="module")
def solver(gl_lib, cuda_ok):
    from paper_1707_04228_gb300 import lib
    s = lib.Solver.from_laminate(inputs.corner_mini(n_arc=5, n_limb=1, n_width=3, nel_layer=1, angles=(0, 45, 90),
                                                    nsub=(3, 1, 1), nev=4, limb_L=3.0, width=3.0))
    yield s
    s.close()


@pytest.fixture(scope="module")
def cudart(cuda_ok):
    import torch
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    return ctypes.CDLL("/usr/local/cuda/lib64/libcudart.so")


def alloc(cudart, size, managed=False):
    p = ctypes.c_void_p()
    rc = cudart.cudaMallocManaged(ctypes.byref(p), ctypes.c_size_t(size), 1) if managed else \
        cudart.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size))
    assert rc == 0
    return p.value


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("call,short", [
    ("apply_K", 0), ("apply_K", 1), ("stress", 0), ("stress", 1), ("stress", 2), ("failure", 0), ("failure", 1),
    ("vjp", 0), ("vjp", 1), ("vjp", 2), ("vjp", 3), ("vjp", 4), ("adjoint", 0), ("adjoint", 1), ("adjoint", 2),
])
def test_short_array_is_refused(solver, cudart, call, short):
    import torch
    from paper_1707_04228_gb300 import lib
    s, N, E = solver, solver.n_dof, solver.n_elem
    assert 8 * E > SHORT and 8 * N < 64 << 10
    sizes = {"apply_K": (N, N), "stress": (N, E, E), "failure": (N, E), "vjp": (N, E, E, N, E),
             "adjoint": (N, N, E)}[call]
    a = [torch.from_numpy(1e-3 * inputs.random_vector(n, 7)).cuda() for n in sizes]
    torch.cuda.synchronize()
    base = alloc(cudart, ALLOC)
    try:
        a[short] = Raw(base + ALLOC - SHORT)
        with pytest.raises(lib.GLError) as e:
            if call == "apply_K":
                s.apply_K(a[0], a[1])
            elif call == "stress":
                s.stress(a[0], a[1], a[2])
            elif call == "failure":
                s.failure_index(a[0], F=a[1])
            elif call == "vjp":
                s.stress_vjp(a[0], a[1], a[2], a[3], a[4])
            else:
                s.adjoint(a[0], a[1], a[2])
        assert e.value.code == -3      # GL_ERR_CUDA, from the copy
    finally:
        assert cudart.cudaFree(ctypes.c_void_p(base)) == 0


def test_overlapping_arrays(solver):
    import torch
    s, N, E = solver, solver.n_dof, solver.n_elem
    u = 1e-3 * inputs.random_vector(N, 8)
    w = inputs.random_vector(E, 9)
    r33, r13, rpeak = s.stress(u)
    rF, rFmax, re = s.failure_index(u)
    rK = s.apply_K(u)
    rgu, rgt = s.stress_vjp(u, w, w)
    def dev():
        b = torch.zeros(N + 8, dtype=torch.float64, device="cuda")
        b[:N] = torch.from_numpy(u)
        torch.cuda.synchronize()
        return b
    for shift in (0, 3):
        b = dev()
        t13 = torch.empty(E, dtype=torch.float64, device="cuda")
        _, _, peak = s.stress(b[:N], b[shift:shift + E], t13)
        assert np.array_equal(b[shift:shift + E].cpu().numpy(), r33) and np.array_equal(t13.cpu().numpy(), r13)
        assert peak == rpeak
        b = dev()
        _, Fmax, e = s.failure_index(b[:N], F=b[shift:shift + E])
        assert np.array_equal(b[shift:shift + E].cpu().numpy(), rF) and (Fmax, e) == (rFmax, re)
        b = dev()
        s.apply_K(b[:N], b[shift:shift + N])
        assert rel(b[shift:shift + N].cpu().numpy(), rK) <= 1e-12
        b = dev()
        wd = torch.from_numpy(w).cuda()
        s.stress_vjp(b[:N], wd, wd, b[shift:shift + N], wd)
        assert rel(b[shift:shift + N].cpu().numpy(), rgu) <= 1e-12 and rel(wd.cpu().numpy(), rgt) <= 1e-12
    # both outputs in one place: the one written last, t13, stays
    o = torch.empty(E, dtype=torch.float64, device="cuda")
    _, _, peak = s.stress(u, o, o)
    assert np.array_equal(o.cpu().numpy(), r13) and peak == rpeak


@pytest.mark.parametrize("kind", ["odd", "managed", "host_out"])
def test_staged_arrays(solver, cudart, kind):
    import torch
    s, N, E = solver, solver.n_dof, solver.n_elem
    u = 1e-3 * inputs.random_vector(N, 10)
    r33, r13, rpeak = s.stress(u)
    rK = s.apply_K(u)
    if kind == "host_out":
        ud = torch.from_numpy(u).cuda()
        torch.cuda.synchronize()
        s33, t13, peak = s.stress(ud)
        assert np.array_equal(s33, r33) and np.array_equal(t13, r13) and peak == rpeak
        assert rel(s.apply_K(ud), rK) <= 1e-12
        return
    base = [alloc(cudart, 8 * N + 16, kind == "managed") for _ in range(3)]
    try:
        at = [b + (4 if kind == "odd" else 0) for b in base]
        copy = lambda dst, src, n: cudart.cudaMemcpy(ctypes.c_void_p(dst), ctypes.c_void_p(src),
                                                     ctypes.c_size_t(n), 4)
        assert copy(at[0], u.ctypes.data, 8 * N) == 0
        _, _, peak = s.stress(Raw(at[0]), Raw(at[1]), Raw(at[2]))
        s33, t13, y = np.empty(E), np.empty(E), np.empty(N)
        assert copy(s33.ctypes.data, at[1], 8 * E) == 0 and copy(t13.ctypes.data, at[2], 8 * E) == 0
        assert np.array_equal(s33, r33) and np.array_equal(t13, r13) and peak == rpeak
        s.apply_K(Raw(at[0]), Raw(at[1]))
        assert copy(y.ctypes.data, at[1], 8 * N) == 0
        assert rel(y, rK) <= 1e-12
    finally:
        for b in base:
            assert cudart.cudaFree(ctypes.c_void_p(b)) == 0
