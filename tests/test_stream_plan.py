"""The packed factor stream and its entry codes (csrc/setup.cpp, build_stream),
walked on the CPU as the chain kernel walks them, against the rows of the plan:
every row's blocks come once and in order, the pieces end at the row's end and at
the multiples of the cut, and the walk solves the subdomain's triangular systems
(Sec. 3, Eq. 16)."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

import vesselmesh as vm

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_04289_gb300", "csrc")
PIECE, ROW, STAGE, NONE, EMPTY, BACKWARD = 16, 32, 64, 128, 129, 130


@pytest.fixture(scope="module")
def lib():
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tempfile.mkdtemp(prefix="fsi_stream_")
    so = os.path.join(d, "libstream.so")
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-fopenmp", "-shared", "-fPIC", "-I", CSRC,
                        os.path.join(ROOT, "tests", "native", "stream_export.cpp"),
                        os.path.join(CSRC, "setup.cpp"), "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(so)
    P, I = ctypes.c_void_p, ctypes.c_int64
    L.stream_new.restype, L.stream_new.argtypes = P, [I, P, I, P, ctypes.c_int32, ctypes.c_int32, ctypes.c_int32, P, I, I, I]
    L.stream_free.argtypes = [P]
    L.stream_array.restype, L.stream_array.argtypes = P, [P, ctypes.c_char_p, ctypes.POINTER(I)]
    yield L
    shutil.rmtree(d, ignore_errors=True)


def plan(L, m, np_, fill, ordering, cut, most, stage):
    X = np.ascontiguousarray(m.X, dtype=np.float64)
    T = np.ascontiguousarray(m.tets, dtype=np.int32)
    tag = m.node_tag
    rk = np.where((tag & vm.INTERFACE) != 0, 1, np.where((tag & vm.FLUID) != 0, 0, 2)).astype(np.uint8)
    h = L.stream_new(m.n_nodes, X.ctypes.data, m.n_tets, T.ctypes.data, np_, fill, ordering, rk.ctypes.data, cut, most, stage)
    out, types = {}, {"stage": np.uint8, "col": np.int32, "bcol": np.int32, "code": np.uint32}
    for name in ("sd_row", "row_ptr", "col", "diag", "L_off", "U_off", "src", "piv", "code", "code_off", "bcol", "stage",
                 "stage_off"):
        n = ctypes.c_int64()
        ptr = L.stream_array(h, name.encode(), ctypes.byref(n))
        dt = types.get(name, np.int64)
        out[name] = np.ctypeslib.as_array(ctypes.cast(ptr, ctypes.POINTER(np.ctypeslib.as_ctypes_type(dt))),
                                          shape=(n.value,)).copy()
    L.stream_free(h)
    return out


@pytest.mark.parametrize("ordering", [0, 1, 2])
@pytest.mark.parametrize("np_,fill,cut", [(4, 1, 1 << 40), (1, 2, 28), (64, 0, 1), (16, 1, 16), (7, 3, 5)])
@pytest.mark.parametrize("most,stage", [(8, 8), (8, 29), (16, 16), (16, 64)])
def test_walk_solves_the_subdomains(lib, most, stage, ordering, np_, fill, cut):
    m = vm.tube_config("tube-12x8x4")
    S = plan(lib, m, np_, fill, ordering, cut, most, stage)
    rng = np.random.default_rng(4)
    fac = rng.normal(size=len(S["col"])) * 0.1          # one number per block stands for the block
    seen = np.zeros(len(fac), dtype=int)
    for s in range(len(S["sd_row"]) - 1):
        a, b = S["sd_row"][s], S["sd_row"][s + 1]
        r = rng.normal(size=b - a)
        # the plain triangular solves on the plan's rows (diag holds the inverted pivot)
        want = r.copy()
        for q in range(a, b):
            e = slice(S["row_ptr"][q], S["diag"][q])
            want[q - a] -= fac[e] @ want[S["col"][e] - a]
        for q in range(b - 1, a - 1, -1):
            e = slice(S["diag"][q] + 1, S["row_ptr"][q + 1])
            want[q - a] = fac[S["diag"][q]] * (want[q - a] - fac[e] @ want[S["col"][e] - a])
        # the walk
        w, q, dq, tot, acc = r.copy(), 0, 1, 0.0, 0.0
        k, part, rows = S["L_off"][s], S["L_off"][s], 0
        words = S["code"][S["code_off"][s]:S["code_off"][s + 1]]
        codes = [(int(x) >> (8 * i)) & 255 for x in words for i in range(4)]
        assert codes[-8:] == [NONE] * 8
        sizes, in_stage = S["stage"][S["stage_off"][s]:S["stage_off"][s + 1]].astype(int).tolist(), 0
        assert sum(sizes) == S["L_off"][s + 1] - S["L_off"][s] and max(sizes) <= stage
        for c in codes:
            if c == EMPTY:
                assert S["diag"][a + q] == S["row_ptr"][a + q]
                q += dq
            elif c == BACKWARD:
                assert q == b - a and k == S["U_off"][s]
                q, dq, part = b - a - 1, -1, k
            elif c < NONE:
                n = (c & 15) + 1
                assert n <= most
                for i in range(k, k + n):
                    seen[S["src"][i]] += 1
                    v = fac[S["src"][i]] if S["piv"][i] < 0 else -fac[S["piv"][i]] * fac[S["src"][i]]
                    acc += v * w[S["bcol"][i]]
                assert (k - part) // cut == (k + n - 1 - part) // cut      # within one window of the cut
                k += n
                in_stage += n
                if c & STAGE:
                    assert in_stage == sizes.pop(0)
                    in_stage = 0
                if c & PIECE:
                    assert c & ROW or (k - part) % cut == 0
                    tot, acc = tot + acc, 0.0
                    if c & ROW:
                        w[q] = w[q] - tot if dq > 0 else tot
                        q, tot, rows = q + dq, 0.0, rows + 1
            else:
                assert c == NONE
        assert sizes == [in_stage]
        assert q == -1 and (S["L_off"][s + 1] == k)
        assert np.abs(w - want).max() <= 1e-12 * max(1.0, np.abs(want).max())
    assert np.all(seen == 1)


@pytest.mark.parametrize("ordering", [0, 1, 2])
@pytest.mark.parametrize("np_,fill,stage", [(4, 1, 16), (1, 2, 64), (64, 0, 13), (7, 3, 29), (200, 1, 16)])
def test_lookahead_walk_solves_the_subdomains(lib, np_, fill, stage, ordering):
    """The FP64 team's stream: a step's near block multiplies the row solved just
    before, its far blocks were summed a step earlier, before that row was known."""
    m = vm.tube_config("tube-12x8x4")
    S = plan(lib, m, np_, fill, ordering, 0, 0, stage)
    rng = np.random.default_rng(5)
    fac = rng.normal(size=len(S["col"])) * 0.1
    seen = np.zeros(len(fac), dtype=int)
    for s in range(len(S["sd_row"]) - 1):
        a, b = S["sd_row"][s], S["sd_row"][s + 1]
        n = b - a
        r = rng.normal(size=n)
        want = r.copy()
        for q in range(a, b):
            e = slice(S["row_ptr"][q], S["diag"][q])
            want[q - a] -= fac[e] @ want[S["col"][e] - a]
        for q in range(b - 1, a - 1, -1):
            e = slice(S["diag"][q] + 1, S["row_ptr"][q + 1])
            want[q - a] = fac[S["diag"][q]] * (want[q - a] - fac[e] @ want[S["col"][e] - a])
        w, k, t, far, nxt, in_stage = r.copy(), S["L_off"][s], 0, 0.0, 0.0, 0
        sizes = S["stage"][S["stage_off"][s]:S["stage_off"][s + 1]].astype(int).tolist()
        assert max(sizes) <= stage
        row = lambda i: i if i < n else 2 * n - 1 - i
        val = lambda i: fac[S["src"][i]] if S["piv"][i] < 0 else -fac[S["piv"][i]] * fac[S["src"][i]]
        for x in S["code"][S["code_off"][s]:S["code_off"][s + 1]]:
            for c in [(int(x) >> (8 * i)) & 255 for i in range(4)]:
                if c == NONE:
                    continue
                nf, near, solved = c & 15, 1 if c & 32 else 0, None
                assert nf <= 12
                for i in range(k, k + nf):
                    seen[S["src"][i]] += 1
                    assert t == 0 or S["bcol"][i] != row(t) or row(t + 1) == row(t)
                    nxt += val(i) * w[S["bcol"][i]]
                if near:
                    seen[S["src"][k + nf]] += 1
                    assert S["bcol"][k + nf] == row(t - 1)
                    far += val(k + nf) * w[S["bcol"][k + nf]]
                k += nf + near
                in_stage += nf + near
                if c & STAGE:
                    assert in_stage == sizes.pop(0)
                    in_stage = 0
                if c & 16:
                    w[row(t)] = w[row(t)] - far if t < n else far
                    far, nxt, t = nxt, 0.0, t + 1
                else:
                    assert not near
        assert t == 2 * n and k == S["L_off"][s + 1] and sizes == [in_stage]
        assert np.abs(w - want).max() <= 1e-12 * max(1.0, np.abs(want).max())
    assert np.all(seen == 1)
