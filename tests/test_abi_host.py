"""The C boundary without a GPU: the library loads, exports every symbol the
header declares, and rejects bad arguments on the host before touching CUDA."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2303_08810_b200 import build, binding
    build.build_library()
    return binding.load_library()


def declared_symbols():
    names = set()
    for fn in os.listdir(os.path.join(ROOT, "include")):
        if fn.endswith(".h"):
            text = open(os.path.join(ROOT, "include", fn)).read()
            text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
            names |= set(re.findall(r"\b(bra_[a-z_]+)\s*\(", text))
    return names


def test_library_exports_every_declared_symbol(lib):
    names = declared_symbols()
    assert {"bra_route", "bra_attend", "bra_forward", "bra_backward", "bra_workspace_bytes",
            "bra_device_status", "bra_status_string", "bra_version"} <= names
    for n in names:
        assert hasattr(lib, n), f"{n} declared in include/ but not exported"


def test_version_and_status_strings(lib):
    assert lib.bra_version() >= 100
    seen = set()
    for code in range(0, 12):                     # BRA_OK .. BRA_ERR_STATIC_LIMIT
        s = lib.bra_status_string(code).decode()
        assert s and s != "unknown status"
        seen.add(s)
    assert len(seen) == 12
    assert lib.bra_status_string(99).decode() == "unknown status"


def problem(**kw):
    from paper_2303_08810_b200 import binding
    base = dict(B=2, H=16, W=16, C=64, heads=2, S=4, topk=2, dtype="bf16")
    base.update(kw)
    return binding.make_problem(**base)


def test_workspace_bytes(lib):
    from paper_2303_08810_b200 import binding
    p = problem()
    n = binding.workspace_bytes(p)
    assert n > 0 and n % 256 == 0
    # holds at least the two mean tensors and the index
    assert n >= 2 * 4 * p.B * 16 * p.C + 4 * p.B * p.heads * 16 * p.topk
    assert binding.workspace_bytes(problem(B=4)) > n
    assert binding.workspace_bytes(problem(S=0)) == 0          # invalid problem
    assert binding.workspace_bytes(problem(S=3)) > n           # S does not divide the map: room for the padded copies


def test_every_included_file_makes_the_library_stale(monkeypatch, tmp_path):
    """A change of any source or header is a change of the library: all files of csrc/ that a source includes, transitively,
    and the public header."""
    from paper_2303_08810_b200 import build
    seen, todo = set(), list(build.sources())
    while todo:
        path = os.path.realpath(todo.pop())
        if path in seen:
            continue
        seen.add(path)
        for name in re.findall(r'^\s*#include "([^"]+)"', open(path).read(), flags=re.M):
            todo.append(os.path.join(os.path.dirname(path), name))
    assert any(p.endswith(".cuh") for p in seen) and any(p.endswith("bra.h") for p in seen)
    assert seen <= {os.path.realpath(p) for p in build.dependencies()}
    lib = tmp_path / "lib.so"
    lib.write_bytes(b"")
    monkeypatch.setattr(build, "LIB_PATH", str(lib))
    newest = max(os.path.getmtime(p) for p in build.dependencies())
    os.utime(lib, (newest + 1,) * 2)
    assert not build.is_stale()
    os.utime(lib, (newest - 1,) * 2)
    assert build.is_stale()


A = 0x10000  # a fake, aligned, never dereferenced device address


@pytest.mark.parametrize("kw,code", [
    (dict(B=0), 2), (dict(H=-1), 2), (dict(S=0), 2), (dict(heads=3), 2),
    (dict(topk=0), 3), (dict(topk=17), 3),
])
def test_route_rejects_bad_problems(lib, kw, code):
    from paper_2303_08810_b200 import binding
    p = problem(**kw)
    rc = lib.bra_route(ctypes.byref(p), A, A, A, A, A, A, 1 << 30, None)
    assert rc == code


def test_bad_dtype_lce_impl(lib):
    p = problem()
    p.dtype = 7
    assert lib.bra_route(ctypes.byref(p), A, A, A, A, A, A, 1 << 30, None) == 4
    p = problem()
    p.lce_ksize = 3
    assert lib.bra_attend(ctypes.byref(p), A, A, A, A, A, None, A, None, A, 1 << 30, None) == 7
    p = problem()
    p.impl = 9
    assert lib.bra_attend(ctypes.byref(p), A, A, A, A, A, None, A, None, A, 1 << 30, None) == 7
    p = problem(C=24, heads=2)           # head dim 12: no 16-byte channel vectors
    assert lib.bra_attend(ctypes.byref(p), A, A, A, A, A, None, A, None, A, 1 << 30, None) == 7


def test_null_alignment_workspace_checks(lib):
    from paper_2303_08810_b200 import binding
    p = problem()
    need = binding.workspace_bytes(p)
    ref = ctypes.byref(p)
    assert lib.bra_route(None, A, A, A, A, A, A, need, None) == 1
    assert lib.bra_route(ref, None, A, A, A, A, A, need, None) == 1
    assert lib.bra_route(ref, A, A, A, A, None, A, need, None) == 1            # index is required
    assert lib.bra_route(ref, A, A, A, A, A, None, need, None) == 1            # ws is required
    assert lib.bra_route(ref, A + 8, A, A, A, A, A, need, None) == 5
    assert lib.bra_route(ref, A, A, A, A, A, A + 16, need, None) == 5          # ws wants 256
    assert lib.bra_route(ref, A, A, A, A, A, A, need - 1, None) == 6
    # attend: LCE weights required unless LCE is off; O required
    assert lib.bra_attend(ref, A, A, A, A, None, None, A, None, A, need, None) == 1
    assert lib.bra_attend(ref, A, A, A, A, A, None, None, None, A, need, None) == 1
    assert lib.bra_attend(ref, A, A, A + 2, A, A, None, A, None, A, need, None) == 5
    assert lib.bra_forward(ref, A, A, None, A, None, A, None, None, A, need, None) == 1
    assert lib.bra_forward(ref, A, A, A, A, None, A, None, None, A, 16, None) == 6
    # backward: lse and dO required
    args = [A] * 12
    bad = list(args); bad[5] = None                                           # lse
    assert lib.bra_backward(ref, *bad, A, need, None) == 1
    bad = list(args); bad[6] = None                                           # dO
    assert lib.bra_backward(ref, *bad, A, need, None) == 1
    assert lib.bra_device_status(None, None) == 1


def test_workspace_init_checks_its_arguments(lib):
    from paper_2303_08810_b200 import binding
    p = problem()
    need = binding.workspace_bytes(p)
    assert lib.bra_workspace_init(ctypes.byref(p), None, need, None) == 1
    assert lib.bra_workspace_init(ctypes.byref(p), A + 8, need, None) == 5
    assert lib.bra_workspace_init(ctypes.byref(p), A, need - 1, None) == 6
    bad = problem(S=0)
    assert lib.bra_workspace_init(ctypes.byref(bad), A, need, None) == 2


def test_injection_switch_is_validated(lib):
    p = problem()
    p.inject = 5
    assert lib.bra_attend(ctypes.byref(p), A, A, A, A, A, None, A, None, A, 1 << 30, None) == 7


def test_unsupported_impl_for_problem(lib):
    from paper_2303_08810_b200 import binding
    p = problem(dtype="f32", impl=binding.IMPL_MMA)      # tensor-core paths are bf16 only
    need = binding.workspace_bytes(p)
    assert lib.bra_attend(ctypes.byref(p), A, A, A, A, A, None, A, None, A, need, None) == 7


def test_binding_fails_loudly_without_gpu():
    import torch
    from paper_2303_08810_b200 import binding
    if torch.cuda.is_available():
        pytest.skip("has a GPU")
    with pytest.raises(RuntimeError, match="no CPU fallback"):
        binding.workspace(problem())


# ------------------------------------------------------------------ what is accepted
def status_without_gpu(lib, call, **kw):
    """What `call` answers for a problem: 7 (no kernel) or, past every host check, 8 - the launch finds no device."""
    import torch
    if torch.cuda.is_available():
        pytest.skip("the made-up addresses must not reach a GPU")
    p = problem(**kw)
    big = 1 << 62
    if call == "attend":
        return lib.bra_attend(ctypes.byref(p), A, A, A, A, A, A, A, A, A, big, None)
    return lib.bra_backward(ctypes.byref(p), *([A] * 12), A, big, None)


# regions whose tokens times listed tokens pass 2^32: the kernels divide token numbers exactly, whatever their product
@pytest.mark.parametrize("call,kw", [
    ("attend", dict(H=256, W=256, S=1, topk=1, dtype="f32")),
    ("attend", dict(H=512, W=512, S=4, topk=1, dtype="f32")),
    ("attend", dict(H=736, W=736, S=8, topk=4, dtype="f32")),
    ("attend", dict(H=512, W=512, S=4, topk=16, dtype="bf16")),
    ("attend", dict(H=8192, W=8192, S=2, topk=4, C=16, heads=1, dtype="f32")),
    ("backward", dict(H=512, W=512, S=4, topk=1, dtype="f32")),
    ("backward", dict(H=512, W=512, S=4, topk=1, dtype="bf16")),
    ("backward", dict(H=728, W=728, S=8, topk=4, dtype="bf16")),
    ("backward", dict(H=1024, W=1024, S=16, topk=4, dtype="bf16")),
    ("backward", dict(H=1024, W=1024, S=16, topk=4, C=128, dtype="bf16")),
])
def test_large_regions_are_accepted(lib, call, kw):
    assert status_without_gpu(lib, call, **{"B": 1, **kw}) == 8


@pytest.mark.parametrize("many", [dict(B=70000), dict(B=1, C=70000 * 32, heads=70000)], ids=["images", "heads"])
@pytest.mark.parametrize("call", ["attend", "backward"])
@pytest.mark.parametrize("kw", [dict(dtype="f32"), dict(dtype="bf16"), dict(dtype="bf16", H=7, W=7, S=7, topk=7)])
def test_more_images_or_heads_than_a_grid_extent_are_accepted(lib, call, kw, many):
    if "heads" not in many:
        many = dict(many, C=32, heads=1)
    assert status_without_gpu(lib, call, **{**dict(H=8, W=8, S=2, topk=2), **kw, **many}) == 8


def test_every_region_size_is_accepted(lib):
    """fp32 has only the CUDA-core kernels, so they take every region size, list length and batch: no layout of their shared
    memory is too large."""
    for d in (16, 32, 64, 128):
        for dtype in ("f32", "bf16"):
            for hs, ws in ((1, 1), (1, 2), (2, 1), (2, 2), (1, 3), (3, 3), (2, 5), (4, 4), (3, 7), (8, 8), (7, 11), (16, 16), (1, 300), (40, 3)):
                for S in (1, 2, 4, 7, 14, 16, 31):
                    for topk in {1, min(4, S * S), S * S}:
                        for B, heads in ((1, 1), (8, 2), (64, 4)):
                            kw = dict(B=B, H=hs * S, W=ws * S, C=heads * d, heads=heads, S=S, topk=topk, dtype=dtype, impl=1)
                            assert status_without_gpu(lib, "attend", **kw) == 8, kw
                            if d <= 64 and S * S <= 1000:
                                assert status_without_gpu(lib, "backward", **kw) == 8, kw


def test_division_by_multiplication_is_exact(tmp_path):
    """csrc/fast_div.h on the host: every divisor of a spread, dividends next to every kind of multiple."""
    import subprocess
    src = tmp_path / "t.cpp"
    src.write_text('''
#include "fast_div.h"
#include <stdio.h>
int main() {
    const uint32_t top = 0x7fffffffu;
    long long bad = 0;
    auto check = [&](uint32_t n, uint32_t d, const bra::FastDiv& f) { if (bra::fdiv(n, f) != n / d) { if (!bad++) printf("%u / %u\\n", n, d); } };
    auto divisor = [&](uint32_t d) {
        const bra::FastDiv f = bra::fast_div((int)d);
        for (uint64_t m = 1; m * d <= top; m = m < 40 ? m + 1 : m + m / 3)
            for (int o = -1; o <= 1; ++o) if (m * d + o <= top) check((uint32_t)(m * d + o), d, f);
        const uint32_t last = top / d * d;
        check(0, d, f); check(last, d, f); check(last - 1, d, f); check(top, d, f);
    };
    for (uint32_t d = 1; d < 70000; ++d) divisor(d);
    for (uint32_t s = 3; s < 31; ++s) for (int o = -2; o <= 2; ++o) divisor((1u << s) + o);
    for (uint32_t d = 70001; d < top - 99991; d += d / 7 + 1) divisor(d);
    divisor(top);
    return bad ? 1 : 0;
}
''')
    exe = tmp_path / "t"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2303_08810_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
