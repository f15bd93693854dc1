"""CPU-side checks of the boundary: the shared library builds, loads and exports every symbol
the header declares (no compute calls: there is no GPU here)."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "elitekv.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(elitekv_[a-z_]+)\s*\(", text)))


def test_header_declares_the_three_hot_path_calls():
    names = _declared_symbols()
    for must in ("elitekv_append", "elitekv_absorb_query", "elitekv_decode"):
        assert must in names


def test_library_builds_and_exports_every_declared_symbol():
    from paper_2503_01586_b200 import build
    path = build.build()
    assert os.path.exists(path)
    lib = ctypes.CDLL(path)
    for name in _declared_symbols():
        assert hasattr(lib, name), name
    lib.elitekv_strerror.restype = ctypes.c_char_p
    assert lib.elitekv_strerror(0) == b"ok"
    assert b"page" in lib.elitekv_strerror(-6)


def test_binding_exposes_the_same_names():
    from paper_2503_01586_b200 import binding
    for name in _declared_symbols():
        if name in ("elitekv_layer_create", "elitekv_layer_destroy", "elitekv_strerror"):
            continue   # wrapped by binding.Layer / binding.strerror
        assert hasattr(binding, name), name


def test_search_workspace_is_what_the_call_uses():
    """Single distances and one round bring no room for sums between rounds, whose size is a head's pairs; the least is tables
    and item results, as for a search that never keeps anything."""
    from paper_2503_01586_b200 import binding as ek
    for H, n, d_h in ((32, 2048, 128), (4, 300, 64), (1, 1, 64), (1024, 2048, 128), (2, 1 << 20, 128)):
        most = ek.elitekv_ropelite_workspace_size(H, n, d_h)
        least = ek.elitekv_ropelite_workspace_size_rounds(H, n, d_h, 0)
        for r in (1, 2, 8, d_h // 2):
            assert least <= ek.elitekv_ropelite_workspace_size_rounds(H, n, d_h, r) <= most
        # (cos, sin) and sines, items of a 128 x 128 tile at most, masks; four paddings to 256 bytes
        half, tiles = d_h // 2, (n + 127) // 128
        items = min(tiles * (tiles + 1) // 2, 16 * tiles) if n > 128 else max(tiles, -(-n // 16))
        assert least <= half * (12 * n + 4 * (128 + 256) + 4 * H * items) + 8 * H + 1024
    assert ek.elitekv_ropelite_workspace_size_rounds(32, 2048, 128, 1) < 3 << 20 < 300 << 20 < \
        ek.elitekv_ropelite_workspace_size_rounds(32, 2048, 128, 8)
    for bad in (-1, 65):
        with pytest.raises(ek.ElitekvError):
            ek.elitekv_ropelite_workspace_size_rounds(4, 300, 128, bad)


def test_struct_layouts_match_the_header(tmp_path):
    """sizeof/offsetof as the C compiler sees the header vs. the ctypes mirror."""
    import subprocess
    from paper_2503_01586_b200 import binding
    src = tmp_path / "layout.c"
    fields_p = [f[0] for f in binding.Params._fields_]
    fields_c = [f[0] for f in binding.CacheDesc._fields_]
    lines = ['#include <stdio.h>', '#include <stddef.h>', '#include "elitekv.h"', 'int main(void){',
             'printf("%zu\\n", sizeof(elitekv_params));']
    lines += [f'printf("%zu\\n", offsetof(elitekv_params, {f}));' for f in fields_p]
    lines += ['printf("%zu\\n", sizeof(elitekv_cache));']
    lines += [f'printf("%zu\\n", offsetof(elitekv_cache, {f}));' for f in fields_c]
    lines += ['return 0;}']
    src.write_text("\n".join(lines))
    exe = tmp_path / "layout"
    subprocess.run(["gcc", "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True)
    got = [int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]
    want = [ctypes.sizeof(binding.Params)] + [getattr(binding.Params, f).offset for f in fields_p]
    want += [ctypes.sizeof(binding.CacheDesc)] + [getattr(binding.CacheDesc, f).offset for f in fields_c]
    assert got == want


def test_copy_takes_no_memory_of_another_device(tmp_path):
    """The rule of elitekv_copy on the attributes that the runtime reports of a pointer."""
    import subprocess
    src = tmp_path / "rule.cpp"
    src.write_text('''#include "copy.cuh"
#include <cstdio>
#include <initializer_list>
int main() {
  char x, y;
  const cudaMemoryType kinds[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged};
  for (cudaMemoryType k : kinds)
    for (int device = 0; device < 2; ++device)
      for (void* p : {(void*)&x, (void*)&y}) {
        cudaPointerAttributes at = {};
        at.type = k; at.device = device; at.devicePointer = p;
        std::printf("%d", (int)ekv_addressable(at, &x, 0));
      }
}''')
    exe = tmp_path / "rule"
    subprocess.run(["g++", "-std=c++17", "-I/usr/local/cuda/include", "-I", os.path.join(ROOT, "paper_2503_01586_b200", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    # same address or another, on this device and on another one: unregistered, pinned, device, managed
    assert got == "0000" + "1010" + "1000" + "1010"
