"""CPU-only checks of the boundary: the library loads and exports every declared symbol,
and the host-side validation paths that need no device work behave as documented."""
import ctypes as C
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_1911_00472_b200 import build
    path = build.build()
    return C.CDLL(path)


def _declared():
    text = open(os.path.join(ROOT, "include", "pcr.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(pcr_[a-z_]+)\s*\(", text)))


def test_library_exports_every_declared_symbol(lib):
    names = _declared()
    assert {"pcr_open", "pcr_decode", "pcr_close"} <= set(names)
    for n in names:
        assert hasattr(lib, n), n


def test_binding_lists_the_same_names():
    from paper_1911_00472_b200 import binding
    assert sorted(binding.EXPORTS) == _declared()


def test_argument_errors_need_no_device(lib):
    lib.pcr_open.argtypes = [C.c_void_p, C.c_size_t, C.POINTER(C.c_void_p)]
    h = C.c_void_p()
    assert lib.pcr_open(None, 10, C.byref(h)) == -1
    buf = (C.c_uint8 * 128)()
    assert lib.pcr_open(buf, 128, C.byref(h)) == -2 and not h.value       # bad magic
    assert lib.pcr_open(buf, 10, C.byref(h)) == -2                          # too short
    lib.pcr_num_images.argtypes = [C.c_void_p]
    assert lib.pcr_num_images(None) == -1
    lib.pcr_out_bytes.restype = C.c_size_t
    lib.pcr_out_bytes.argtypes = [C.c_void_p]
    assert lib.pcr_out_bytes(None) == 0
    lib.pcr_decode.argtypes = [C.c_void_p, C.c_int, C.c_void_p, C.c_void_p]
    assert lib.pcr_decode(None, 1, None, None) == -1
    lib.pcr_close.argtypes = [C.c_void_p]
    lib.pcr_close(None)
    lib.pcr_strerror.restype = C.c_char_p
    assert lib.pcr_strerror(-3) == b"corrupt entropy-coded data"


@pytest.mark.parametrize("cache", [0, 1 << 30])
def test_offsets_near_the_end_of_the_64_bit_range(tmp_path, lib, cache):
    """Offsets so large that adding a length to them wraps are refused like any other offset past the end; with the cache of
    closed records on too, which looks at the record before it is opened.  (In a child, behind a page without access: a wrong
    check reads in front of the record.)"""
    import struct
    import subprocess
    import sys
    import pcr_synth
    rec = pcr_synth.make_record(0, n_images=3).bytes
    index_off = struct.unpack_from("<Q", rec, 32)[0]
    chunk = index_off + 8 * 11
    names = []
    for at in (24, 32, 40, index_off, index_off + 8 * 10, chunk, chunk + 16 * 7):      # meta, index, data, group ends, chunks
        for value in ((1 << 64) - 16, (1 << 64) - 64, (1 << 63), (1 << 32) - 16):
            bad = rec.copy()
            struct.pack_into("<Q", bad, at, value)
            names.append(str(tmp_path / f"{at}_{value}"))
            bad.tofile(names[-1])
    code = ("import ctypes, mmap, sys\n"
            "lib = ctypes.CDLL(sys.argv[1])\n"
            "lib.pcr_set_record_cache.argtypes = [ctypes.c_size_t]\n"
            "lib.pcr_set_record_cache(int(sys.argv[2]))\n"
            "lib.pcr_open.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.POINTER(ctypes.c_void_p)]\n"
            "page = mmap.PAGESIZE\n"
            "libc = ctypes.CDLL(None, use_errno=True)\n"
            "libc.mprotect.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]\n"
            "for name in sys.argv[3:]:\n"
            "    raw, h = open(name, 'rb').read(), ctypes.c_void_p()\n"
            "    m = mmap.mmap(-1, page + len(raw))\n"
            "    m[page:] = raw\n"
            "    at = ctypes.addressof(ctypes.c_char.from_buffer(m))\n"
            "    assert libc.mprotect(at, page, 0) == 0\n"
            "    print(lib.pcr_open(at + page, len(raw), ctypes.byref(h)), flush=True)\n"
            "    libc.mprotect(at, page, 3)\n")
    res = subprocess.run([sys.executable, "-c", code, lib._name, str(cache)] + names, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""),
                         capture_output=True, text=True, timeout=120)
    assert res.returncode == 0 and res.stdout.split() == ["-2"] * len(names), res


def test_open_without_threads_to_be_had(tmp_path, lib):
    """pcr_open walks the images on a few threads; where none can be started it does the work itself, and nothing is thrown
    through the C ABI.  (A preloaded pthread_create that always fails; no device, so a valid record ends with PCR_E_CUDA.)"""
    import subprocess
    import sys
    import pcr_synth
    rec = pcr_synth.make_record(0, n_images=200)
    rec.bytes.tofile(tmp_path / "record")
    damaged = rec.bytes.copy()
    damaged[int.from_bytes(damaged[40:48].tobytes(), "little") + 4] ^= 0xFF       # the first image's first marker segment
    damaged.tofile(tmp_path / "damaged")
    (tmp_path / "shim.c").write_text("#include <errno.h>\nint pthread_create(void* a, const void* b, void* (*f)(void*), void* p) "
                                     "{ (void)a; (void)b; (void)f; (void)p; return EAGAIN; }\n")
    shim = tmp_path / "shim.so"
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-o", str(shim), str(tmp_path / "shim.c")])
    code = ("import ctypes, sys\n"
            "lib = ctypes.CDLL(sys.argv[1])\n"
            "lib.pcr_open.argtypes = [ctypes.c_char_p, ctypes.c_size_t, ctypes.POINTER(ctypes.c_void_p)]\n"
            "for name in sys.argv[2:]:\n"
            "    raw, h = open(name, 'rb').read(), ctypes.c_void_p()\n"
            "    print(lib.pcr_open(raw, len(raw), ctypes.byref(h)))\n")
    env = dict(os.environ, LD_PRELOAD=str(shim), CUDA_VISIBLE_DEVICES="")
    res = subprocess.run([sys.executable, "-c", code, lib._name, str(tmp_path / "record"), str(tmp_path / "damaged")], env=env,
                         capture_output=True, text=True, timeout=120)
    assert res.returncode == 0 and res.stdout.split() == ["-5", "-2"], res


def test_product_path_does_not_touch_the_oracle():
    """Neither the package nor the generator imports or mentions the oracle."""
    for folder in ("paper_1911_00472_b200", "pcr_synth"):
        for dirpath, _, files in os.walk(os.path.join(ROOT, folder)):
            for f in files:
                if f.endswith((".py", ".cu", ".cuh", ".h", ".c")):
                    text = open(os.path.join(dirpath, f)).read()
                    assert "import oracle" not in text and "from oracle" not in text and "pcr_oracle" not in text, f
