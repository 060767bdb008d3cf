"""CPU-side checks of the boundary: the shared library loads and exports every symbol the
header declares; the binding's structs match the header's field order."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2603_14549_b200 import binding as A
from paper_2603_14549_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = open(os.path.join(ROOT, "include", "asap.h")).read()


@pytest.fixture(scope="module")
def lib():
    build.build_library()
    return ctypes.CDLL(A.LIB_PATH)


def test_every_declared_symbol_is_exported(lib):
    declared = set(re.findall(r"\b(asap_[a-z_]+)\s*\(", HEADER))
    assert declared == set(A.EXPORTS), declared ^ set(A.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


@pytest.mark.parametrize("lang,std", [("c", "c99"), ("c++", "c++17")])
def test_the_header_is_c_and_declares_every_function(tmp_path, lang, std):
    """A C program that takes the address of every exported function compiles against the header alone."""
    src = tmp_path / "use.c"
    src.write_text('#include "asap.h"\nvoid *use[] = {' + ", ".join(f"(void *)&{n}" for n in A.EXPORTS) + "};\n"
                   "unsigned long size(void) { return (unsigned long)sizeof(asap_kernel_time); }\n")
    res = subprocess.run(["gcc", "-x", lang, f"-std={std}", "-Wall", "-Wextra", "-Werror", "-fsyntax-only",
                          "-I", os.path.join(ROOT, "include"), str(src)], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr


def _struct_fields(name):
    body = re.search(r"typedef struct \{([^}]*)\}\s*" + name + ";", HEADER, re.S).group(1)
    body = re.sub(r"/\*.*?\*/", "", body, flags=re.S)
    fields = []
    for decl in body.split(";"):
        decl = decl.strip()
        if not decl:
            continue
        for part in decl.split(","):
            fields.append(re.findall(r"\*?\s*([A-Za-z_0-9]+)\s*(?:\[\d+\])?$", part.strip())[0])
    return fields


@pytest.mark.parametrize("cname,cls", [("asap_inputs", A.CInputs), ("asap_params", A.CParams),
                                       ("asap_outputs", A.COutputs), ("asap_kernel_time", A.CKernelTime)])
def test_binding_struct_matches_header(cname, cls):
    assert _struct_fields(cname) == [f[0] for f in cls._fields_]


def test_init_without_gpu_fails_cleanly(lib):
    import torch
    if torch.cuda.is_available():
        pytest.skip("a GPU is present")
    with pytest.raises(A.AsapError):
        A.asap_init(0, 1000, 1, 1, 128)


def test_missing_library_is_a_loud_error(monkeypatch, tmp_path):
    monkeypatch.setattr(A, "_lib", None)
    monkeypatch.setattr(A, "LIB_PATH", str(tmp_path / "libasap.so"))
    with pytest.raises(FileNotFoundError):
        A.load_library()
