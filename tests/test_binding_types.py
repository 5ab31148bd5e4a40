"""The binding's declared types against include/msp.h: every entry point has its
argument types and its result type, so that neither an address nor a count of
bytes is cut to 32 bits on the way."""
import ctypes as C
import os
import re

import pytest

from paper_2301_10570_gb300 import build, msp

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include", "msp.h")
SCALARS = {"int": C.c_int, "int64_t": C.c_int64, "uint64_t": C.c_uint64, "double": C.c_double}


def _declarations():
    with open(HEADER) as f:
        text = re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S)
    for res, name, args in re.findall(r"^([\w ]+?[ *]+)(msp_[a-z_]+)\(([^;]*)\);", text, flags=re.M):
        yield name, res.strip(), [a.strip() for a in args.split(",")]


@pytest.mark.parametrize("name,res,args", list(_declarations()), ids=lambda v: v if isinstance(v, str)
                         and v.startswith("msp_") else "")
def test_types_are_declared_as_in_the_header(name, res, args):
    build.build()
    fn = getattr(msp.load(), name)
    want = {"msp_status": C.c_int, "const char *": C.c_char_p, "const char*": C.c_char_p}
    assert fn.restype is want.get(res, SCALARS.get(res)), name
    if args == ["void"]:
        assert not fn.argtypes
        return
    assert fn.argtypes is not None and len(fn.argtypes) == len(args), name
    for t, a in zip(fn.argtypes, args):
        if "*" in a:
            assert t is C.c_void_p or issubclass(t, C._Pointer), (name, a)
        else:
            assert t is SCALARS[a.split()[-2]], (name, a)


def test_every_exported_entry_point_is_in_the_header():
    assert sorted(n for n, _, _ in _declarations()) == sorted(msp.EXPORTED)
