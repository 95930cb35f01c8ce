"""Host-side checks of the C-ABI library that need no GPU: it loads, exports every symbol the
header declares, and classifies expressions (Sec. 2.2) without a device."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def binding():
    from paper_2404_04541_b200 import build, binding
    build.build()
    return binding


def declared_functions():
    text = open(os.path.join(ROOT, "include", "spws.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(spws_[a-z_0-9]+)\s*\(", text)))


def test_library_exports_every_declared_symbol(binding):
    names = declared_functions()
    assert len(names) >= 12
    L = ctypes.CDLL(binding.LIB_PATH)
    for n in names:
        assert hasattr(L, n), f"{n} declared in spws.h but not exported"
    assert set(names) == set(binding.EXPORTS)


def test_status_strings(binding):
    seen = {binding.status_string(s) for s in range(0, 11)}
    assert len(seen) == 11 and "ok" in seen
    assert binding.status_string(99) == "unknown status"


@pytest.mark.parametrize("expr,fmts,ok", [
    ("C(i,j)=A(i,k)*B(k,j)", (0, 0, 0), True),
    ("  Out( r , c ) = X(r, t) * Y( t ,c)", (0, 0, 0), True),
    ("C(i,j) += A(i,k) * B(k,j)", (0, 0, 0), True),
    ("C(i,j,l)=A(i,j,k)*B(k,l)", (1, 1, 0), True),
    ("Z(a,b,c) = T(a,b,x) * M(x,c)", (1, 1, 0), True),
    ("C(i,j)=A(i,k)*B(k,j)", (0, 1, 0), False),        # formats do not fit the order
    ("C(i,j,l)=A(i,j,k)*B(k,l)", (0, 0, 0), False),
    ("C(i,j)=A(k,i)*B(k,j)", (0, 0, 0), True),         # outer-product order: second-order scatter
    ("R(u,v) = P(w,u) * Q(w,v)", (0, 0, 0), True),
    ("C(i,j)=A(k,i)*B(k,j)", (0, 1, 0), False),
    ("C(i,j)=A(k,j)*B(k,i)", (0, 0, 0), False),        # outer-product order with the output transposed
    ("C(j,i)=A(i,k)*B(k,j)", (0, 0, 0), False),        # transposed output
    ("C(i,j)=A(i,k)*B(j,k)", (0, 0, 0), False),        # B accessed against its storage order
    ("C(i,j)=A(i,j)*B(i,j)", (0, 0, 0), False),        # element-wise: no reduction variable
    ("C(i,j,l)=A(k,i,j)*B(k,l)", (1, 1, 0), False),    # contraction of the outermost mode needs a COO result
    ("C(i,j,l)=A(k,i,j)*B(k,l)", (2, 1, 0), True),     # SpTTM, third-order scatter
    ("C(k,j,l)=A(k,i,j)*B(i,l)", (2, 1, 0), True),     # SpTTM-I
    ("C(i,j,l)=A(i,j,k)*B(k,l)", (2, 1, 0), False),    # the first-order form has a CSF result
    ("C(k,j,l)=A(k,i,j)*B(i,l)", (2, 0, 0), False),
    ("C(i,j)=A(i,k)+B(k,j)", (0, 0, 0), False),
    ("C(i,j)=A(i,k)*B(k,j)*D(j,j)", (0, 0, 0), False),
    ("C(i,i)=A(i,k)*B(k,i)", (0, 0, 0), False),
    ("C(i,j)=C(i,k)*B(k,j)", (0, 0, 0), False),
    ("C(i,j)=A(i,k)*B(k,j", (0, 0, 0), False),
    ("", (0, 0, 0), False),
])
def test_expression_classification(binding, expr, fmts, ok):
    st = binding.check_expression(expr, fmts)
    assert st == (binding.SPWS_OK if ok else binding.SPWS_UNSUPPORTED_EXPRESSION)


def test_tensor_arrays_with_unused_levels_left_out(binding):
    """Level lists as short as the order, dims without the unused one and sizes of any number type give the same C
    struct as their full forms; arrays without elements have no address."""
    import numpy as np
    import torch
    pos, crd, val = torch.zeros(4, dtype=torch.int64), torch.zeros(5, dtype=torch.int32), torch.zeros(5)
    full = bytes(binding.TensorArrays(2, (3, 7, 0), [None, pos, None], [None, crd, None], val, [3, 5, 0]).c_struct())
    for dims, p, c, n in (((3, 7), [None, pos], [None, crd], [3, 5, 0]), ((3, 7, 0), [None, pos, None], [None, crd], [3, 5, 0]),
                          ((3, 7), [None, pos, None], [None, crd, None], [np.int64(3), torch.tensor(5), 0]),
                          ((np.int32(3), 7.0), [None, pos, None], [None, crd, None], [3.0, 5.0, 0])):
        assert bytes(binding.TensorArrays(2, dims, p, c, val, n).c_struct()) == full
    empty = binding.TensorArrays(2, (0, 7), [None, pos[:0]], [], np.empty(0), [0, 0, 0]).c_struct()
    assert not any(empty.pos) and not any(empty.crd) and not empty.val and list(empty.dims) == [0, 7, 0]
    cube = binding.TensorArrays(3, (2, 3, 4), [pos, pos, pos], [crd, crd, crd], val, [1, 2, 5]).c_struct()
    assert list(cube.dims) == [2, 3, 4] and set(cube.pos) == {pos.data_ptr()} and list(cube.n) == [1, 2, 5]


def test_no_device_is_reported_not_faked(binding):
    """Without a CUDA device the library reports an error; it never computes on the CPU."""
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present")
    with pytest.raises(binding.SpwsError) as e:
        binding.Handle()
    assert e.value.status == binding.SPWS_CUDA_ERROR
    from paper_2404_04541_b200 import api
    with pytest.raises(RuntimeError):
        api.Context()


def test_chained_kernels_load_nothing_read_only_before_their_wait():
    """A kernel whose blocks are placed before the kernel ahead of it is done may not load through a read-only pointer at an address
    that it knows on entry, unless the pointer has passed not_before()."""
    folder = os.path.join(ROOT, "paper_2404_04541_b200", "csrc")
    seen = 0
    for name in sorted(os.listdir(folder)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(folder, name)).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+_kernel)\(([^{;]*)\)\s*\{(.*?)\n\}", text, flags=re.S):
            kernel, params, body = m.groups()
            if "chained_start(" not in body:
                continue
            seen += 1
            known = {re.search(r"(\w+)\s*$", p).group(1) for p in params.split(",")}
            for pointer in re.findall(r"const \w+\* __restrict__ (\w+)", params):
                for at in re.findall(r"\b%s(?:\[| \+ )\s*(\w+)" % pointer, body):
                    assert at not in known and not at.isdigit() or f"not_before({pointer})" in body, (kernel, pointer, at)
    assert seen >= 12


def test_bounds_lists_hold_as_many_rows_however_many_blocks_are_resident():
    """The blocks of the bounds kernel that are resident at once list at least as many long and mid rows together as 16 blocks an SM
    with lists of 32 and 64."""
    text = open(os.path.join(ROOT, "paper_2404_04541_b200", "csrc", "setup.cu")).read()
    blocks = [int(x) for x in re.search(r"__launch_bounds__\(256, SUMMARY \? (\d+) : (\d+)\) row_bounds_kernel", text).groups()]
    for name, least in (("LONG_LIST", 16 * 32), ("MID_LIST", 16 * 64)):
        assert min(blocks) * int(re.search(r"constexpr int %s = (\d+);" % name, text).group(1)) >= least
