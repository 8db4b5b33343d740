"""The Python extension that marshals calls: words converted to the declared parameter types, specs that do not
fit a function refused, a file name that names the interpreter.  No GPU: the calls return before they would
use one."""
import ctypes as C
import sysconfig

import pytest

from paper_2604_10235_b200 import binding, build


@pytest.fixture()
def handle():
    lib = binding.load_library()
    context = C.create_string_buffer(4096)       # a context that was never created: argument checks only
    return lib, C.addressof(context), context


def test_words_become_the_declared_types(handle):
    lib, ctx, _keep = handle
    select = lib.calls["cc_select_chunks"]       # (ctx, score, num_chunks, k, chosen, stream)
    assert select(0, None, 1, 1, None, 0) == binding.CC_ERR_INVALID_ARG
    assert select(ctx, None, -1, 1, None, 0) == binding.CC_ERR_INVALID_ARG           # 32 bits, sign and all
    assert select(ctx, None, 8193, 1, None, 0) == binding.CC_ERR_UNSUPPORTED
    assert select(ctx, None, 8192, 0, None, 0) == binding.CC_OK
    assert select(ctx, None, 5 + 2 ** 32, 0, None, 2 ** 64 - 1) == binding.CC_OK     # masked, as ctypes does
    assert lib.calls["cc_ppl_chunk_scores"](ctx, None, binding.CC_F32, 0, 1, 7, 2 ** 40, 7, None, None, None,
                                            0) == binding.CC_OK


def test_wrong_arguments_raise(handle):
    lib, ctx, _keep = handle
    select = lib.calls["cc_select_chunks"]
    with pytest.raises(TypeError):
        select(ctx, None, 1, 1, None)
    with pytest.raises(TypeError):
        select(ctx, None, 1.5, 1, None, 0)
    with pytest.raises(AttributeError):
        select(ctx, object(), 1, 1, None, 0)
    import torch
    with pytest.raises(ValueError):
        select(ctx, torch.zeros(1), 1, 1, None, 0)


def test_specs_that_do_not_fit_are_refused():
    binding.load_library()
    for name, spec in (("cc_select_chunks", b"itiit"), ("cc_select_chunks", b"itiitii"), ("cc_select_chunks", b"itiit?"),
                       ("cc_create", b"ii"), ("no_such_function", b"i")):
        with pytest.raises(ValueError):
            binding._BIND(name, 0, spec)


def test_file_is_tagged_with_the_interpreter():
    assert build.CALL_PATH.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert sysconfig.get_config_var("SOABI") in build.CALL_PATH
