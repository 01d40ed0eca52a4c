"""The C-ABI library builds, loads without a GPU, and exports what include/impact.h declares."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_1912_00167_b200 import build, binding
    build.build()
    return binding.load_library()


def _declared():
    text = open(os.path.join(ROOT, "include", "impact.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(impact_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    from paper_1912_00167_b200 import binding
    names = _declared()
    assert len(names) >= 19
    for n in names:
        assert hasattr(lib, n), n
    assert sorted(binding.EXPORTS) == names


def test_housekeeping_calls(lib):
    assert lib.impact_version() == 300
    assert lib.impact_status_string(0) == b"ok"
    assert b"full" in lib.impact_status_string(-5)
    assert b"empty" in lib.impact_status_string(-4)
    assert lib.impact_loss_workspace_bytes(0, 5) == 0
    assert lib.impact_loss_workspace_bytes(1024, 128) >= 1024 * 32


def test_struct_layout_matches_header():
    from paper_1912_00167_b200.binding import impact_coefficients
    assert ctypes.sizeof(impact_coefficients) == 48
    assert impact_coefficients.rho_tw.offset == 16 and impact_coefficients.objective.offset == 32
    assert impact_coefficients.global_steps.offset == 40


def test_host_side_validation_needs_no_gpu(lib):
    # null pointers and bad sizes are refused before any CUDA call
    from paper_1912_00167_b200.binding import impact_coefficients
    cf = impact_coefficients(0.5, 0.01, 0.0, 1.0, 1.0, 0, 0, 0, 0)
    st = lib.impact_loss_fwd_bwd(None, None, None, None, None, None, None, None, 1.0, 1.0, 0.2, ctypes.pointer(cf),
                                 4, 4, 4, 0, None, None, None, None, None, None, 0, None)
    assert st == -1
    fb = (ctypes.c_size_t * 1)(0)
    assert lib.impact_buffer_storage_bytes(4, 1, fb) == 0
    fb = (ctypes.c_size_t * 2)(100, 300)
    assert lib.impact_buffer_storage_bytes(4, 2, fb) == 4 * (256 + 512)
    h = ctypes.c_void_p()
    assert lib.impact_buffer_create(0, 1, 2, fb, 0, 0, None, ctypes.byref(h)) == -1
    assert lib.impact_buffer_create(2, 2, 2, fb, 0, 5, None, ctypes.byref(h)) == -1
    assert lib.impact_gather_rows(None, None, 1, 1, 4, None, None) == -1


def test_ring_bookkeeping_runs_on_caller_storage_without_a_gpu(lib, oracle):
    # with caller-provided storage and no copies requested, push/sample touch only host state
    fb = (ctypes.c_size_t * 1)(64)
    h = ctypes.c_void_p()
    fake_storage = ctypes.c_void_p(256 * 1024)  # never dereferenced: every field source below is NULL
    assert lib.impact_buffer_create(4, 2, 1, fb, 77, 0, fake_storage, ctypes.byref(h)) == 0
    ref = oracle.Ring(4, 2, 0, seed=77)
    src = (ctypes.c_void_p * 1)(None)
    slot, k = ctypes.c_int32(), ctypes.c_int32()
    for i in range(5):
        st = lib.impact_buffer_push(h, src, 0, ctypes.byref(slot), None)
        rst, rslot = ref.push()
        assert (st == -5) == (rst == ref.FULL)
        if st == 0:
            assert slot.value == rslot
    for i in range(9):
        st = lib.impact_buffer_sample(h, ctypes.byref(slot), ctypes.byref(k), None, None)
        rst, rslot, rk = ref.sample()
        assert (st == -4) == (rst == ref.EMPTY)
        if st == 0:
            assert (slot.value, k.value) == (rslot, rk)
    assert lib.impact_buffer_destroy(h) == 0


def test_a_call_packed_as_bytes_is_the_structure(lib):
    """The direct call packs impact_loss_call in one go: the bytes are those of the ctypes structure, field by field."""
    from paper_1912_00167_b200 import binding as b
    head = [11 * (i + 1) for i in range(8)] + [1.5, 2.5, 3.5, 1]
    coef = [0.5, 0.25, 0.125, 4.0, 5.0, 1, 2, 1, 0, 12345678901]
    tail = [7, 8, 9, 1001, 1002, 1003, 0, 1005, 1006, 777, 0, 0]
    want = bytes(b.impact_loss_call(*head, b.impact_coefficients(*coef), *tail))
    assert b._CALL.pack(*head, *coef, *tail) == want
    assert b._call_packed(want, None) == -1  # it reaches the library, which refuses the unaligned addresses


def test_the_direct_call_names_the_argument_at_fault(lib):
    """Arguments that the quick check turns away get the ordinary check's error."""
    import torch
    from paper_1912_00167_b200 import binding as b
    f = lambda *s: torch.zeros(*s)  # (CPU tensors: there is no CPU path)
    with pytest.raises(ValueError, match="learner_logits must be a CUDA tensor"):
        b.impact_loss_fwd_bwd(f(2, 3, 4), f(2, 3, 4), f(2, 3), f(2, 3).int(), f(2, 3), f(2, 3), f(2, 3), f(2),
                              b.Coefficients(), loss_terms=f(8), dlogits=f(2, 3, 4), dvalues=f(2, 3),
                              workspace=torch.zeros(10, dtype=torch.uint8))
    with pytest.raises(ValueError, match="logits must be float32 or bfloat16"):
        b.impact_loss_fwd_bwd(f(2, 3, 4).double(), f(2, 3, 4), f(2, 3), f(2, 3).int(), f(2, 3), f(2, 3), f(2, 3), f(2),
                              b.Coefficients(), loss_terms=f(8), dlogits=f(2, 3, 4), dvalues=f(2, 3),
                              workspace=torch.zeros(10, dtype=torch.uint8))


def _cpu_ring(lib, nbytes):
    import torch
    from paper_1912_00167_b200 import binding as b
    N = 3
    raw = torch.zeros(b.ImpactBuffer.storage_bytes(N, nbytes) + 256, dtype=torch.uint8)
    at = -raw.data_ptr() % 256
    return b.ImpactBuffer(N, 2, nbytes, storage=raw[at:at + raw.numel() - 256])


def test_nothing_needs_the_native_check_of_direct_calls(lib):
    """Without the binding's native part the library loads and a direct loss call is checked in Python: it says so once, and
    names the argument at fault."""
    import subprocess
    import sys
    code = """
import sys, warnings
import torch
import paper_1912_00167_b200 as ip
from paper_1912_00167_b200.build import marshal_name
sys.modules["paper_1912_00167_b200." + marshal_name()] = None
assert ip.load_library() is not None and ip.impact_version() > 0
with warnings.catch_warnings(record=True) as said:
    warnings.simplefilter("always")
    z, v = torch.zeros(2, 3, 4), torch.zeros(2, 3)
    for _ in range(2):
        try:
            ip.impact_loss_fwd_bwd(z, z, v, v.int(), v, v, v, v[:, 0], ip.Coefficients(), loss_terms=torch.zeros(8), dlogits=z,
                                   dvalues=v, workspace=torch.zeros(64, dtype=torch.uint8))
        except ValueError as e:
            assert "learner_logits" in str(e), e
        else:
            raise SystemExit("served")
assert len(said) == 1 and "rebuild" in str(said[0].message), said
"""
    done = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert done.returncode == 0, done.stderr


def test_the_native_part_builds_with_nvcc_by_any_name(lib, monkeypatch, tmp_path):
    """A bare name that is found on the path, and a wrapper that lies elsewhere."""
    import shutil
    import subprocess
    from paper_1912_00167_b200 import build
    real = shutil.which(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))
    wrapper = tmp_path / "nvcc"
    wrapper.write_text('#!/bin/sh\nexec "%s" "$@"\n' % real)
    wrapper.chmod(0o755)
    monkeypatch.setattr(build, "marshal_path", lambda: str(tmp_path / "made.so"))
    for name, path in (("nvcc", os.path.dirname(real)), (str(wrapper), None)):
        monkeypatch.setenv("NVCC", name)
        if path:
            monkeypatch.setenv("PATH", path + os.pathsep + os.environ["PATH"])
        build.build_marshal()
        names = subprocess.run(["nm", "-D", "--defined-only", build.marshal_path()], capture_output=True, text=True, check=True)
        assert "PyInit_" + build.marshal_name() in names.stdout
        os.remove(build.marshal_path())


def test_a_native_part_built_for_another_torch_is_not_this_one(lib, monkeypatch):
    """The module's name says what it was built for: with another torch (or Python) the one that is there counts as missing, is
    not loaded, and a build makes a new one."""
    import torch
    from paper_1912_00167_b200 import binding as b, build
    assert os.path.exists(build.marshal_path()) and not build.needs_build()
    name = build.marshal_name()
    monkeypatch.setattr(b, "_loss_direct", b._bind_loss_direct)
    assert b._loss_direct(*[None] * 17) is None and b._loss_direct.__module__ == "_marshal"  # (found; it serves no such call)
    for what, value in (("__version__", "2.12.0"), ("version", type("version", (), dict(git_version="0" * 40)))):
        with monkeypatch.context() as other:
            other.setattr(torch, what, value)
            assert build.marshal_name() != name and build.needs_build()
            other.setattr(b, "_loss_direct", b._bind_loss_direct)
            with pytest.warns(RuntimeWarning, match="rebuild"):
                assert b._loss_direct(*[None] * 17) is None
            assert b._loss_direct is b._not_served
    with monkeypatch.context() as other:
        other.setattr(build.sysconfig, "get_config_var", lambda name: "cpython-313-x86_64-linux-gnu")
        assert build.marshal_name() != name and build.needs_build()


def test_a_slot_view_is_the_slots_bytes_and_nothing_else(lib):
    """Views of every shape and type name the bytes that the library names; a closed buffer and bad places are refused."""
    import torch
    ring = _cpu_ring(lib, [4 * 35, 2 * 35 * 3])
    for slot in range(3):
        for field, dtype, shape in ((0, torch.float32, (5, 7)), (0, torch.int32, (35,)), (1, torch.bfloat16, (5, 7, 3)),
                                    (1, torch.uint8, (210,)), (0, torch.float32, [5, 7]), (0, torch.float32, (5, -1))):
            view = ring.slot_view(slot, field, dtype, shape)
            assert view.data_ptr() == ring.slot_ptr(slot, field) and view.dtype is dtype and view.is_contiguous()
            assert view.nbytes == ring.field_bytes[field]
    for bad in ((3, 0), (-1, 0), (0, 2)):
        with pytest.raises(ValueError):
            ring.slot_view(*bad, torch.float32, (5, 7))
    with pytest.raises(RuntimeError):
        ring.slot_view(0, 0, torch.float32, (5, 8))
    ring.close()
    with pytest.raises(ValueError):
        ring.slot_view(0, 0, torch.float32, (5, 7))


@pytest.mark.parametrize("native", [True, False])
def test_a_prepared_step_keeps_its_buffer_and_ends_with_it(lib, monkeypatch, native):
    """The call holds the handle by its address: the buffer is there for as long as the call is, and a closed one is refused
    before anything looks at the handle."""
    import gc
    import torch
    import weakref
    from paper_1912_00167_b200 import binding as b
    if not native:
        monkeypatch.setattr(b, "_marshal", False)
    ring = _cpu_ring(lib, [4 * 35, 24])
    step = ring.prepare_device_step({"rewards": 0}, record=torch.zeros(128, dtype=torch.uint8))
    assert (step._capsule is not None) == native
    ref = weakref.ref(ring)
    del ring
    gc.collect()
    assert ref() is not None and ref()._h
    for call in (step, step.on_stream):
        with pytest.raises(b.ImpactError):  # (the library's own: not in device mode)
            call(0)
    ref().close()

    def issued(*args):
        raise AssertionError("a closed buffer's handle")

    step._fn = step._issue = issued
    for call in (step, step.on_stream):
        with pytest.raises(b.ImpactError) as e:
            call(0)
        assert e.value.status == b.ERR_INVALID_ARG


def test_a_slot_view_does_not_depend_on_earlier_ones(lib):
    """A first view, or the buffer itself, made under inference mode leaves later views ordinary tensors that autograd may
    save."""
    import torch
    ring = _cpu_ring(lib, [4 * 35])
    with torch.inference_mode():
        from paper_1912_00167_b200 import binding as b
        ring.slot_view(0, 0, torch.float32, (5, 7))
        other = b.ImpactBuffer(3, 2, [4 * 35], storage=ring._storage)
    for r in (ring, other):
        weight = torch.ones(5, 7, requires_grad=True)
        (weight * r.slot_view(0, 0, torch.float32, (5, 7))).sum().backward()
        assert weight.grad is not None


def test_two_copies_of_the_library_share_nothing(lib):
    """No exported symbol is of the kind that a process merges across libraries: a launch rule's per-device state is one
    copy's own."""
    import subprocess
    from paper_1912_00167_b200 import binding as b
    names = subprocess.run(["nm", "-D", "--defined-only", b.LIB_PATH], capture_output=True, text=True, check=True).stdout
    assert "impact_loss_fwd_bwd" in names
    assert not [line for line in names.splitlines() if line.split()[-2] == "u"]
