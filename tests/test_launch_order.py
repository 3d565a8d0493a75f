"""The order that the host code gives its launches, on a machine without a GPU: linked with a stand-in for the CUDA runtime
(tests/cuda/fake_runtime.c). What a failed call leaves behind, by failing the n-th for every n; which launches may start early; and
grids at the largest sizes."""
import ctypes
import os
import random
import subprocess

import pytest

from paper_2406_05317_b200 import build


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    objects = sorted((build.PKG / "_build").glob("*.o"))
    if len(objects) < len(build.sources()) or build.stale():
        build.build(force=True)
        objects = sorted((build.PKG / "_build").glob("*.o"))
    out = tmp_path_factory.mktemp("fake") / "liblococo_fake.so"
    src = build.PKG.parent / "tests" / "cuda" / "fake_runtime.c"
    obj = out.with_suffix(".o")
    subprocess.check_call(["gcc", "-O1", "-w", "-fPIC", "-c", str(src), "-o", str(obj)])
    layout = out.with_name("group_layout.o")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-I", str(build.INCLUDE),
                           "-I", str(build.CSRC), "-c", str(src.with_name("group_layout.cpp")), "-o", str(layout)])
    # (its own names first: another CUDA runtime may be loaded in this process)
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-o", str(out), str(obj), str(layout), *map(str, objects)])
    lib = ctypes.CDLL(str(out))
    lib.fake_stream.restype = ctypes.c_void_p
    lib.fake_calls.restype = lib.fake_queries.restype = ctypes.c_long
    lib.fake_fail_at.argtypes = [ctypes.c_long]
    lib.fake_joined.argtypes = [ctypes.c_void_p]
    lib.fake_capture.argtypes = [ctypes.c_ulonglong]
    from paper_2406_05317_b200 import api
    lib.fake_group_overrun.restype = ctypes.c_longlong
    lib.fake_group_overrun.argtypes = [ctypes.POINTER(api.Config), ctypes.c_int, ctypes.c_int, ctypes.c_size_t, ctypes.c_void_p]
    for name, args in api._SIGNATURES.items():
        getattr(lib, name).argtypes = args
    return lib


def test_a_failed_backward_leaves_nothing_beside_the_callers_stream(fake):
    # The backward pass runs part of a step on a stream of its own. Whichever call fails, the caller learns of it, and everything
    # that was queued is ahead of what the caller queues next on their stream: their buffers may be freed in its order.
    from paper_2406_05317_b200 import api
    batch, heads, d, M, k, B, L = 1, 2, 64, 40, 5, 100, 350
    stream = fake.fake_stream()
    handle = ctypes.c_void_p()
    cfg = api.Config(batch, heads, d, M, k, d, 0, api.BF16, 0.0, 1e-6, B, api.PATH_AUTO)
    at = 1 << 30                       # nothing reads the memory: any aligned address will do
    view = lambda tokens: api.Tensor(at, heads * tokens * d, tokens * d, d)
    none = api.Tensor(None, 0, 0, 0)
    size = ctypes.c_size_t()

    def backward():
        tokens, cache = view(L), view(M)
        return fake.lococo_process_sequence_backward(
            handle, tokens, tokens, tokens, tokens, L, B, 0, at, tokens, cache, cache, tokens, tokens, tokens, at, None, none, none,
            at, size.value, stream)

    n = total = 0
    while n <= total:                  # n = 0: nothing fails
        fake.fake_fail_at(0)
        assert fake.lococo_create(ctypes.byref(cfg), ctypes.byref(handle)) == api.OK
        assert fake.lococo_workspace_bytes(handle, ctypes.byref(size)) == api.OK
        assert fake.lococo_set_workspace(handle, at, size.value, stream) == api.OK
        assert fake.lococo_set_weights(handle, at, None, stream) == api.OK
        assert fake.lococo_backward_scratch_bytes(handle, L, B, ctypes.byref(size)) == api.OK
        fake.fake_fail_at(n)
        status = backward()
        if n == 0:
            total = fake.fake_calls()
            assert total > 40
        assert status == (api.OK if n == 0 else api.ERR_CUDA), n
        assert fake.fake_joined(stream), n
        fake.lococo_destroy(handle)
        n += 1


@pytest.mark.parametrize("tokens", [1, 8])     # the generation stage's kernel; the short chunks'
def test_weights_are_read_early_only_behind_a_kernel_that_waited_for_them(fake, tokens):
    # Both kernels ask for weight tiles before they wait for the kernel before them, which is sound only where that kernel itself
    # came after the packing: not straight after lococo_set_weights, and not because a step was recorded that has not run.
    from paper_2406_05317_b200 import api
    stream = fake.fake_stream()
    handle, size = ctypes.c_void_p(), ctypes.c_size_t()
    cfg = api.Config(1, 4, 128, 128, 5, 128, 0, api.BF16, 0.0, 1e-6, tokens, api.PATH_AUTO)
    at = 1 << 30
    fake.fake_fail_at(0)
    assert fake.lococo_create(ctypes.byref(cfg), ctypes.byref(handle)) == api.OK
    assert fake.lococo_workspace_bytes(handle, ctypes.byref(size)) == api.OK
    assert fake.lococo_set_workspace(handle, at, size.value, stream) == api.OK

    def set_weights():
        assert fake.lococo_set_weights(handle, at, None, stream) == api.OK

    def step(K_cache):                 # (a cache of its own each time: no call repeats another)
        view = lambda ptr, n: api.Tensor(ptr, 4 * n * 128, n * 128, 128)
        c = ctypes.c_int32(128)
        chunk = view(at, tokens)
        assert fake.lococo_process_sequence(handle, chunk, chunk, chunk, tokens, tokens, view(at + (1 << 20), tokens),
                                            view(at + (K_cache << 21), 128), view(at + (1 << 27), 128), ctypes.byref(c), None, stream) == api.OK
        return bool(fake.fake_overlapped())

    set_weights()
    assert [step(1), step(2), step(3)] == [False, True, True]
    set_weights()
    fake.fake_capture(7)
    assert [step(1), step(2)] == [False, True]       # recorded one behind the other
    fake.fake_capture(0)
    assert [step(3), step(4)] == [False, True]       # nothing has run since the packing
    fake.fake_capture(8)
    assert [step(1), step(2)] == [True, True]        # weights packed, and read by a kernel, before whatever this records
    set_weights()                                    # recorded as well
    assert [step(3), step(4)] == [False, True]
    fake.fake_capture(9)
    assert [step(1), step(2)] == [False, True]
    fake.fake_capture(0)
    fake.lococo_destroy(handle)


@pytest.mark.parametrize("d,heads,k", [(64, 1100, 61), (128, 1500, 45)])
def test_grids_of_many_weight_sets(fake, d, heads, k):
    # more (set, tap) pairs than two of a grid's three axes can count
    from paper_2406_05317_b200 import api
    stream, handle, size, at = fake.fake_stream(), ctypes.c_void_p(), ctypes.c_size_t(), 1 << 30
    M, L = 128, 300
    cfg = api.Config(1, heads, d, M, k, 2 * d, 1, api.BF16, 0.0, 1e-6, L, api.PATH_AUTO)
    fake.fake_fail_at(0)
    assert fake.lococo_create(ctypes.byref(cfg), ctypes.byref(handle)) == api.OK
    assert fake.lococo_workspace_bytes(handle, ctypes.byref(size)) == api.OK
    assert fake.lococo_set_workspace(handle, at, size.value, stream) == api.OK
    assert fake.lococo_set_weights(handle, at, None, stream) == api.OK
    view = lambda tokens, ptr=at: api.Tensor(ptr, heads * tokens * d, tokens * d, d)
    none, c = api.Tensor(None, 0, 0, 0), ctypes.c_int32(0)
    tokens, cache = view(L), view(M)
    assert fake.lococo_process_sequence(handle, tokens, tokens, tokens, L, L, view(L, at + (1 << 32)), cache, view(M, at + (1 << 33)),
                                        ctypes.byref(c), at, stream) == api.OK
    assert fake.lococo_backward_scratch_bytes(handle, L, L, ctypes.byref(size)) == api.OK
    assert fake.lococo_process_sequence_backward(handle, tokens, tokens, tokens, tokens, L, L, 0, at, tokens, cache, cache, tokens,
                                                 tokens, tokens, at, None, none, none, at, size.value, stream) == api.OK
    fake.lococo_destroy(handle)


def test_every_group_of_a_backward_pass_fits_its_scratch(fake):
    # A call's chunks go in groups of as many as 128 MB hold, and the group that is left over has fewer: fewer tiles, more
    # partial sums of the convolution each.
    from paper_2406_05317_b200 import api
    rng = random.Random(4)
    # sizes whose left-over group would be split further than a whole one: 27 chunks behind three groups of 28; and others
    sizes = [(16, 128, 16, 128, 200, 22200), (1, 128, 16, 128, 5620, 39 * 5620), (4, 128, 16, 128, 1092, 68 * 1092), (12, 128, 16, 128, 196, 151 * 196),
             (8, 128, 16, 128, 224, 391 * 224), (8, 64, 48, 64, 100, 12100)]
    for _ in range(4000):
        d = rng.choice([64, 128])
        M = rng.randint(1, 6144 // d)
        B = int(16 * 512 ** rng.random())
        sizes.append((rng.choice([1, 2, 4, 8, 12, 16, 24, 32, 48]), d, M, d * rng.choice([1, 2]), B, B * rng.randint(2, 700) - rng.randint(0, B - 1)))
    left_over = 0
    for units, d, M, c_in, B, L in sizes:
        cfg, chunks = api.Config(1, units, d, M, 5, c_in, 0, api.F32, 0.0, 1e-6, B, api.PATH_AUTO), ctypes.c_int()
        for room in (1 << 40, rng.randint(1, 1 << 25)):      # all that a call asks for; what a caller has
            over = fake.fake_group_overrun(ctypes.byref(cfg), L, B, room, ctypes.byref(chunks))
            assert over in (0, -1), (units, d, M, c_in, B, L, room, over)
            left_over += over == 0 and -(-L // B) % chunks.value != 0
    assert left_over > 100


def test_scratch_of_a_larger_call_serves_a_smaller_one(fake):
    # A trainer's scratch is made once, for the longest sequence and the largest chunk.
    from paper_2406_05317_b200 import api
    rng, stream, at = random.Random(5), fake.fake_stream(), 1 << 30
    none = api.Tensor(None, 0, 0, 0)
    sizes = [(8, 64, 48, 12100, 100, 12200, 100), (8, 64, 48, 777, 64, 777, 512)]      # (L, B of the call; L, B that the scratch is made for)
    for _ in range(300):
        L, B = int(64 * 200 ** rng.random()), int(8 * 64 ** rng.random())
        sizes.append((rng.choice([1, 4, 8, 16]), rng.choice([64, 128]), rng.randint(4, 100), L, B, int(L * rng.uniform(1, 3)), int(B * rng.uniform(1, 8))))
    smaller = grouped = 0
    for heads, d, M, L, B, L_most, B_most in sizes:
        handle, size, whole = ctypes.c_void_p(), ctypes.c_size_t(), ctypes.c_size_t()
        cfg = api.Config(1, heads, d, M, 5, d, 0, api.F32, 0.0, 1e-6, B_most, api.PATH_AUTO)
        fake.fake_fail_at(0)
        assert fake.lococo_create(ctypes.byref(cfg), ctypes.byref(handle)) == api.OK
        assert fake.lococo_workspace_bytes(handle, ctypes.byref(size)) == api.OK
        assert fake.lococo_set_workspace(handle, at, size.value, stream) == api.OK
        assert fake.lococo_set_weights(handle, at, None, stream) == api.OK
        assert fake.lococo_backward_scratch_bytes(handle, L, B, ctypes.byref(whole)) == api.OK
        assert fake.lococo_backward_scratch_bytes(handle, L_most, B_most, ctypes.byref(size)) == api.OK
        smaller += size.value < whole.value
        tokens, cache = (api.Tensor(at, heads * n * d, n * d, d) for n in (L, M))
        grad = api.Tensor(2 * at, heads * L * d, L * d, d)

        def backward(scratch, grads=(grad, grad, grad)):
            before, after = ctypes.c_int64(), ctypes.c_int64()
            fake.lococo_launch_count(handle, ctypes.byref(before))
            status = fake.lococo_process_sequence_backward(handle, tokens, tokens, tokens, tokens, L, B, 0, at, tokens, cache, cache, *grads,
                                                           at, None, none, none, at, scratch, stream)
            fake.lococo_launch_count(handle, ctypes.byref(after))
            launches.append(after.value - before.value)
            return status

        launches = []
        assert backward(size.value) == api.OK, (heads, d, M, L, B, L_most, B_most)
        # gradients in the place of keys or values: a chunk at a time, which is done with a chunk's rows when it writes their gradients
        assert backward(whole.value, (grad, tokens, grad)) == backward(whole.value, (grad, grad, tokens)) == api.OK
        full = [min(M, n * B) + min(B, L - n * B) > M for n in range(-(-L // B))]
        assert launches[1] == launches[2] == 2 + sum(4 if compress else 2 for compress in full)
        # nor is there a chain to take apart with fewer than two compress steps
        assert launches[0] == launches[1] or sum(full) >= 2
        grouped += launches[0] < launches[1]
        assert backward(4 * heads * (2 * M * d + L)) == api.ERR_WORKSPACE      # (no room for anything but the cache's gradients and delta)
        fake.lococo_destroy(handle)
    assert smaller > 5 and grouped > 50


def test_a_small_call_asks_the_device_little(fake):
    # A one-chunk call is a launch of a few microseconds: what its plan needs to know of the device is asked in the first call.
    from paper_2406_05317_b200 import api
    stream, at, handle, size = fake.fake_stream(), 1 << 30, ctypes.c_void_p(), ctypes.c_size_t()
    cfg = api.Config(1, 4, 64, 32, 5, 64, 0, api.F32, 0.0, 1e-6, 16, api.PATH_AUTO)
    fake.fake_fail_at(0)
    assert fake.lococo_create(ctypes.byref(cfg), ctypes.byref(handle)) == api.OK
    assert fake.lococo_workspace_bytes(handle, ctypes.byref(size)) == api.OK
    assert fake.lococo_set_workspace(handle, at, size.value, stream) == api.OK
    assert fake.lococo_set_weights(handle, at, None, stream) == api.OK
    view = lambda ptr, n: api.Tensor(ptr, 4 * n * 64, n * 64, 64)
    for i in range(3):                 # (outputs of its own each time: nothing is replayed)
        c, x = ctypes.c_int32(32), view(at, 16)
        fake.fake_queries()
        assert fake.lococo_process_sequence(handle, x, x, x, 16, 16, view(at * (2 + i), 16), view(at * 8, 32), view(at * 9, 32), ctypes.byref(c), None, stream) == api.OK
        asked = fake.fake_queries()
        assert i == 0 or asked <= 2, asked
    fake.lococo_destroy(handle)


@pytest.mark.parametrize("units,d,M,B,L,k,c_mult,cache_len,one_launch", [
    (1, 64, 16, 16, 256, 5, 1, 0, True),
    (1600, 128, 8, 16, 32, 5, 1, 8, True),        # many units of few slots: blocks and tiles that the launches fill to a tenth
    (1600, 64, 4, 4, 12, 5, 1, 0, True),
    (1600, 64, 24, 4, 4, 1, 1, 24, True),
    (32, 128, 48, 8, 8, 9, 2, 0, False),          # chunks that only fill the cache, with weights that nobody needs
    (310, 128, 24, 1, 1, 31, 1, 0, False),
    (1310, 128, 87, 3, 18, 3, 1, 0, False),
    (1932, 128, 29, 2, 4, 9, 2, 29, True),
])
def test_way_of_a_small_fp32_loop(fake, units, d, M, B, L, k, c_mult, cache_len, one_launch):
    from paper_2406_05317_b200 import api
    stream, at, handle, size = fake.fake_stream(), 1 << 30, ctypes.c_void_p(), ctypes.c_size_t()
    cfg = api.Config(1, units, d, M, k, c_mult * d, 0, api.F32, 0.0, 1e-6, B, api.PATH_AUTO)
    fake.fake_fail_at(0)
    assert fake.lococo_create(ctypes.byref(cfg), ctypes.byref(handle)) == api.OK
    assert fake.lococo_workspace_bytes(handle, ctypes.byref(size)) == api.OK
    assert fake.lococo_set_workspace(handle, at, size.value, stream) == api.OK
    assert fake.lococo_set_weights(handle, at, None, stream) == api.OK
    view = lambda ptr, n: api.Tensor(ptr, units * n * d, n * d, d)
    c, before, after = ctypes.c_int32(cache_len), ctypes.c_int64(), ctypes.c_int64()
    fake.lococo_launch_count(handle, ctypes.byref(before))
    assert fake.lococo_process_sequence(handle, *[view(at, L)] * 3, L, B, view(2 * at, L), view(8 * at, M), view(9 * at, M), ctypes.byref(c), None, stream) == api.OK
    assert c.value == min(M, cache_len + L)
    fake.lococo_launch_count(handle, ctypes.byref(after))
    assert (after.value - before.value == 1) == one_launch
    fake.lococo_destroy(handle)
