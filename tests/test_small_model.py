"""Exchanges of the cluster kernel of small models, modelled on the host (tests/small_model.cpp): no copy lands on what its receiver has
still to read, whatever order the 16 thread blocks run in.  The header that the kernel takes its places and participants from
(csrc/ada_small_shape.h) is compiled with g++."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("small") / "small_model")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2412_18910_b200", "csrc"), "-o", exe,
                           os.path.join(ROOT, "tests", "small_model.cpp")])
    return lambda *a: subprocess.run([exe] + [str(x) for x in a], capture_output=True, text=True)


# d_model, heads, d_ffn, vocabulary, n_max: thread blocks without columns of d (128, 192), without a head (192), without tiles of gate/up
SHAPES = [(128, 2, 144, 272, 8), (128, 2, 128, 128, 1), (192, 3, 688, 4096, 8), (192, 3, 656, 4096, 11), (128, 2, 144, 272, 15),
          (256, 4, 688, 4096, 8), (256, 4, 656, 5136, 7), (256, 4, 128, 16384, 8)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("draft", [False, True])
def test_exchanges_are_ordered(model, shape, draft):
    n_max = shape[4]
    for rows in {1, min(5, n_max + 1), n_max + 1}:
        r = model(*shape, rows, 1 if draft else 4, n_max if draft else 0, 0, 60)
        assert r.returncode == 0, (rows, r.stdout + r.stderr)


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[0] < 256])
def test_the_model_sees_what_is_not_ordered(model, shape):
    """Thread blocks without a share that say nothing: found for every model narrower than 256."""
    r = model(*shape, 2, 4, 0, 1, 200)
    assert r.returncode == 1 and "lands on" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("draft", [False, True])
def test_a_wait_that_gives_up(model, shape, draft):
    """Its thread block takes no part any more, and nobody leaves before all copies have landed."""
    n_max = shape[4]
    for rows in {1, n_max + 1}:
        r = model(*shape, rows, 1 if draft else 4, n_max if draft else 0, 0, 300, 1)
        assert r.returncode == 0, (rows, r.stdout + r.stderr)


@pytest.mark.parametrize("gives_up,draft,found", [(2, False, "twice"), (2, True, "twice"), (3, False, "have left")])
def test_the_model_sees_a_thread_block_that_goes_on(model, gives_up, draft, found):
    """Barriers armed twice where a thread block that gave up goes on, copies to thread blocks that have left where it alone stays for
    them."""
    r = model(*SHAPES[-3], 9, 1 if draft else 4, 8 if draft else 0, 0, 3000, gives_up)
    assert r.returncode == 1 and found in r.stdout, r.stdout + r.stderr


def test_candidates_that_nobody_wrote(model):
    """Whatever lies in memory where a candidate should, the row that is read is one of the vocabulary's."""
    i = [0, 1, 4095, 4096, 2**31 - 1, -1, -2**31, 0x7f800000, 0x3f800000]
    r = model("token", 4096, *i)
    assert r.returncode == 0 and [int(x) for x in r.stdout.split()] == [0, 1, 4095] + [0] * 6


def test_shapes_of_the_other_kernels(model):
    """What the tests of the persistent pass and of the multi-row path run is refused by the cluster kernel's plan."""
    import synth_inputs as si
    from tests import test_gpu_routes
    for shape in test_gpu_routes.SHAPES:
        sh = si.scaled(si.SHAPES["tiny"], **shape)
        r = model(sh.d_model, sh.n_heads, sh.d_ffn, sh.vocab, sh.n_max, 1, sh.n_layers, 0, 0, 1)
        assert r.returncode == 3, (shape, r.stdout + r.stderr)
