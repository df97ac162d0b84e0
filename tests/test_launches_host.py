"""Launches of the host code, run against a CUDA runtime without a device.

Slab launches (a film in the shared memory of one CTA or one cluster) of a
handle whose couplings or bulk field change between sweeps must allocate what
the present descriptor needs, in the form that fits it; a film set's launches
have a block per entry of the owner table."""
import os
import re
import subprocess

import pytest

from paper_1411_5588_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    B.build()
    exe = str(tmp_path_factory.mktemp("slab") / "launches")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    objs = [os.path.join(B.BUILD, o) for o in ("ising_api.o", "ising_kernels.o", "ising_noalloc.o", "ising_tune.o")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", cuda, "-I", B.INCLUDE, "-I", B.CSRC,
                    os.path.join(HERE, "host", "launches.cpp")] + objs + ["-lpthread", "-o", exe], check=True)
    return exe


AUTO, RESIDENT, CLUSTER = 0, 1, 5


# Sizes whose need differs between the three- and the seven-mask tables, by less
# and by more than the launch's padding, and where the task form stops fitting.
@pytest.mark.parametrize("Lx,Ly,Lz,shape", [
    (8, 8, 8, AUTO), (24, 601, 4, CLUSTER), (64, 768, 2, CLUSTER), (64, 153, 10, AUTO), (41, 47, 34, RESIDENT),
    (64, 128, 128, CLUSTER), (96, 192, 64, CLUSTER), (16, 150, 130, CLUSTER), (96, 192, 384, CLUSTER)])
def test_launch_holds_the_present_tables(harness, Lx, Ly, Lz, shape):
    out = subprocess.run([harness, "slab", str(Lx), str(Ly), str(Lz), str(shape)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    lines = [dict(zip(l.split()[::2], map(int, l.split()[1::2]))) for l in out.stdout.splitlines()]
    assert len(lines) == 5, out.stdout
    for n, l in enumerate(lines):
        assert l["smem"] >= l["need"], (n, l)
        assert l["tasks"] == l["fit"] and l["threads"] == l["want"], (n, l)
    # the same tables, the same launch
    assert lines[0] == lines[2] == lines[4] and lines[1] == lines[3]


# Words per CTA on both sides of one turn of drawing threads: 576, 768 and 1728 of
# eight calls, 1224 of two.
@pytest.mark.parametrize("Lx,Ly,Lz,tasks", [(48, 96, 64, 1), (64, 96, 64, 0), (48, 96, 192, 0), (64, 153, 10, 1)])
def test_slabs_of_many_words_are_columns(harness, Lx, Ly, Lz, tasks):
    out = subprocess.run([harness, "slab", str(Lx), str(Ly), str(Lz), str(CLUSTER)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    lines = [dict(zip(l.split()[::2], map(int, l.split()[1::2]))) for l in out.stdout.splitlines()]
    assert lines and all(l["C"] == 8 and l["tasks"] == tasks for l in lines), out.stdout


def test_adds_to_one_sum_have_one_scope():
    """In a cluster a layer's magnetisation gets adds from its own CTA and, in the
    same half-sweep, from the peer that holds the layer's wrap partner.  PTX:
    atomics on one address race unless each one's scope includes the other's
    thread.  So adds of CTA scope go to the CTA's own sums and nothing else does;
    what peers reach (through the table of shared addresses, or rank 0's
    totals) gets cluster scope from everyone."""
    with open(os.path.join(B.CSRC, "ising_kernels.cu")) as f:
        src = f.read()
    slab = src[src.index("slab path"):src.index("set-up")]
    own = set(re.findall(r"sadd<false>\((.*?), ", slab))
    assert own == {"smem_addr(s_m + kx - 1)"}
    shared = re.findall(r"sadd<(?:CL|true)>\((.*?), ", slab)
    assert sorted(set(shared)) == ["s.lm[kx - 1]", "tot", "tot + 4"]
    # the shared table's sums are not the CTA's own
    assert re.search(r"am = smem_addr\(s_m \+ \(CL \? s\.Lx \+ k : k\)\)", slab)


@pytest.mark.parametrize("items", [0, 1, 2])
def test_a_block_per_owner_entry(harness, items):
    """update_kernel takes the film of its block from the owner table and makes
    no second turn: every launch of a film set has a block per entry."""
    out = subprocess.run([harness, "grid", str(items), "0", "0", "0"], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    lines = [l.split() for l in out.stdout.splitlines()]
    assert len(lines) == 4 and all(l[1] == l[3] and int(l[3]) > 152 * 8 for l in lines), out.stdout


def test_a_measured_shape_is_for_its_table_form(harness):
    """A film in a bulk field draws seven masks per word where it draws three
    without one: the autotuner's choice for one is not taken for the other."""
    out = subprocess.run([harness, "tune", "41", "47", "34"], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    shapes = [int(l.split()[1]) for l in out.stdout.splitlines()]
    assert shapes == [CLUSTER, RESIDENT, CLUSTER, RESIDENT]


# kFormColumns, kFormColumnsLook, kFormWord, kFormWordLook
MASKS, COLUMNS_LOOK, WORD, WORD_LOOK = range(4)


@pytest.mark.parametrize("Lx,Ly,Lz,shape,H,form", [
    (120, 240, 1600, 4, 0.0, MASKS), (120, 240, 1600, 3, 0.0, MASKS), (120, 240, 1600, 4, 0.05, COLUMNS_LOOK),
    (120, 240, 1600, 3, -0.3, COLUMNS_LOOK), (32, 96, 64, 4, 0.05, COLUMNS_LOOK), (120, 240, 1600, 2, 0.0, WORD),
    (120, 240, 1600, 2, 0.05, WORD_LOOK), (64, 256, 512, 2, 0.05, WORD), (32, 96, 64, 2, 0.05, WORD)])
def test_films_in_a_field_look_thresholds_up(harness, Lx, Ly, Lz, shape, H, form):
    """Where a launch is bound by the integer pipes, a film in a bulk field
    compares each site with one looked-up threshold, not with seven."""
    out = subprocess.run([harness, "film", str(Lx), str(Ly), str(Lz), str(shape), str(H)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    forms = [int(l.split()[1]) for l in out.stdout.splitlines()]
    assert forms == [form, form], out.stdout


@pytest.mark.parametrize("items,H,form", [
    (0, (0, 0, 0), COLUMNS_LOOK), (2, (0, 0, 0.1), COLUMNS_LOOK), (1, (0, 0, 0), WORD), (1, (0.1, 0.1, 0), WORD),
    (1, (0, 0, 0.1), WORD_LOOK)])
def test_sets_look_thresholds_up(harness, items, H, form):
    """Sets of films: in columns always, at one word per thread where most words
    of a large launch are in a bulk field."""
    out = subprocess.run([harness, "grid", str(items)] + [str(h) for h in H], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert [int(l.split()[5]) for l in out.stdout.splitlines()] == [form] * 4, out.stdout


@pytest.mark.parametrize("Lx,Ly,Lz,rows", [
    (128, 512, 16, 1), (256, 512, 8, 1), (64, 128, 12, 1), (256, 1024, 16, 1), (512, 1024, 16, 4), (128, 512, 32, 1),
    (64, 256, 20, 1), (256, 1024, 32, 2), (512, 1024, 24, 2), (512, 1022, 16, 2), (512, 1024, 34, 1)])
@pytest.mark.parametrize("shape", [2, 3, 4])
def test_thin_films_pack_where_they_fill_the_gpu(harness, Lx, Ly, Lz, rows, shape):
    out = subprocess.run([harness, "film", str(Lx), str(Ly), str(Lz), str(shape), "0"], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert [int(l.split()[3]) for l in out.stdout.splitlines()] == [rows, rows], out.stdout


@pytest.mark.parametrize("Lx,Ly,Lz,every,shape", [
    (8, 8, 8, 1, RESIDENT), (16, 48, 32, 10, CLUSTER), (32, 48, 64, 0, CLUSTER), (32, 48, 64, 1, CLUSTER),
    (4, 128, 128, 0, CLUSTER), (2, 128, 256, 0, 2), (2, 128, 256, 10, 2), (2, 128, 256, 1, CLUSTER), (3, 128, 192, 0, 2),
    (64, 153, 10, 0, 2), (64, 153, 10, 1, CLUSTER), (2, 480, 34, 0, 2), (1, 64, 256, 0, RESIDENT),
    (400, 30, 8, 0, 2), (400, 30, 8, 1, CLUSTER), (1, 500, 64, 0, 2),
    (64, 128, 128, 0, 2), (120, 240, 1600, 0, 4)])
def test_unmeasured_films_take_clusters_of_few_words(harness, Lx, Ly, Lz, every, shape):
    out = subprocess.run([harness, "auto", str(Lx), str(Ly), str(Lz), str(every)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.split() == ["shape", str(shape)]


@pytest.mark.parametrize("items,thick,H,form", [(0, 0, 0, MASKS), (2, 0, 0, MASKS), (0, 1, 0, COLUMNS_LOOK),
                                                (0, 0, 0.2, COLUMNS_LOOK), (1, 0, 0, WORD)])
def test_sets_of_short_words_go_by_masks(harness, items, thick, H, form):
    out = subprocess.run([harness, "thin", str(items), str(thick), str(H)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert [int(l.split()[5]) for l in out.stdout.splitlines()] == [form] * 4, out.stdout


@pytest.mark.parametrize("n,rows", [(1, [1, 1, 1, 1, 1]), (3, [1, 2, 1, 1, 1]), (4, [4, 2, 1, 1, 1]), (16, [4, 2, 1, 1, 1])])
def test_sets_of_thin_and_thick_films_pack_by_their_work(harness, n, rows):
    """The thick films' words are eight calls each, the thinnest's two: a set fills
    the GPU by its calls, not by its words."""
    out = subprocess.run([harness, "pack", str(n)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert [int(l.split()[1]) for l in out.stdout.splitlines()] == rows * n, out.stdout
