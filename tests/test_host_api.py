"""The C ABI's host side on the CPU: the library's host sources compiled over
a stand-in for the CUDA runtime (host_api.cpp), so that what it uploads, and
what it does when memory runs out, can be looked at without a GPU."""
import os
import subprocess

import numpy as np
import pytest

from paper_2102_01366_gb300 import _build
from paper_2102_01366_gb300 import inputs as I

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host_api(tmp_path_factory):
    """check(name, mesh, kinds): the output of one check of host_api.cpp."""
    d = tmp_path_factory.mktemp("host_api")
    exe = str(d / "host_api")
    src = [os.path.join(HERE, "host_api.cpp")] + [os.path.join(_build.CSRC, f) for f in ("gks_mesh.cpp", "gks_stencil.cpp")]
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(_build._cuda_home(), "include"),
                    "-I", _build.INCLUDE, "-I", _build.CSRC] + src + ["-o", exe], check=True)

    def check(name, mesh, kinds):
        path = str(d / "mesh.bin")
        with open(path, "wb") as f:
            np.array([len(mesh["xyz"]), len(mesh["tet"])], np.int64).tofile(f)
            for a, t in ((mesh["xyz"], np.float64), (mesh["period"], np.float64), (mesh["tet"], np.int64),
                         (mesh["shift"], np.int8), (kinds, np.int8)):
                np.ascontiguousarray(a, dtype=t).tofile(f)
        r = subprocess.run([exe, name, path], capture_output=True, text=True, timeout=600)
        assert r.returncode == 0 and r.stdout.startswith("ok"), (r.returncode, r.stdout, r.stderr)
        return [int(x) for x in r.stdout.split()[1:]]
    return check


# 162 cells: one thread; 2,058: several threads in every loop over cells and faces
@pytest.mark.parametrize("dims", [(3, 3, 3), (7, 7, 7)])
def test_memory_that_cannot_be_had_is_reported(host_api, dims):
    """Each allocation of each call fails once: the call returns GKS_E_NOMEM
    (or succeeds without it), no exception leaves it, and a refused change of
    the face or cell order leaves the device's arrays as they were."""
    mesh = I.box_mesh(dims, jitter=0.1, seed=81, periodic=(False, True, True))
    kinds = I.boundary_kinds(mesh, {(0, "lo"): I.BC_NOSLIP_WALL, (0, "hi"): I.BC_FIXED})
    refused, = host_api("allocations", mesh, kinds)
    assert refused > 50


# a ragged last block of cells; one thread, and several in every loop: from
# 1,536 cells on for the cells, 16,384 faces and cells for the faces
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 3, 1), (8, 8, 4), (17, 13, 13)])
def test_a_states_mesh_arrays_are_the_meshs(host_api, dims):
    mesh = I.box_mesh(dims, jitter=0.1, seed=82, periodic=(False,) * 3)
    kinds = I.boundary_kinds(mesh, {(0, "lo"): I.BC_SLIP_WALL, (1, "hi"): I.BC_FIXED, (2, "lo"): I.BC_MOVING_WALL})
    assert host_api("arrays", mesh, kinds) == [2 + 6 + 6]


def test_a_state_keeps_its_boundary_kinds(host_api):
    """Kinds set on the mesh after a state's creation are for later states: a
    change of order uploads the state's own, with the operators its workspace
    has room for, and a state without fixed faces refuses a fixed state."""
    mesh = I.box_mesh((3, 2, 2), jitter=0.1, seed=83, periodic=(False,) * 3)
    assert host_api("kinds", mesh, I.boundary_kinds(mesh, {(0, "lo"): I.BC_NOSLIP_WALL})) == [3 * 2 * 6]


def test_misaligned_adjoint_scratch_is_refused(host_api):
    mesh = I.box_mesh((3, 2, 2), jitter=0.1, seed=84, periodic=(False,) * 3)
    assert host_api("scratch", mesh, I.wall_kinds(mesh, (0,))) == [2]


def test_a_state_without_a_step_has_no_residual(host_api):
    """Its residual is zero, whatever the workspace held before; the time step
    query no longer writes the sums."""
    mesh = I.box_mesh((3, 2, 2), jitter=0.1, seed=86, periodic=(False,) * 3)
    assert host_api("residual", mesh, I.wall_kinds(mesh, (0,))) == [3 * 5]


def test_fp64_flux_blocks_follow_the_devices_sms(host_api):
    """Blocks of 21 faces exactly where they leave the fullest SM of this
    device fewer warps than blocks of 32 do."""
    small, = host_api("flux_blocks", I.box_mesh((2, 2, 2), jitter=0.1, seed=85), np.zeros((48, 4)))
    assert small > 20
