"""Host tables of the persistent Krylov cycle and of the gathered assembly (no GPU), against the mesh's pattern and
its chunk tables, which have tests of their own."""
import numpy as np
import pytest

from synthetic import batch, bifurcation, cube_kuhn, cylinder


@pytest.fixture(scope="module")
def L():
    from paper_2304_12032_gb300 import build

    build.build()
    from paper_2304_12032_gb300 import lfx

    return lfx


def mesh_of(which):
    return {"cube1": lambda: cube_kuhn(1, seed=1), "cube6": lambda: cube_kuhn(6, seed=6),
            "pipe": lambda: cylinder(1.0, 3.0, n_tets=20000, seed=7),
            "batch": lambda: batch([cube_kuhn(n, seed=n) for n in (2, 9, 3)] + [bifurcation(n_tets=4000, seed=1001)],
                                   tag_stride=0)}[which]()


def internal_pattern(mesh):
    """(row pointers, columns) in internal numbering, and the internal number of each caller node."""
    rp, ci = mesh.pattern()
    node = mesh.row_tiles()["row_node"]
    new = np.empty_like(node)
    new[node] = np.arange(node.size)
    cols = [np.sort(new[ci[rp[i]:rp[i + 1]]]) for i in node]
    return np.concatenate([[0], np.cumsum([c.size for c in cols])]), np.concatenate(cols), new


@pytest.mark.parametrize("which,ctas", [("cube1", 1), ("cube1", 3), ("cube6", 1), ("cube6", 42), ("pipe", 97),
                                        ("pipe", 151), ("batch", 7), ("batch", 151)])
def test_cycle_partition(L, which, ctas):
    """Row ranges cover every row once, in nearly equal shares, and inside one piece each where asked; the halo
    is exactly the columns of other CTAs; own rows followed by the halo, indexed by the local columns, give back
    the pattern block by block.  Twice the same."""
    m = mesh_of(which)
    mesh = L.Mesh.from_synthetic(m)
    rp, ci, new = internal_pattern(mesh)
    V = m.n_nodes
    for segments in ((False, True) if which == "batch" else (False,)):
        p = mesh.cycle_partition(ctas, segments)
        off, ho = p["row_off"], p["halo_off"]
        rows = np.diff(off)
        assert off[0] == 0 and off[-1] == V and rows.min() >= (1 if V >= ctas else 0)
        assert p["segments"] == (mesh.info()["n_components"] if segments else 1)
        assert p["max_rows"] == rows.max() and p["max_loc"] == (rows + np.diff(ho)).max()
        if segments:
            size = np.bincount(p["cta_seg"], weights=rows).astype(int)
            assert np.array_equal(np.sort(size), np.sort(np.diff(np.append(m.meta["node_offsets"], V)[: size.size + 1])))
            assert np.all(np.diff(p["cta_seg"]) >= 0)
            assert all(np.ptp(rows[p["cta_seg"] == c]) <= 1 for c in range(p["segments"]))
            # the largest share is the least possible: a smaller one would take more CTAs
            assert rows.max() == 1 or sum(-(-n // (rows.max() - 1)) for n in size) > ctas
        else:
            assert np.ptp(rows) <= 1 and not p["cta_seg"].any()
        for b in range(ctas):
            r0, r1 = off[b], off[b + 1]
            cols = ci[rp[r0]:rp[r1]]
            halo = p["halo"][ho[b]:ho[b + 1]]
            assert np.array_equal(halo, np.unique(cols[(cols < r0) | (cols >= r1)]))
            local = np.concatenate([np.arange(r0, r1), halo])
            assert np.array_equal(local[p["local_col"][rp[r0]:rp[r1]]], cols)
        q = mesh.cycle_partition(ctas, segments)
        assert all(np.array_equal(p[k], q[k]) for k in p)


def test_cycle_partition_arguments(L):
    mesh = L.Mesh.from_synthetic(mesh_of("batch"))
    for ctas, segments in ((0, False), (-1, False), (3, True)):       # four pieces
        with pytest.raises(L.LfxError) as err:
            mesh.cycle_partition(ctas, segments)
        assert err.value.status == L.LFX_ERR_INVALID_ARG


@pytest.mark.parametrize("which", ["cube1", "cube6", "pipe", "batch"])
def test_gather_tables(L, which):
    """Every run in the list of its block once, ascending; diagonal runs numbered one by one in run order."""
    mesh = L.Mesh.from_synthetic(mesh_of(which))
    g, ch = mesh.gather(), mesh.chunks()
    rp, ci, new = internal_pattern(mesh)
    row = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    assert np.array_equal(row[g["run_block"]], new[ch["run_row"]]) and np.array_equal(ci[g["run_block"]], new[ch["run_col"]])
    off, run = g["block_off"], g["block_run"]
    assert off[0] == 0 and off[-1] == run.size and np.array_equal(np.sort(run), np.arange(run.size))
    assert np.array_equal(g["run_block"][run], np.repeat(np.arange(ci.size), np.diff(off)))
    inside = np.ones(run.size, bool)
    inside[off[:-1][np.diff(off) > 0]] = False                        # first run of each block
    assert np.all(np.diff(run)[inside[1:]] > 0)
    diag = ch["run_row"] == ch["run_col"]
    assert g["diagonal_runs"] == diag.sum()
    assert np.array_equal(g["run_diag"][diag], np.arange(diag.sum())) and np.all(g["run_diag"][~diag] == -1)


def test_large_meshes_have_no_gather_tables(L):
    """Past 6,144 chunks of 32 elements (the scratch would exceed 160 MB)."""
    mesh = L.Mesh.from_synthetic(cube_kuhn(33, seed=1))
    assert len(mesh.chunks()["chunk_elem_off"]) - 1 > 6144 and mesh.gather() == {}
