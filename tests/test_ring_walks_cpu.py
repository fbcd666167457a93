"""The walks around the nodes that the membrane's node pass follows
(csrc/topology.cpp), on the host: every triangle is visited once from each of
its corners with its own neighbours and edges, whatever the valence of a node
and however many fans of triangles meet in it."""
import os
import subprocess

import numpy as np
import pytest

from workloads import mesh

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1312_3426_gb300", "csrc")
HERE = os.path.dirname(os.path.abspath(__file__))
START = 0x8000


def bipyramid(n):
    """n-gon with two apexes of valence n (n + 2 nodes), inward."""
    a = 2 * np.pi * np.arange(n) / n
    x = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, 1], [0, 0, -1]]])
    i, j = np.arange(n), (np.arange(n) + 1) % n
    t = np.concatenate([np.stack([j, i, i * 0 + n], 1), np.stack([i, j, i * 0 + n + 1], 1)])
    return x, t.astype(np.int32)


def pinched():
    """Two tetrahedra that share one node: two fans meet in it."""
    x, t = mesh.tetrahedron()
    y = x - x[3] + x[0]
    m = np.array([4, 5, 6, 0])
    return np.concatenate([x, y[:3]]), np.concatenate([t, m[t]]).astype(np.int32)


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("ring_walks") / "ring_walks")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, os.path.join(HERE, "ring_walks.cpp"),
                    os.path.join(CSRC, "topology.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("m", [mesh.tetrahedron(), mesh.icosphere(2), mesh.biconcave(3), bipyramid(5), bipyramid(70),
                               pinched()], ids=["tetrahedron", "icosphere2", "biconcave3", "valence5", "valence70",
                                                "two_fans"])
def test_walks_visit_every_corner_once(driver, m):
    nodes, tris = m
    text = f"{len(nodes)} {len(tris)}\n" + " ".join(map(repr, map(float, nodes.reshape(-1)))) + "\n" + \
        " ".join(map(str, tris.reshape(-1)))
    out = np.array(subprocess.run([driver], input=text, capture_output=True, text=True, check=True).stdout.split(),
                   np.int64)
    ne = 3 * len(tris) // 2
    edges, out = out[:2 * ne].reshape(-1, 2), out[2 * ne:]
    number = {tuple(sorted(e)): i for i, e in enumerate(edges.tolist())}
    n_slots, n_rec = out[:2]
    slots, rec = out[2:2 + 3 * n_slots].reshape(-1, 3), out[2 + 3 * n_slots:].reshape(-1, 4)
    assert n_slots % 32 == 0 and len(rec) == n_rec
    assert sorted(s for s in slots[:, 0].tolist() if s >= 0) == list(range(len(nodes)))
    seen = []
    for k, (v, first, n) in enumerate(slots.tolist()):
        if v < 0:
            assert n == 0
            continue
        assert first % 32 == k % 32 and first + 32 * (n - 1) < n_rec and n >= 4
        p = None
        for q, e_vq, e_pq, t in rec[first:first + 32 * n:32].tolist():
            start, q = bool(q & START), q & (START - 1)
            assert number[tuple(sorted((v, q)))] == e_vq
            if start:
                p = q
                continue
            assert number[tuple(sorted((p, q)))] == e_pq
            corner = tris[t].tolist()
            i = corner.index(v)
            assert [corner[(i + 1) % 3], corner[(i + 2) % 3]] == [p, q]
            seen.append((t, v))
            p = q
    assert len(seen) == len(set(seen)) == 3 * len(tris)
