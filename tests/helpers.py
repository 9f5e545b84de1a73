"""Shared helpers for the tests: tiny seeded problems and independent numpy restatements used as pins."""
import math

import numpy as np
import torch

from paper_2609_22098_b200 import synth


def tiny_problem(seed, V=8, D=3, r=4, u_std=1.5, z_sigma=1.0, bias_scale=1.0):
    """Random fp32 inputs for a tiny vocabulary: U [D+1][V], A [V][r], W [r][V]."""
    U = (synth.normals(seed, 40, 0, (D + 1) * V).reshape(D + 1, V) * u_std).float().numpy()
    A = (synth.normals(seed, 41, 0, V * r).reshape(V, r) * bias_scale / math.sqrt(r)).float().numpy()
    W = (synth.normals(seed, 42, 0, r * V).reshape(r, V)).float().numpy()
    return U, A, W


def tiny_z_path(seed, U, A, W, D, sigma=1.0, anchor=0):
    """Target logits for every token path of length 0..D over a tiny vocabulary (row order: by
    length, then base-V value of the path)."""
    V = U.shape[1]
    rows = sum(V ** k for k in range(D + 1))
    noise = synth.normals(seed, 43, 0, rows * V).reshape(rows, V).numpy()
    Z = np.empty((rows, V), np.float32)
    idx = 0
    for k in range(D + 1):
        for p in range(V ** k):
            last = anchor if k == 0 else p % V
            base = U[k].astype(np.float64) + A[last].astype(np.float64) @ W.astype(np.float64)
            Z[idx] = (base + sigma * noise[idx]).astype(np.float32)
            idx += 1
    return Z


def path_row(path, V):
    off = sum(V ** k for k in range(len(path)))
    idx = 0
    for t in path:
        idx = idx * V + int(t)
    return off + idx


def node_path(tree, i):
    seq = []
    while i >= 0:
        seq.append(int(tree["tok"][i]))
        i = int(tree["parent"][i])
    return tuple(reversed(seq))


def z_rows_for_tree(tree, Z_path, V):
    n = int(tree["n"])
    rows = [Z_path[0]]
    for i in range(n):
        rows.append(Z_path[path_row(node_path(tree, i), V)])
    return np.stack(rows)


def np_logits(U_row, a_row, W):
    return U_row.astype(np.float64) + a_row.astype(np.float64) @ W.astype(np.float64)


def np_softmax(l, T=1.0):
    x = (l - l.max()) / T
    e = np.exp(x)
    return e / e.sum()


def sigmoid(x):
    return 1.0 / (1.0 + math.exp(-x))


def logit(q):
    return math.log(q) - math.log1p(-q)


# (vocabulary, rank, batch) of walks -> is W streamed, requests a pass, sets of warps that share a range's tiles, tiles of a set together
# (148 SMs): one of every form that the walk's shared-memory plan can take
WALK_SHAPES = {
    (4104, 64, 97): (0, 64, 1, 1),      # one tile, passes of 64 and 33
    (2501, 16, 70): (0, 64, 1, 1),      # ragged rows, passes of 64 and 6
    (696, 8, 300): (0, 64, 1, 1),       # dozens of requests an owner
    (50257, 32, 9): (0, 16, 1, 3),      # three tiles in one set, ragged rows
    (64008, 32, 20): (0, 32, 2, 2),     # four tiles in two sets
    (100000, 64, 70): (0, 64, 2, 3),    # six, passes of 64 and 6
    (128256, 64, 36): (0, 64, 4, 2),    # seven: all of tensor memory
    (128256, 128, 70): (1, 64, 4, 2),   # the same streamed, passes of 64 and 6
    (151936, 96, 40): (1, 32, 4, 3),    # nine, streamed, passes of 32 and 8
    (151643, 64, 24): (0, 32, 4, 3),    # ragged rows
    (100277, 128, 20): (0, 16, 2, 3),   # ragged rows, passes of 16 and 4
    (113001, 128, 12): (0, 8, 2, 3),    # ragged rows, passes of 8 and 4
    (45000, 256, 20): (0, 32, 1, 3),    # an odd number of half tiles at the largest rank
    (230003, 64, 10): (0, 8, 4, 2),     # thirteen tiles, two rounds, ragged rows, passes of 8 and 2
}
