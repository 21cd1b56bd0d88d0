"""The search with its form chosen by the caller: one warp per query, or a team
of a control warp with one to three expander warps (the library chooses by the
queries that share an SM).  Also how long a wait of the team form may last and
a query whose first expander answers nothing."""
import ctypes

import numpy as np

import paper_2401_11324_gb300 as bang

ONE_WARP = 1                    # form 1 + E: a team with E expanders; 0: the library's choice


def search(ix, q, k, L, ids, dist, params=None, k_per_q=None, L_per_q=None, form=0, wait_cycles=0, mute=None):
    """bang_search (with k_per_q and L_per_q: bang_search_batched) of an Index; returns the form that ran."""
    ran = ctypes.c_uint32(0)
    f = bang.lib().bang_internal_search
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_uint32] + [ctypes.c_void_p] * 2 + [
        ctypes.c_uint32] * 2 + [ctypes.c_void_p] * 4 + [ctypes.c_uint32, ctypes.c_longlong, ctypes.c_uint32,
                                                        ctypes.c_void_p]
    p = bang._ptr
    bang._check(f(ix.h, p(q), q.shape[0], p(k_per_q), p(L_per_q), k, L,
                  None if params is None else ctypes.addressof(params), p(ids), p(dist), None, form, wait_cycles,
                  0 if mute is None else 1 + mute, ctypes.addressof(ran)))
    return ran.value


def server_form(srv, form=0, wait_cycles=0, mute=None):
    """The launches of an idle Server from now on."""
    f = bang.lib().bang_internal_server_form
    f.argtypes = [ctypes.c_void_p, ctypes.c_uint32, ctypes.c_longlong, ctypes.c_uint32]
    bang._check(f(srv.h, form, wait_cycles, 0 if mute is None else 1 + mute))


def shard_graph(X, centres, ell, R, Lb, alpha, batch_frac, log2z, form=0, wait_cycles=0, mute=None):
    """bang_build_shard_graph with host arrays; returns the adjacency."""
    adj = np.zeros((len(X), R), np.uint32)
    f = bang.lib().bang_internal_build_shard_graph
    u, p, fl = ctypes.c_uint32, ctypes.c_void_p, ctypes.c_float
    f.argtypes = [ctypes.c_int, p, ctypes.c_int, ctypes.c_uint64, u, p, u, u, u, u, fl, fl, u, u, p, p, p, u,
                  ctypes.c_longlong, u]
    bang._check(f(0, bang._ptr(X), bang._DTYPES[X.dtype], len(X), X.shape[1], bang._ptr(centres), len(centres), ell, R,
                  Lb, alpha, batch_frac, log2z, 0, bang._ptr(adj), None, None, form, wait_cycles,
                  0 if mute is None else 1 + mute))
    return adj


def choice(dtype, n, d, M, R, mode, log2z, L, k, nq, link=0, batched=0, overlapped=0, sms=152):
    """(form, shared memory per query) that the library takes; needs no GPU."""
    b = ctypes.c_uint32(0)
    f = bang.lib().bang_internal_form
    f.argtypes = [ctypes.c_int, ctypes.c_uint64] + [ctypes.c_uint32] * 12 + [ctypes.c_void_p]
    return f(dtype, n, d, M, R, mode, log2z, L, k, nq, link, batched, overlapped, sms, ctypes.addressof(b)), b.value
