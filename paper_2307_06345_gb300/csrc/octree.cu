// The build of one set as two calls: everything up to the leaf array, whose size the caller needs for
// its tree arrays, and the tree. Each strings the single steps' entry points together on one
// workspace, so that a program pays for the calls, checks and size queries of a binding twice per build
// and not seven times: up to some 10^5 particles the kernels finish before the next call arrives, and the
// calls set the time (through the Python binding, 20,000 particles with multipoles: 298 -> 241 us;
// 65,536 without: 203 -> 171; 1,000,000: 313 -> 290). Host code only: every step runs in the library's
// kernels.
#include "common.cuh"

namespace CST_NS {

int link_tree(const char* who, const void* leaves, long long n_leaves, void* node_keys, int* child, int* level_offsets,
              int* leaf_to_node, int* parent, const u32* leaf_offsets, u32* node_counts, void* ws, size_t ws_bytes,
              cudaStream_t st);

namespace {

inline size_t larger(size_t a, size_t b) { return a > b ? a : b; }

}  // namespace
}  // namespace CST_NS

extern "C" {

int CSTONE_FN(build_set_workspace_size)(int64_t n, int64_t leaf_cap, int32_t max_iters, size_t* bytes) {
    if (!bytes)
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(build_set_workspace_size)) ": bad argument");
    size_t box = 0, sort = 0, leaves = 0;
    if (int rc = cstone_bbox_workspace_size(n, &box)) return rc;
    if (int rc = CSTONE_FN(sort_workspace_size)(n, &sort)) return rc;
    if (int rc = CSTONE_FN(leaves_workspace_size)(n, leaf_cap, max_iters, &leaves)) return rc;
    *bytes = CST_NS::larger(box, CST_NS::larger(sort, leaves));
    return CSTONE_OK;
}

int CSTONE_FN(build_set)(const cstone_set_input* in, const cstone_set_params* prm, const cstone_set_buffers* out,
                         int64_t* n_leaves, int32_t* iters, void* ws, size_t ws_bytes, void* stream) {
    if (!in || !prm || !out || !n_leaves || (in->m && (!out->records || !out->records_ws)) ||
        (!in->box && !out->box_out))
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(build_set)) ": bad argument");
    const double* box = in->box;
    CST_KEY_C* keys = static_cast<CST_KEY_C*>(out->keys);
    CST_KEY_C* sorted = static_cast<CST_KEY_C*>(out->sorted_keys);
    if (!box) {
        if (int rc = cstone_bbox(in->x, in->y, in->z, in->n, out->box_out, ws, ws_bytes, stream)) return rc;
        box = out->box_out;
    }
    if (in->m) {
        if (int rc = CSTONE_FN(keys_records)(in->x, in->y, in->z, in->m, in->n, box, prm->curve, keys, out->records,
                                             out->records_ws, out->records_ws_bytes, stream))
            return rc;
    } else if (int rc = CSTONE_FN(keys)(in->x, in->y, in->z, in->n, box, prm->curve, keys, stream)) {
        return rc;
    }
    if (int rc = CSTONE_FN(sort)(keys, sorted, out->perm, in->n, ws, ws_bytes, stream)) return rc;
    return CSTONE_FN(build_leaves)(sorted, in->n, prm->ncrit, static_cast<CST_KEY_C*>(out->leaves), out->leaf_cap,
                                   n_leaves, out->leaf_counts, out->leaf_offsets, prm->max_iters, iters, ws, ws_bytes,
                                   stream);
}

int CSTONE_FN(build_tree_workspace_size)(int64_t n_leaves, int32_t with_masses, size_t* bytes) {
    if (!bytes)
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(build_tree_workspace_size)) ": bad argument");
    size_t link = 0, moments = 0;
    if (int rc = CSTONE_FN(link_workspace_size)(n_leaves, &link)) return rc;
    if (with_masses)
        if (int rc = CSTONE_FN(multipole_workspace_size)(0, n_leaves, &moments)) return rc;
    *bytes = CST_NS::larger(link, moments);
    return CSTONE_OK;
}

int CSTONE_FN(build_tree)(const cstone_set_buffers* set, int64_t n, int64_t n_leaves, const double* box,
                          const cstone_tree_buffers* out, void* ws, size_t ws_bytes, void* stream) {
    if (!set || !out || !set->leaf_offsets || !out->node_counts || (out->mass && (!box || !set->records)))
        return cst::fail(CSTONE_ERR_INVALID_ARG, CST_STR(CSTONE_FN(build_tree)) ": bad argument");
    if (int rc = CST_NS::link_tree(CST_STR(CSTONE_FN(build_tree)), set->leaves, n_leaves, out->node_keys, out->child,
                                   out->level_offsets, out->leaf_to_node, out->parent, set->leaf_offsets,
                                   out->node_counts, ws, ws_bytes, cst::as_stream(stream)))
        return rc;
    if (!out->mass) return CSTONE_OK;
    return CSTONE_FN(upsweep_multipoles_records)(set->records, set->perm, n, set->leaf_offsets, n_leaves,
                                                 out->leaf_to_node, out->child, out->level_offsets, box, out->mass,
                                                 out->com, out->quad, ws, ws_bytes, stream);
}

}  // extern "C"
