// Host-side launch helpers for the pair enumeration kernels (enumerate.cuh).
#pragma once
#include <algorithm>

#include "context.cuh"
#include "enumerate.cuh"
#include "opposite.cuh"

namespace shci {

inline EnumArgs enum_args(const shci_ctx *c) {
    EnumArgs A{};
    A.dets = c->dets.p;
    A.astr = c->astr.p;
    A.bstr = c->bstr.p;
    A.ga_off = c->ga_off.p;
    A.gb_off = c->gb_off.p;
    A.ga_det = c->ga_det.p;
    A.gb_det = c->gb_det.p;
    A.ga_str = c->ga_str.p;
    A.gb_str = c->gb_str.p;
    A.as_off = c->as_off.p;
    A.as_idx = c->as_idx.p;
    A.work_counter = c->counter.p + 1;
    A.opp_lookup = c->opp_lookup ? 1 : 0;
    A.opp_hybrid = c->opp_hybrid ? 1 : 0;
    A.opp_factor = c->opp_factor;
    A.ia = c->ia.p;
    A.ib = c->ib.p;
    A.bs_off = c->bs_off.p;
    A.bs_idx = c->bs_idx.p;
    A.occ = c->occ.p;
    A.occ_words = c->occ_words;
    A.ow_off = c->ga_off.p;
    A.ow_ib = c->ga_ib.p;
    A.ow_det = c->ga_det.p;
    A.n_beta_str = c->Ub;
    A.opp_rows = opp_item_rows(c->n_det, c->n_sm);
    A.opp_beta_singles = (int)ceil_div(c->n_beta_singles, std::max<int64_t>(c->Ub, 1));
    A.bs_pair = c->bs_pair.p;
    A.ma = c->have_moves ? c->move_a.p : nullptr;
    A.mb = c->have_moves ? c->move_b.p : nullptr;
    A.n_pair = c->n_orb * (c->n_orb + 1) / 2;
    return A;
}

// One pass of the alpha-grouped (alpha_part) or beta-grouped enumeration:
// a persistent grid whose CTAs take work items from an atomic counter.
// opp: the opposite-spin doubles in the alpha-grouped part although the context
// has a pass for them.
template <int W, int MODE, int K>
void launch_enum(shci_ctx *c, EnumArgs A, const DevInts &I, bool alpha_part, bool opp = false) {
    CUDA_TRY(cudaMemsetAsync(c->counter.p + 1, 0, sizeof(int), c->st));
    if (!A.item_group) {                    // the context's items unless the caller gave its own
        A.item_group = alpha_part ? c->item_a_group.p : c->item_b_group.p;
        A.item_first = alpha_part ? c->item_a_first.p : c->item_b_first.p;
        A.n_items = alpha_part ? c->n_items_a : c->n_items_b;
    }
    const int blocks = c->n_sm * (2048 / ENUM_THREADS);
    if (alpha_part && c->opp_pass && !opp) k_enum_alpha<W, MODE, K, false><<<blocks, ENUM_THREADS, 0, c->st>>>(A, I);
    else if (alpha_part) k_enum_alpha<W, MODE, K, true><<<blocks, ENUM_THREADS, 0, c->st>>>(A, I);
    else k_enum_beta<W, MODE, K><<<blocks, ENUM_THREADS, 0, c->st>>>(A, I);
    KERNEL_CHECK();
    g_kernel_launches += 1;
}

// out[p] = x of the member at place p, k interleaved values each
static __global__ void k_group_vectors(const int32_t *__restrict__ mdet, int64_t n, int k, const double *__restrict__ x,
                                       double *__restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * k; e += (int64_t)gridDim.x * blockDim.x)
        out[e] = __ldg(&x[(int64_t)mdet[e / k] * k + e % k]);
}

// Does a product or gradient of k vectors take the opposite-spin pass?  Where the
// memory for its grouped vectors is not there, the alpha-grouped kernel finds those
// pairs instead, by the choice per alpha single.
inline bool takes_opposite_pass(shci_ctx *c, int k) {
    return c->opp_pass && try_alloc(c->x_grouped, (size_t)c->n_det * k);
}

// A.x in the order of the alpha groups' members, for the opposite-spin pass on
// the fly: a pair's place is then where its coefficient is.
inline void group_vectors(shci_ctx *c, EnumArgs &A, int k) {
    const int64_t n = c->n_det;
    c->x_grouped.alloc((size_t)n * k);
    const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(n * k, 256), (int64_t)c->n_sm * 16);
    k_group_vectors<<<blocks, 256, 0, c->st>>>(c->ga_det.p, n, k, A.x, c->x_grouped.p);
    KERNEL_CHECK();
    g_kernel_launches += 1;
    A.x_grouped = c->x_grouped.p;
}

template <int W, int MODE, int K, bool CHOICE>
void launch_opposite_as(shci_ctx *c, const EnumArgs &A, const DevInts &I) {
    const size_t smem = opp_smem(A.opp_rows, c->Ub);
    // the limit belongs to the kernel, not to the launch: always the largest table's,
    // so that contexts of other sizes in other host threads cannot lower it in between
    CUDA_TRY(cudaFuncSetAttribute(k_opposite<W, MODE, K, CHOICE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)OPP_SMEM_MAX));
    int per_sm = 0;
    CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_opposite<W, MODE, K, CHOICE>, ENUM_THREADS,
                                                           smem));
    const int blocks = (int)std::min<int64_t>(A.n_items, (int64_t)c->n_sm * std::max(per_sm, 1));
    k_opposite<W, MODE, K, CHOICE><<<blocks, ENUM_THREADS, smem, c->st>>>(A, I);
    KERNEL_CHECK();
    g_kernel_launches += 1;
}

// The opposite-spin pass (opposite.cuh) over the context's items, or the
// caller's (rows from A.row_det, ends in A.item_end).
template <int W, int MODE, int K>
void launch_opposite(shci_ctx *c, EnumArgs A, const DevInts &I) {
    CUDA_TRY(cudaMemsetAsync(c->counter.p + 1, 0, sizeof(int), c->st));
    if (!A.item_group) {
        A.item_group = c->item_o_group.p;
        A.item_first = c->item_o_first.p;
        A.n_items = c->n_items_o;
        A.row_det = c->ga_det.p;
    }
    if (A.n_items == 0) return;
    // growth has groups without new members; the other passes choose where k_opp_costs says so
    if (ModeOf<MODE>::inc || c->opp_choice) launch_opposite_as<W, MODE, K, true>(c, A, I);
    else if constexpr (!ModeOf<MODE>::inc) launch_opposite_as<W, MODE, K, false>(c, A, I);
}

}  // namespace shci
