// Which kernels may share an SM, as far as tensor memory goes.
//
// tcgen05.alloc waits without a limit until its columns are free.  That is safe
// while every CTA that holds some finishes by itself.  CTAs of a cluster do not:
// they hold theirs until their peers have come as far.  Two kernels of such
// clusters on different streams could wait for each other for good, one's CTA
// holding what the other's peer needs on another SM, if the CTAs that fit an SM by
// their shared memory could want more than its 512 columns.  So they must not
// fit:
//   the split attention forward (256 columns, two CTAs an SM) takes so much
//   shared memory that two of its CTAs leave no room for a cluster product's;
//   cluster products (at most 128 columns) take at least kClusterProductSmem.
// (The persistent product takes a whole SM, and everything else that allocates
// finishes by itself.)
#pragma once

namespace sky {

constexpr int kSmemPerSM = 233472, kSmemPerCta = 1024;  // of an SM; reserved for a CTA
constexpr int kClusterProductSmem = 80 * 1024;          // dynamic shared memory, at least
constexpr int kSplitAttentionSmem = 73 * 1024;
static_assert(2 * (kSplitAttentionSmem + kSmemPerCta) + kClusterProductSmem + kSmemPerCta > kSmemPerSM,
              "two split attention CTAs and a cluster product on an SM");
static_assert(2 * (kSplitAttentionSmem + kSmemPerCta) <= kSmemPerSM, "two split attention CTAs on an SM");

}  // namespace sky
